"""The blocks that bring results to the host (csrc/report_block.h) against a stand-in of the CUDA
calls (CPU): kept for the next call, given back with the last handle, and a report still
arrives where no page-locked memory can be had."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def cuda_include():
    for nvcc in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if nvcc and os.path.exists(nvcc):
            return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    pytest.skip("no CUDA headers")


def test_report_blocks(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "report_block_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-I", os.path.join(ROOT, "paper_1903_11714_gb300", "csrc"),
                    "-I", cuda_include(), os.path.join(ROOT, "tests", "report_block_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")
    assert [line for line in out if line and line != "ok"] == []
    assert out.count("ok") >= 10
