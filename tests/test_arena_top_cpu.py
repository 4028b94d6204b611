"""Blocks placed from the end of the batch arena (FreeList::alloc_top, CPU): the last gap that holds
the rounded size, its end; merged with its neighbours on release like any other."""
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path_factory.mktemp("arena") / "arena_top_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-I", os.path.join(ROOT, "paper_1903_11714_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "arena_top_check.cpp"), "-o", exe], check=True)
    return exe


def run(exe, lines):
    out = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True).stdout.split()
    return [int(v) for v in out]


def test_gives_way_and_merges(exe):
    # 4,096 bytes: a lattice at the bottom, a workspace at the top; it gives way to a lattice that
    # needs the whole rest, and everything merges again
    out = run(exe, ["reset 4096", "alloc 1000", "top 2048", "alloc 2000", "free 2048 2048", "alloc 3000", "top 1", "free 0 1000",
                    "free 1024 3000"])
    assert out == [0, 2048, -1, 1024, -1, 0, 1]


def test_random_against_a_model(exe):
    rng, size = random.Random(5), 1 << 16
    lines, want, live = [f"reset {size}"], [], []
    for _ in range(3000):
        if live and rng.random() < 0.45:
            off, n = live.pop(rng.randrange(len(live)))
            lines.append(f"free {off} {n}")
            continue
        n, top = rng.randint(1, 9000), rng.random() < 0.5
        need, pos, gaps = -(-n // 256) * 256, 0, []
        for off, m in sorted(live):
            gaps.append((pos, off - pos))
            pos = off + -(-m // 256) * 256
        gaps = [g for g in gaps + [(pos, size - pos)] if g[1] >= need]
        off = -1 if not gaps else (gaps[-1][0] + gaps[-1][1] - need if top else gaps[0][0])
        lines.append(f"{'top' if top else 'alloc'} {n}")
        want.append(off)
        if off >= 0:
            live.append((off, n))
    got = run(exe, lines)
    assert got[:-2] == want
    assert got[-2] == sum(-(-n // 256) * 256 for _, n in live)
