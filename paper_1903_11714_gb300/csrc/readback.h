// Kernels that fill the blocks of the synchronising calls (readback.cu).
#pragma once
#include <cuda_runtime.h>

#include "ising_device.cuh"
#include "report_block.h"

namespace ising {

constexpr int64_t kLastEntry = -1;
// out[0] = *status (0 for null), out[1] = desc's sweep count (0 for null desc), out[2 ..] = (M, E)
// entries first .. first + count - 1 of desc's history (of hist for null desc), left out where
// they lie beyond desc's sweep count; first = kLastEntry: desc's entry after its last sweep.
cudaError_t launch_report(const LatticeDesc* desc, const int64_t* hist, int64_t first, int64_t count, const int* status,
                          int64_t* out, cudaStream_t s);
// out[0] = *status (0 for null), the n words from out[2] on.
cudaError_t launch_report_words(const uint32_t* words, int64_t n, const int* status, int64_t* out, cudaStream_t s);

}  // namespace ising
