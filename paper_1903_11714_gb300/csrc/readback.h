// Page-locked blocks and the kernels that fill them (readback.cu).
#pragma once
#include <cuda_runtime.h>

#include "ising_device.cuh"

namespace ising {

// One more (+1) or one fewer (-1) handle or batch alive.
void readback_user(int change);

// A block held for the duration of a call.  ok() is false where none could be had.
struct PinnedBlock {
    static constexpr int64_t kBytes = 64 * 1024;
    static constexpr int64_t kEntries = (kBytes - 16) / 16;  // (M, E) entries behind status and sweep count
    void* p = nullptr;
    cudaError_t error = cudaSuccess;
    PinnedBlock();
    ~PinnedBlock();
    PinnedBlock(const PinnedBlock&) = delete;
    PinnedBlock& operator=(const PinnedBlock&) = delete;
    bool ok() const { return p != nullptr; }
    int64_t* words() const { return static_cast<int64_t*>(p); }
};

constexpr int64_t kLastEntry = -1;
// out[0] = *status (0 for null), out[1] = desc's sweep count (0 for null desc), out[2 ..] = (M, E)
// entries first .. first + count - 1 of desc's history (of hist for null desc), left out where
// they lie beyond desc's sweep count; first = kLastEntry: desc's entry after its last sweep.
cudaError_t launch_report(const LatticeDesc* desc, const int64_t* hist, int64_t first, int64_t count, const int* status,
                          int64_t* out, cudaStream_t s);
// out[0] = *status (0 for null), out[4 ..] = the n words.
cudaError_t launch_report_words(const uint32_t* words, int64_t n, const int* status, uint32_t* out, cudaStream_t s);

}  // namespace ising
