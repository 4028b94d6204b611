// Blocks that the report kernels (readback.cu) fill for the synchronising calls.  Host code only.
//
// A block is page-locked memory that a kernel writes straight into.  Blocks are shared by
// the process: a call takes one for its duration, so two threads never share one; at most kKept
// wait for the next call, and all are given back when the last handle is freed.  Where no
// page-locked memory can be had, a call takes a block of device memory and copies it.
#pragma once
#include <cstdint>
#include <cstdlib>
#include <mutex>
#include <vector>

#include <cuda_runtime_api.h>

namespace ising {

struct ReportPool {
    static constexpr size_t kKept = 8;
    std::mutex mu;
    std::vector<void*> free;
    int64_t users = 0;  // handles and batches alive
};
inline ReportPool& report_pool()
{
    static ReportPool* pool = new ReportPool;  // never destroyed: handles may outlive static objects
    return *pool;
}

// One more (+1) or one fewer (-1) handle or batch alive.
inline void readback_user(int change)
{
    ReportPool& pool = report_pool();
    std::vector<void*> unused;
    {
        std::lock_guard<std::mutex> lock(pool.mu);
        pool.users += change;
        if (pool.users == 0) unused.swap(pool.free);
    }
    for (void* p : unused) cudaFreeHost(p);
}

// A block held for the duration of a call.  ok() is false where none could be had.
class ReportBlock {
public:
    static constexpr int64_t kBytes = 64 * 1024;
    static constexpr int64_t kEntries = (kBytes - 16) / 16;  // (M, E) entries behind status and sweep count
    cudaError_t error = cudaSuccess;

    ReportBlock()
    {
        ReportPool& pool = report_pool();
        {
            std::lock_guard<std::mutex> lock(pool.mu);
            if (!pool.free.empty()) {
                host_ = pool.free.back();
                pool.free.pop_back();
            }
        }
        if (host_) return;
        if (cudaHostAlloc(&host_, kBytes, cudaHostAllocPortable | cudaHostAllocMapped) == cudaSuccess) return;
        cudaGetLastError();
        host_ = nullptr;
        error = cudaMalloc(&device_, kBytes);
        if (error != cudaSuccess) {
            device_ = nullptr;
            return;
        }
        host_ = std::malloc(kBytes);
        if (!host_) error = cudaErrorMemoryAllocation;
    }
    ~ReportBlock()
    {
        if (device_) {
            cudaFree(device_);
            std::free(host_);
            return;
        }
        if (!host_) return;
        {
            ReportPool& pool = report_pool();
            std::lock_guard<std::mutex> lock(pool.mu);
            if (pool.users > 0 && pool.free.size() < ReportPool::kKept) {
                pool.free.push_back(host_);
                return;
            }
        }
        cudaFreeHost(host_);
    }
    ReportBlock(const ReportBlock&) = delete;
    ReportBlock& operator=(const ReportBlock&) = delete;

    bool ok() const { return host_ != nullptr; }
    // Where a kernel writes.
    int64_t* target() const { return static_cast<int64_t*>(device_ ? device_ : host_); }
    // Waits for the stream; the first `bytes` of what a kernel wrote are then at words().
    cudaError_t fetch(size_t bytes, cudaStream_t s)
    {
        if (device_) {
            const cudaError_t e = cudaMemcpyAsync(host_, device_, bytes, cudaMemcpyDeviceToHost, s);
            if (e != cudaSuccess) return e;
        }
        return cudaStreamSynchronize(s);
    }
    const int64_t* words() const { return static_cast<const int64_t*>(host_); }

private:
    void* host_ = nullptr;
    void* device_ = nullptr;  // only where host_ is not page-locked
};

}  // namespace ising
