// Drives the report blocks (report_block.h) against a stand-in of the CUDA calls that they make:
// "page-locked" memory that can be refused, and "device" memory that the host cannot see
// except by a copy.  Prints one line per check, "ok" or what went wrong.
#include <cstdio>
#include <cstring>
#include <map>

#include "report_block.h"

namespace {
bool refuse_pinned = false, refuse_device = false;
std::map<void*, char> alive;  // 'p' page-locked, 'd' device
int copies = 0, waits = 0;

cudaError_t give(void** p, size_t n, char kind, bool refuse)
{
    if (refuse) return cudaErrorMemoryAllocation;
    *p = std::calloc(n, 1);
    alive[*p] = kind;
    return cudaSuccess;
}
cudaError_t take(void* p, char kind)
{
    if (!alive.count(p) || alive[p] != kind) return cudaErrorInvalidValue;
    alive.erase(p);
    std::free(p);
    return cudaSuccess;
}
int count(char kind)
{
    int n = 0;
    for (auto& a : alive) n += a.second == kind;
    return n;
}
void check(bool good, const char* what) { std::printf("%s\n", good ? "ok" : what); }
}  // namespace

cudaError_t cudaHostAlloc(void** p, size_t n, unsigned int) { return give(p, n, 'p', refuse_pinned); }
cudaError_t cudaFreeHost(void* p) { return take(p, 'p'); }
cudaError_t cudaMalloc(void** p, size_t n) { return give(p, n, 'd', refuse_device); }
cudaError_t cudaFree(void* p) { return take(p, 'd'); }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return ++waits, cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t)
{
    std::memcpy(dst, src, n);
    return ++copies, cudaSuccess;
}

int main()
{
    using ising::ReportBlock;
    auto kernel = [](int64_t* out) {  // what a report kernel does
        for (int k = 0; k < 19; ++k) out[k] = 100 + k;
    };
    ising::readback_user(1);
    for (int round = 0; round < 2; ++round) {
        ReportBlock a, b;
        check(a.ok() && b.ok() && a.target() != b.target(), "two calls share a block");
        kernel(a.target());
        check(a.fetch(19 * 8, nullptr) == cudaSuccess && a.words()[18] == 118, "page-locked report");
    }
    check(count('p') == 2 && copies == 0 && waits == 2, "blocks are not kept for the next call");

    // no page-locked memory beyond what is held: the third call at a time takes device memory
    refuse_pinned = true;
    {
        ReportBlock a, b, c;
        check(c.ok(), "no block without page-locked memory");
        if (c.ok()) {
            kernel(c.target());
            check(c.target() != c.words(), "the kernel would write pageable memory");
            check(c.fetch(19 * 8, nullptr) == cudaSuccess && c.words()[0] == 100 && c.words()[18] == 118, "copied report");
        }
        check(copies == 1 && count('d') == 1, "one device block, one copy");
        refuse_device = true;
        ReportBlock d;
        check(!d.ok() && d.error == cudaErrorMemoryAllocation, "neither kind of memory");
    }
    check(count('d') == 0 && count('p') == 2, "device blocks are kept");
    ising::readback_user(-1);
    check(alive.empty(), "blocks outlive the last handle");
    return 0;
}
