// Exact moments of the per-sweep magnetisation and energy (Sec. 4.1: average
// magnetisation and the Binder parameter U4 = 1 - <m^4> / (3 <m^2>^2)).
//
// Over the samples s in [first, first + count) the kernel forms the exact
// integer sums S1 = sum |M| (64-bit), S2 = sum M^2 (128-bit), S4 = sum M^4
// (256-bit: |M| can reach 2^32 at L = 65,536), SE = sum E (signed 128-bit) and
// SE2 = sum E^2 (128-bit).  Integer addition is order-free, so any thread order
// gives the same sums; FP64 is used only once, on those exact sums:
//   <|m|> = S1 / (n N), <m^2> = S2 / (n N^2), <m^4> = S4 / (n N^4),
//   <e> = SE / (n N), <e^2> = SE2 / (n N^2), U4 = 1 - <m^4> / (3 <m^2>^2).
#include "ising_internal.cuh"

namespace ising {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kLimbs = 11;              // S1 | S2 (2) | S4 (4) | SE (2) | SE2 (2)
constexpr int kDigits = 3 * kLimbs;     // 22-bit digits of the limbs: 22 + 22 + 20 bits
constexpr int kDigitRow = 36;           // a warp's digits in shared memory, in whole 16-byte words
constexpr int kAhead = 4;               // samples a thread loads before it adds them

template <int N>
__device__ __forceinline__ void add_limbs(uint64_t* a, const uint64_t* b)
{
    uint64_t carry = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const uint64_t s = a[k] + b[k];
        const uint64_t c1 = s < a[k];
        const uint64_t s2 = s + carry;
        const uint64_t c2 = s2 < s;
        a[k] = s2;
        carry = c1 | c2;
    }
}

__device__ __forceinline__ void add_sample(uint64_t (&acc)[kLimbs], int64_t M, int64_t E)
{
    const uint64_t a = M < 0 ? (uint64_t)(-M) : (uint64_t)M;
    // S1
    acc[0] += a;
    // S2: a^2 as (lo, hi)
    const uint64_t lo = a * a, hi = __umul64hi(a, a);
    const uint64_t sq[2] = {lo, hi};
    add_limbs<2>(acc + 1, sq);
    // S4: (hi 2^64 + lo)^2 = lo^2 + 2 lo hi 2^64 + hi^2 2^128
    const uint64_t p_ll[4] = {lo * lo, __umul64hi(lo, lo), 0, 0};
    const uint64_t x0 = lo * hi, x1 = __umul64hi(lo, hi);
    const uint64_t p_lh[4] = {0, x0 << 1, (x1 << 1) | (x0 >> 63), x1 >> 63};
    const uint64_t p_hh[4] = {0, 0, hi * hi, __umul64hi(hi, hi)};
    add_limbs<4>(acc + 3, p_ll);
    add_limbs<4>(acc + 3, p_lh);
    add_limbs<4>(acc + 3, p_hh);
    // SE (two's complement 128-bit)
    const uint64_t se[2] = {(uint64_t)E, E < 0 ? ~0ull : 0ull};
    add_limbs<2>(acc + 7, se);
    // SE2
    const uint64_t ae = E < 0 ? (uint64_t)(-E) : (uint64_t)E;
    const uint64_t e2[2] = {ae * ae, __umul64hi(ae, ae)};
    add_limbs<2>(acc + 9, e2);
}

// One CTA: a query is a few hundred samples, and what it takes is a chain of latencies.  So the
// sums over a warp are single reduction instructions on 22-bit digits (32 of them add up to 27
// bits, 16 warps' to 31), one barrier joins the warps, one lane per quantity puts its digits
// together, and the five quotients are one FP64 division in five lanes.  A thread has kAhead
// samples' loads in flight, for histories of many samples.  A query of 200, 10,000, 100,000
// samples takes 20.9, 29.5, 106 us from the call to its result (of which 15.5 any read-back of
// one entry); with 256 threads, a tree of eight barriers over the limbs and one thread's six
// quotients it took 22.1, 36.5, 159.
// desc: a batch lattice, whose history and sweep count are read from there (the samples then are
// those from `first` on); report (may be null) receives the status word and the sweep count.
__global__ void __launch_bounds__(kThreads) moments_kernel(const LatticeDesc* desc, const int64_t* hist, int64_t first,
                                                           int64_t count, int64_t N, double* out6, uint64_t* sums_out,
                                                           const int* status, int64_t* report)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (desc) {
        hist = desc->hist;
        count = (int64_t)desc->sweep - first;
    }
    if (report && threadIdx.x == kThreads - 1) {
        report[0] = status ? *status : 0;
        report[1] = first + count;
    }
    if (count <= 0) return;  // refused by the caller
    __shared__ alignas(16) uint32_t digits[kWarps][kDigitRow];
    __shared__ uint32_t total[kDigits];
    const int used = count < kThreads ? (int)((count + 31) / 32) : kWarps;  // warps with samples
    if (warp < used) {
        uint64_t acc[kLimbs];
#pragma unroll
        for (int k = 0; k < kLimbs; ++k) acc[k] = 0;
        const int64_t* h = hist + 2 * first;
        for (int64_t s0 = threadIdx.x; s0 < count; s0 += kAhead * kThreads) {
            int64_t M[kAhead], E[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const int64_t s = s0 + u * kThreads;  // a missing sample adds nothing: M = E = 0
                M[u] = s < count ? h[2 * s] : 0;
                E[u] = s < count ? h[2 * s + 1] : 0;
            }
#pragma unroll
            for (int u = 0; u < kAhead; ++u)
                if (s0 + u * kThreads < count) add_sample(acc, M[u], E[u]);
        }
        __syncwarp();
        uint32_t d[kDigitRow];
#pragma unroll
        for (int k = 0; k < kLimbs; ++k) {
            d[3 * k] = __reduce_add_sync(~0u, (uint32_t)acc[k] & 0x3FFFFFu);
            d[3 * k + 1] = __reduce_add_sync(~0u, (uint32_t)(acc[k] >> 22) & 0x3FFFFFu);
            d[3 * k + 2] = __reduce_add_sync(~0u, (uint32_t)(acc[k] >> 44));
        }
#pragma unroll
        for (int k = kDigits; k < kDigitRow; ++k) d[k] = 0;
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < kDigitRow; k += 4)
                *reinterpret_cast<uint4*>(&digits[warp][k]) = make_uint4(d[k], d[k + 1], d[k + 2], d[k + 3]);
        }
    }
    __syncthreads();
    if (warp != 0) return;
    for (int k = lane; k < kDigits; k += 32) {
        uint32_t t = 0;
        for (int w = 0; w < used; ++w) t += digits[w][k];
        total[k] = t;
    }
    __syncwarp();
    // lane 0..4: S1, S2, S4, SE, SE2
    const int limb0 = lane == 0 ? 0 : lane == 1 ? 1 : lane == 2 ? 3 : lane == 3 ? 7 : 9;
    const int limbs = lane == 0 ? 1 : lane == 2 ? 4 : 2;
    double value = 0.0;
    if (lane < 5) {
        uint64_t t[4], carry = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            t[k] = 0;
            if (k < limbs) {
                const uint32_t* p = total + 3 * (limb0 + k);
                const unsigned __int128 v = (unsigned __int128)p[0] + ((unsigned __int128)p[1] << 22) +
                                            ((unsigned __int128)p[2] << 44) + carry;
                t[k] = (uint64_t)v;
                carry = (uint64_t)(v >> 64);
                if (sums_out) sums_out[limb0 + k] = t[k];
            }
        }
        const bool negative = lane == 3 && (t[1] >> 63) != 0;
        if (negative) {  // the magnitude of the 128-bit value
            t[0] = ~t[0] + 1ull;
            t[1] = ~t[1] + (t[0] == 0 ? 1ull : 0ull);
        }
        const double word = 18446744073709551616.0;
        const double sum = (((double)t[3] * word + (double)t[2]) * word + (double)t[1]) * word + (double)t[0];
        const double n = (double)count, dN = (double)N;
        const double per = lane == 0 || lane == 3 ? dN : lane == 2 ? (dN * dN) * (dN * dN) : dN * dN;
        value = (negative ? -sum : sum) / (n * per);
        out6[lane] = value;
    }
    const double m2 = __shfl_sync(~0u, value, 1), m4 = __shfl_sync(~0u, value, 2);
    if (lane == 0) out6[5] = m2 > 0.0 ? 1.0 - m4 / (3.0 * m2 * m2) : 0.0;
}

}  // namespace

cudaError_t launch_moments(const LatticeDesc* desc, const int64_t* hist, int64_t first, int64_t count, int64_t N,
                           double* out6, uint64_t* sums, const int* status, int64_t* report, cudaStream_t s)
{
    moments_kernel<<<1, kThreads, 0, s>>>(desc, hist, first, count, N, out6, sums, status, report);
    return cudaGetLastError();
}

}  // namespace ising
