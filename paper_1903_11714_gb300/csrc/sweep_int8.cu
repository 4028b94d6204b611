// Plain int8 checkerboard half-sweep: the GPU analogue of the paper's
// UpdateNaive (Algorithm 1) on a row-major L x L lattice of +1/-1 bytes, with
// the same Philox keying, integer thresholds and fused M/E counts as the
// bit-packed kernel, so both reach the same chain bit for bit.
//
// The start-state kernel works on 8-byte chunks (columns 8g .. 8g+7): the four
// sites of each colour in a chunk lie in one plane word and take their start spins
// from its first random word.  The half-sweep works on plane words, the 32 target sites
// that share a word's random numbers: a 64-byte row segment when L % 64 == 0, else eight
// consecutive 8-byte chunks.  The bytes' signs are packed into bit words (five operations
// per 16 bytes), the neighbour count and the acceptance test are the packed kernel's
// (word_update.cuh), and the flips are spread back over the bytes.
#include "ising_internal.cuh"
#include "word_update.cuh"

namespace ising {
namespace {


__global__ void int8_init_kernel(int8_t* lat, int64_t L, uint64_t key, int start)
{
    const int64_t G = L / 8;
    const int64_t chunks = L * G;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < chunks;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = idx / G, g = idx - i * G;
        uint64_t v = 0;
        if (start == 1) {
            v = 0x0101010101010101ull;
        } else {
            // the chunk's 4 sites of each colour have plane indices p0 .. p0+3, all in
            // plane word p0 >> 5 (p0 is a multiple of 4)
            const uint64_t p0 = (uint64_t)i * (uint64_t)(L / 2) + 4ull * (uint64_t)g;
            for (int c = 0; c < 2; ++c) {
                const uint32_t up_bits = hot_start_word(p0 >> 5, (uint32_t)c, key) >> (p0 & 31);
                const int r = (int)((i + c) & 1);
                for (int b = 0; b < 4; ++b) {
                    const uint64_t byte = ((up_bits >> b) & 1u) ? 0x01ull : 0xFFull;
                    v |= byte << (8 * (2 * b + r));
                }
            }
        }
        *reinterpret_cast<uint64_t*>(lat + i * L + 8 * g) = v;
    }
}

__device__ __forceinline__ void block_add_pair(long long a, long long b, int64_t* slot)
{
    __shared__ long long red[2][32];
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        red[0][warp] = a;
        red[1][warp] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long sa = 0, sb = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            sa += red[0][k];
            sb += red[1][k];
        }
        atomicAdd(reinterpret_cast<unsigned long long*>(slot), (unsigned long long)sa);
        atomicAdd(reinterpret_cast<unsigned long long*>(slot + 1), (unsigned long long)sb);
    }
}

// Signs of 16 bytes of +1 / -1 (four words): bits 2j + h of the low byte are columns
// 4j + 2h, of the next byte columns 4j + 2h + 1 (j = word, h = 0, 1); 1 = -1.  Bits 1 .. 7 of
// a byte all hold its sign, so each word can give a bit at a place of its own.
__device__ __forceinline__ uint32_t pack16(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3)
{
    const uint32_t a = (w0 & 0x07070707u) | (w1 & ~0x07070707u);  // bits 1 (w0) and 3 (w1)
    const uint32_t b = (w2 & 0x3F3F3F3Fu) | (w3 & ~0x3F3F3F3Fu);  // bits 5 (w2) and 7 (w3)
    const uint32_t c = (a & 0x0F0F0F0Fu) | (b & ~0x0F0F0F0Fu);
    // columns 4j, 4j + 1 at bits 2j + 1 of the two low bytes; 4j + 2, 4j + 3 beside them
    return ((c & 0xAAAAAAAAu) | ((c >> 15) & 0x55555555u)) >> 1;
}

// Packed signs of a 64-byte row segment: bit b of `even` is column 2b, of `odd` column 2b + 1.
__device__ __forceinline__ void pack64(const uint4 (&v)[4], uint32_t& even, uint32_t& odd)
{
    uint32_t x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = pack16(v[k].x, v[k].y, v[k].z, v[k].w);
    const uint32_t lo = __byte_perm(x[0], x[1], 0x5140), hi = __byte_perm(x[2], x[3], 0x5140);
    even = __byte_perm(lo, hi, 0x5410);
    odd = __byte_perm(lo, hi, 0x7632);
}

// The byte word with the signs of its target bytes turned where flips says so: bit 7 of byte 0
// for its first target, bit 7 of byte 2 for its second.  spread picks the bytes (kSpread[r]).
__device__ __forceinline__ uint32_t turn(uint32_t w, uint32_t flips, uint32_t spread)
{
    uint32_t bytes;  // (__byte_perm takes no sign selectors)
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(bytes) : "r"(flips), "r"(spread));
    return w ^ (bytes & 0xFEFEFEFEu);  // 0x01 <-> 0xFF
}
// a byte's sign over a whole byte (selector 8 | byte) for the target bytes, else zero
constexpr uint32_t kSpread0 = 0x4A48u, kSpread1 = 0xA484u;

__device__ __forceinline__ void turn64(uint4 (&v)[4], uint32_t f, uint32_t spread)
{
    // bits 2k and 2k + 1 of f at bits 2k and 16 + 2k of (k < 8 ? lo : hi)
    const uint32_t fe = f & 0x55555555u, fo = (f >> 1) & 0x55555555u;
    const uint32_t lo = __byte_perm(fe, fo, 0x5410) << 1, hi = __byte_perm(fe, fo, 0x7632) << 1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t x = k < 2 ? lo : hi;
        const int o = 8 * (k & 1);
        // bits o, o + 2, .. moved to bit 7 of bytes 0 and 2 (x is one place up already)
        v[k].x = turn(v[k].x, o == 0 ? x << 6 : x >> 2, spread);
        v[k].y = turn(v[k].y, o == 0 ? x << 4 : x >> 4, spread);
        v[k].z = turn(v[k].z, o == 0 ? x << 2 : x >> 6, spread);
        v[k].w = turn(v[k].w, o == 0 ? x : x >> 8, spread);
    }
}

__device__ __forceinline__ void load_segment(const int8_t* p, uint4 (&v)[4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = reinterpret_cast<const uint4*>(p)[k];
}

struct Int8Sweep {
    int8_t* lat;
    int64_t L;
    uint64_t key;
    uint32_t t2, t4, all2, all4;
    uint32_t sweep;
    int colour;
    int64_t* hist_slot;
};

// Counts of the white pass: M = N - 2 negs, E = 2 anti - 2N, opened by the black pass.
__device__ __forceinline__ void open_slot(const Int8Sweep& d)
{
    if (d.colour == 0 && blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t N = d.L * d.L;
        d.hist_slot[0] = N;
        d.hist_slot[1] = -2 * N;
    }
}

constexpr int kThreads = 256;
constexpr int kQueue = 96;  // 31 left over and two words a lane

// Words still undecided after two Philox calls wait in a per-warp queue as in the packed kernel;
// an entry is (plane word, undecided sites, h = 2 sites, old target signs).  Their segments are
// already stored as far as decided, so a drained word only turns the bytes of the few sites
// accepted now.
__device__ __forceinline__ void drain_words(const Int8Sweep& d, const PhiloxWordConsts& pc, const uint4* wq, int& qn,
                                            int n, int lane, uint32_t& negs, uint32_t& anti)
{
    uint4 e = make_uint4(0u, 0u, 0u, 0u);
    if (lane < n) e = wq[qn - n + lane];
    qn -= n;
    __syncwarp();  // entries read (and their segments stored) before the next pushes
    const uint32_t thr[2] = {d.t2, d.t4}, sel[1] = {e.z}, ql[1] = {8u * e.x};
    uint32_t und[1] = {e.y}, lt[1] = {0u};
    bitsliced_below<1, 2, 2, 8, true>(und, lt, sel, sel, ql, pc, d.key, thr);
    if (d.colour == 1) {
        negs += __popc(lt[0] & ~e.w) - __popc(lt[0] & e.w);
        anti += 4u * __popc(lt[0]) - 2u * __popc(lt[0] & e.z);
    }
    if (lt[0] != 0u) {
        const unsigned G = (unsigned)(d.L / 64), i = e.x / G, g = e.x - i * G;
        int8_t* p = d.lat + i * d.L + 64 * g + ((i + (unsigned)d.colour) & 1u);
        do {
            const int b = __ffs(lt[0]) - 1;
            p[2 * b] = (int8_t)-p[2 * b];
            lt[0] &= lt[0] - 1u;
        } while (lt[0] != 0u);
    }
}

// L % 64 == 0.  A thread walks a strip of `rows` rows (a divisor of L, even) of one 64-byte
// column of segments, two rows at a time, so that each row is loaded and packed once per strip
// (and the rows beside the strip once more) and two words' Philox calls overlap.  With the
// classes formed byte by byte (about 14 operations a site) the kernel was bound by the ALU pipe
// at 516 flips/ns for every size beyond L2; now 1,263 at L = 65,536, three quarters of what the
// 4 bytes a site that a half-sweep must move allow at the measured copy rate, and 774
// (369 before) at L = 4,096.  Small lattices are bound by the launch: each half-sweep's launch
// overlaps the end of the one before (7.4 us a sweep at L = 64, 12.3 before).
__global__ void __launch_bounds__(kThreads, 2) int8_half_sweep_seg64_kernel(const Int8Sweep d, int rows)
{
    __shared__ uint4 queues[(kThreads / 32) * kQueue];
    const int64_t L = d.L;
    const int G = (int)(L / 64);
    const int lane = threadIdx.x & 31;
    uint4* wq = queues + (threadIdx.x >> 5) * kQueue;
    int qn = 0;
    grid_launch_next();
    const PhiloxWordConsts pc = philox_consts(d.key, 0u, d.sweep, (uint32_t)d.colour);
    const uint32_t thr[2] = {d.t2, d.t4};
    const uint32_t zero2 = (d.t2 == 0u && d.all2 == 0u) ? ~0u : 0u, zero4 = (d.t4 == 0u && d.all4 == 0u) ? ~0u : 0u;
    // at most 2^27 strips (L <= 131,072)
    const int idx = (int)(blockIdx.x * kThreads + threadIdx.x);
    const bool valid = idx < G * (int)(L / rows);  // the votes need the whole warp: a lane past the end keeps nothing
    // a lane past the end counts no words of its own, but does count those that a drain hands it
    const bool counts = valid && d.colour == 1;
    const int strip = valid ? idx / G : 0, g = valid ? idx - strip * G : 0;
    const int64_t i0 = (int64_t)strip * rows;
    grid_wait();
    open_slot(d);
    int8_t* const column = d.lat + 64 * (int64_t)g;
    const int64_t left = g == 0 ? L - 1 : 64 * g - 1, right = g + 1 == G ? 0 : 64 * g + 64;
    uint32_t negs = 0, anti = 0;

    uint4 raw[2][4];               // rows i, i + 1
    uint32_t even[4], odd[4];      // rows i - 1 .. i + 2
    load_segment(column + (i0 == 0 ? L - 1 : i0 - 1) * L, raw[0]);
    pack64(raw[0], even[0], odd[0]);
    load_segment(column + i0 * L, raw[0]);
    pack64(raw[0], even[1], odd[1]);
    for (int64_t i = i0; i < i0 + rows; i += 2) {
        load_segment(column + (i + 1) * L, raw[1]);
        uint4 next[4];
        load_segment(column + (i + 2 == L ? 0 : i + 2) * L, next);
        // the one neighbour of each row outside the segment: column 64g - 1 for targets on even
        // columns (row parity r = 0), 64g + 64 on odd ones
        const bool r0 = ((i + d.colour) & 1) != 0;
        const uint32_t e0 = (uint32_t)(uint8_t)d.lat[i * L + (r0 ? right : left)] >> 7;
        const uint32_t e1 = (uint32_t)(uint8_t)d.lat[(i + 1) * L + (r0 ? left : right)] >> 7;
        pack64(raw[1], even[2], odd[2]);
        pack64(next, even[3], odd[3]);
        uint32_t f[2], und[2], sel[2], ql[2], t[2], same[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bool r = r0 != (k != 0);
            const uint32_t edge = k ? e1 : e0;
            t[k] = r ? odd[k + 1] : even[k + 1];
            same[k] = r ? even[k + 1] : odd[k + 1];
            const uint32_t up = r ? odd[k] : even[k], dn = r ? odd[k + 2] : even[k + 2];
            const uint32_t hz = r ? (same[k] >> 1) | (edge << 31) : (same[k] << 1) | edge;
            uint32_t anti0;
            classify_word(t[k], up, dn, same[k], hz, d.all2, d.all4, zero2, zero4, f[k], und[k], sel[k], anti0);
            if (!valid) und[k] = 0u;
            if (counts) anti += anti0;
            ql[k] = 8u * (uint32_t)((i + k) * G + g);
        }
        // calls 0-1 (planes 0-7) without a test: nearly every word needs both
        bitsliced_below<2, 2, 0, 2, true, false>(und, f, sel, sel, ql, pc, d.key, thr);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            turn64(raw[k], f[k], (r0 != (k != 0)) ? kSpread1 : kSpread0);
            if (valid) {
                uint4* row = reinterpret_cast<uint4*>(column + (i + k) * L);
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    if ((f[k] >> (8 * m)) & 0xFFu) row[m] = raw[k][m];
            }
            if (counts) {
                // the word as decided so far; the drain adds the rest
                negs += __popc(same[k]) + __popc(t[k] ^ f[k]);
                anti += 4u * __popc(f[k]) - 2u * __popc(f[k] & sel[k]);
            }
            const bool pend = und[k] != 0u;
            const uint32_t bal = __ballot_sync(0xffffffffu, pend);
            if (pend)
                wq[qn + __popc(bal & ((1u << lane) - 1u))] = make_uint4(ql[k] >> 3, und[k], sel[k], t[k]);
            qn += __popc(bal);
        }
        while (qn >= 32) {
            __syncwarp();  // pushes and stores visible to the draining lanes
            drain_words(d, pc, wq, qn, 32, lane, negs, anti);
        }
        even[0] = even[2];
        odd[0] = odd[2];
        even[1] = even[3];
        odd[1] = odd[3];
#pragma unroll
        for (int m = 0; m < 4; ++m) raw[0][m] = next[m];
    }
    if (qn > 0) {
        __syncwarp();
        drain_words(d, pc, wq, qn, qn, lane, negs, anti);
    }
    if (d.colour == 1) {
        // a drained word's counts may be negative for the lane that drained it
        block_add_pair(-2ll * (int32_t)negs, 2ll * (int32_t)anti, d.hist_slot);
    }
}

// L % 64 != 0: a plane word is eight consecutive 8-byte chunks in row-major order (the lattice
// has L / 8 chunks a row, each four target sites of either colour), which may lie in
// several rows.  One thread per word: drawn once for its 32 sites instead of once for each of
// its chunks (us a sweep: L = 200 6.2, 8.7 before; 1,000 8.8, 14.4 before; 4,072 41, 94 before).
__global__ void __launch_bounds__(kThreads) int8_half_sweep_chunk8_kernel(const Int8Sweep d)
{
    const int64_t L = d.L;
    const int G = (int)(L / 8), words = (int)(L * L / 64);  // L < 131,072
    grid_launch_next();
    const PhiloxWordConsts pc = philox_consts(d.key, 0u, d.sweep, (uint32_t)d.colour);
    const uint32_t thr[2] = {d.t2, d.t4};
    const uint32_t zero2 = (d.t2 == 0u && d.all2 == 0u) ? ~0u : 0u, zero4 = (d.t4 == 0u && d.all4 == 0u) ? ~0u : 0u;
    uint32_t negs = 0, anti = 0;
    const int word = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const unsigned first = 8u * (unsigned)word;  // chunk, below 2^31
    int64_t i = first / (unsigned)G;
    int g = (int)(first - (unsigned)i * (unsigned)G);
    grid_wait();
    open_slot(d);
    if (word < words) {
        uint64_t cur[8];
        uint32_t t = 0, same = 0, up = 0, dn = 0, hz = 0;
        const int64_t i_first = i;
        const int g_first = g;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int64_t iu = i == 0 ? L - 1 : i - 1, id = i + 1 == L ? 0 : i + 1;
            const bool r = ((i + d.colour) & 1) != 0;
            const int8_t* row = d.lat + i * L;
            const uint2 v = *reinterpret_cast<const uint2*>(row + 8 * g);
            const uint2 u = *reinterpret_cast<const uint2*>(d.lat + iu * L + 8 * g);
            const uint2 w = *reinterpret_cast<const uint2*>(d.lat + id * L + 8 * g);
            cur[c] = (uint64_t)v.y << 32 | v.x;
            // the one neighbour outside the chunk: column 8g - 1 (r = 0) or 8g + 8 (r = 1)
            const int64_t edge_col = r ? (g + 1 == G ? 0 : 8 * g + 8) : (g == 0 ? L - 1 : 8 * g - 1);
            const uint32_t edge = (uint32_t)(uint8_t)row[edge_col] >> 7;
            // four signs of either column parity: even in bits 0-3, odd in bits 8-11
            const uint32_t pv = pack16(v.x, v.y, 0u, 0u), pu = pack16(u.x, u.y, 0u, 0u), pw = pack16(w.x, w.y, 0u, 0u);
            const int st = r ? 8 : 0, ss = 8 - st;
            const uint32_t s4 = (pv >> ss) & 0xFu;
            const uint32_t h4 = r ? (s4 >> 1) | (edge << 3) : ((s4 << 1) & 0xFu) | edge;
            t |= ((pv >> st) & 0xFu) << (4 * c);
            up |= ((pu >> st) & 0xFu) << (4 * c);
            dn |= ((pw >> st) & 0xFu) << (4 * c);
            same |= s4 << (4 * c);
            hz |= h4 << (4 * c);
            if (++g == G) {
                g = 0;
                ++i;
            }
        }
        uint32_t f[1], und[1], sel[1], anti0;
        classify_word(t, up, dn, same, hz, d.all2, d.all4, zero2, zero4, f[0], und[0], sel[0], anti0);
        const uint64_t q = 8ull * (uint64_t)word;
        const uint32_t ql[1] = {(uint32_t)q};
        bitsliced_below<1, 2, 0, 2, false, false>(und, f, sel, sel, ql, pc, d.key, thr);
        bitsliced_below<1, 2, 2, 8>(und, f, sel, sel, ql, pc, d.key, thr);
        i = i_first;
        g = g_first;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint32_t f4 = (f[0] >> (4 * c)) & 0xFu;
            if (f4) {
                const uint32_t spread = ((i + d.colour) & 1) ? kSpread1 : kSpread0;
                // bit 0 / 2 of f4 at bit 7, bit 1 / 3 at bit 23
                const uint32_t x = turn((uint32_t)cur[c], (f4 & 1u) << 7 | (f4 & 2u) << 22, spread);
                const uint32_t y = turn((uint32_t)(cur[c] >> 32), (f4 & 4u) << 5 | (f4 & 8u) << 20, spread);
                *reinterpret_cast<uint2*>(d.lat + i * L + 8 * g) = make_uint2(x, y);
            }
            if (++g == G) {
                g = 0;
                ++i;
            }
        }
        negs = __popc(same) + __popc(t ^ f[0]);
        anti = anti0 + 4u * __popc(f[0]) - 2u * __popc(f[0] & sel[0]);
    }
    if (d.colour == 1) block_add_pair(-2ll * (int32_t)negs, 2ll * (int32_t)anti, d.hist_slot);
}

__global__ void int8_observe_kernel(const int8_t* lat, int64_t L, int64_t* ME)
{
    long long m_acc = 0, e_acc = 0;
    const int64_t N = L * L;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < N;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = idx / L, j = idx - i * L;
        const int s = lat[idx];
        m_acc += s;
        e_acc -= (long long)s * (lat[(i + 1 == L ? 0 : i + 1) * L + j] + lat[i * L + (j + 1 == L ? 0 : j + 1)]);
    }
    block_add_pair(m_acc, e_acc, ME);
}

__global__ void zero_pair_kernel(int64_t* p)
{
    p[0] = 0;
    p[1] = 0;
}

int grid_cap(int64_t work, int threads, int per_sm)
{
    const int64_t want = (work + threads - 1) / threads;
    const int64_t cap = (int64_t)sm_count() * per_sm;
    return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

}  // namespace

cudaError_t launch_int8_init(int8_t* lat, int64_t L, uint64_t key, int start, cudaStream_t s)
{
    int8_init_kernel<<<grid_cap(L * (L / 8), 256, 16), 256, 0, s>>>(lat, L, key, start);
    return cudaGetLastError();
}

cudaError_t launch_int8_half_sweep(int8_t* lat, int64_t L, uint64_t key, uint32_t t2, uint32_t t4, uint32_t all2,
                                   uint32_t all4, uint32_t sweep, int colour, int64_t* hist_slot, cudaStream_t s)
{
    const Int8Sweep d{lat, L, key, t2, t4, all2, all4, sweep, colour, hist_slot};
    if (L % 64 == 0) {
        // the tallest strips (16 rows at most) that still give every SM about 400 of the 512
        // threads it holds.  us a sweep with strips of 2 / 4 / 8 / 16 / 32 rows: L = 2,048: 16.5 /
        // 19.8 / 28 / 43 / 74; L = 4,096: 31 / 27 / 29 / 45 / 75; L = 32,768: 1,230 / 1,035 /
        // 913 / 864 / 872
        const int64_t segments = L * (L / 64), enough = (int64_t)sm_count() * 2 * kThreads * 4 / 5;
        int rows = 2;
        while (rows < 16 && segments / (2 * rows) >= enough) rows *= 2;
        const int64_t grid = (segments / rows + kThreads - 1) / kThreads;
        return launch_following(int8_half_sweep_seg64_kernel, dim3((unsigned)grid), dim3(kThreads), 0, s, d, rows);
    }
    // small blocks, so that a small lattice's words lie on as many SMs as possible.  us a sweep with blocks of
    // 32 / 64 / 128 / 256: L = 200: 6.1 / 6.2 / 6.7 / 9.0; 488: 6.4 / 6.6 / 7.1 / 9.2; 1,000: 8.3 / 8.8 / 9.7 / 13.0; 1,496:
    // 14.2 / 14.0 / 13.8 / 13.9; 2,504: 23.1 / 20.4 / 19.9 / 20.3; 4,072: 43.0 / 41.0 / 40.7 / 42.6
    const int64_t words = L * L / 64;
    const int threads = words < 128ll * sm_count() ? 64 : 128;
    return launch_following(int8_half_sweep_chunk8_kernel, dim3((unsigned)((words + threads - 1) / threads)), dim3(threads),
                            0, s, d);
}

cudaError_t launch_int8_observe(const int8_t* lat, int64_t L, int64_t* ME, cudaStream_t s)
{
    zero_pair_kernel<<<1, 1, 0, s>>>(ME);
    int8_observe_kernel<<<grid_cap(L * L, 256, 8), 256, 0, s>>>(lat, L, ME);
    return cudaGetLastError();
}

}  // namespace ising
