// Sweep of one small or middle-sized bit-packed lattice with its random numbers drawn
// ahead of the update.
//
// A site's uniform U depends only on (seed, sweep, colour, site) and its acceptance
// thresholds T_2, T_4 only on beta, so for every site of every coming half-sweep the two
// decisions U < T_2 and U < T_4 (Sec. 3.1 acceptance rule) can be made before the spins are
// known.  They are drawn as two 32-bit masks per plane word, by all SMs at once and over many
// sweeps; what is left of a half-sweep is about a dozen logic operations a word:
//
//   flip = (n >= 2) | (n odd ? U < T_2 : U < T_4),   n = anti-aligned neighbours (0..4),
//
// which a few CTAs do sweep after sweep with the spins in registers.  Without that split a
// half-sweep of a lattice this small is a chain of Philox rounds that only its own words
// can fill (one CTA) or a launch of its own (the tiled kernel); both leave the GPU idle.
//
// One launch does both halves for consecutive chunks of sweeps: its first CTAs update a tile
// of rows each through chunk k, from masks the launch before drew, and then join the other
// CTAs, which draw the masks of chunk k + 1 into the other buffer.  No CTA waits for
// another: a tile of a lattice of several tiles carries `halo` extra rows above and below its
// own, enough for the whole chunk (one row on each side goes stale per half-sweep), reads
// them from a copy of the planes that no CTA of the launch writes, and writes its own rows
// to the other copy.
#include <algorithm>

#include "ising_internal.cuh"
#include "philox.cuh"
#include "sweep_packed_kernel.cuh"

namespace ising {
namespace {

using sweep::bulk_copy_g2s;
using sweep::fence_mbarrier_init;
using sweep::fence_proxy_async_smem;
using sweep::mbar_expect_tx;
using sweep::mbar_init;
using sweep::mbar_wait_bounded;

constexpr int kStrips = 256;         // threads that hold strips of a tile; as many again count
constexpr int kNT = 2 * kStrips + 32;  // (M, E), and a warp fetches the masks.  One CTA per SM
constexpr int kWarps = kNT / 32;
constexpr int kMaxChunk = 1024;     // sweeps per launch (their counts are kept in shared memory)
constexpr int kRingBytes = 128 * 1024;  // masks of the coming half-sweeps, staged in shared memory
constexpr int kMaxSlots = 16;
constexpr int kMaxStrip = 16;       // rows of a thread's strip at most
constexpr int kItemWords = 128;     // plane words of one drawing step of a warp: four a lane

// Words still undecided after two Philox calls, per warp.
struct DrawQueue {
    uint4 e[kItemWords];     // undecided against T_2, against T_4, below T_2 so far, below T_4
    uint32_t at[kItemWords]; // word
};

struct SharedAhead {
    alignas(128) unsigned char ring[kRingBytes];
    uint64_t full[kMaxSlots];         // a ring slot's masks have arrived
    uint64_t empty[kMaxSlots];        // every warp has read them
    DrawQueue queue[kWarps];
    uint32_t planes[3][kMaxStrip * kStrips];  // the tile's spins, word of thread t's k-th row at [k * kStrips + t]:
                                              // black after even and after odd sweeps, white
    uint32_t sums[2 * kMaxChunk];     // (up spins, anti-aligned bonds) of the tile's own rows after each sweep
};

// One plane of a bit-sliced comparison walked from the least significant plane up: R the
// random plane, K the threshold's bit as a mask.  lt (U < T on the planes seen) and eq (equal
// on all of them) are one three-input operation each, as the planes below only matter
// where this one ties.
__device__ __forceinline__ void compare_plane(uint32_t R, uint32_t K, uint32_t& lt, uint32_t& eq)
{
    lt = (~R & K) | (~R & lt) | (K & lt);
    eq = eq & ~(R ^ K);
}

__device__ __forceinline__ uint32_t plane_mask(uint32_t t, int plane) { return (uint32_t)((int32_t)(t << plane) >> 31); }

// Draws the acceptance masks of words word0 + lane + 32 j (j < G) below `words` of one
// half-sweep into out[word] = (U < T_2, U < T_4).  Two calls (planes 7..4, then 3..0) are drawn
// for every word: they decide about 78 % of the words for all 32 sites and both thresholds;
// the others finish from the warp's queue, a word per lane.
template <int G>
__device__ void draw_words(const AheadLattice& d, uint32_t sweep, int colour, int word0, uint2* __restrict__ out,
                           DrawQueue& q, int lane)
{
    const PhiloxWordConsts pc = philox_consts(d.key, 0u, sweep, (uint32_t)colour);
    uint32_t base[G], lt2[G], lt4[G], eq2[G], eq4[G];
#pragma unroll
    for (int j = 0; j < G; ++j) {
        base[j] = 8u * (uint32_t)(word0 + lane + 32 * j) ^ pc.x0k;
        lt2[j] = lt4[j] = 0u;
        eq2[j] = eq4[j] = ~0u;
    }
#pragma unroll
    for (int c = 1; c >= 0; --c) {
        uint32_t o[G][4];
        philox_calls<G>(base, (uint32_t)c, pc, d.key, o);
#pragma unroll
        for (int m = 3; m >= 0; --m) {
            const uint32_t K2 = plane_mask(d.t2, 4 * c + m), K4 = plane_mask(d.t4, 4 * c + m);
#pragma unroll
            for (int j = 0; j < G; ++j) {
                compare_plane(o[j][m], K2, lt2[j], eq2[j]);
                compare_plane(o[j][m], K4, lt4[j], eq4[j]);
            }
        }
    }
    int qn = 0;
#pragma unroll
    for (int j = 0; j < G; ++j) {
        const int word = word0 + lane + 32 * j;
        const bool valid = word < d.words;
        lt2[j] |= d.all2;  // a threshold of 2^32 accepts every uniform
        lt4[j] |= d.all4;
        eq2[j] &= ~d.all2;
        eq4[j] &= ~d.all4;
        const bool pend = valid && (eq2[j] | eq4[j]) != 0u;
        if (valid && !pend) out[word] = make_uint2(lt2[j], lt4[j]);
        const uint32_t bal = __ballot_sync(0xffffffffu, pend);
        if (pend) {
            const int slot = qn + __popc(bal & ((1u << lane) - 1u));
            q.e[slot] = make_uint4(eq2[j], eq4[j], lt2[j], lt4[j]);
            q.at[slot] = (uint32_t)word;
        }
        qn += __popc(bal);
    }
    __syncwarp();
    for (int first = 0; first < qn; first += 32) {
        const bool act = first + lane < qn;
        uint4 e = make_uint4(0u, 0u, 0u, 0u);
        uint32_t at = 0u;
        if (act) {
            e = q.e[first + lane];
            at = q.at[first + lane];
        }
        const uint32_t b1[1] = {8u * at ^ pc.x0k};
        for (int c = 2; c < 8 && __any_sync(0xffffffffu, (e.x | e.y) != 0u); ++c) {
            uint32_t o[1][4];
            philox_calls<1>(b1, (uint32_t)c, pc, d.key, o);
            uint32_t l2 = 0u, l4 = 0u, t2 = e.x, t4 = e.y;
#pragma unroll
            for (int m = 3; m >= 0; --m) {
                compare_plane(o[0][m], plane_mask(d.t2, 4 * c + m), l2, t2);
                compare_plane(o[0][m], plane_mask(d.t4, 4 * c + m), l4, t4);
            }
            e.z |= e.x & l2;
            e.w |= e.y & l4;
            e.x = t2;
            e.y = t4;
        }
        // a site still tied after all 32 planes has U equal to its threshold: not below
        if (act) out[at] = make_uint2(e.z, e.w);
    }
    __syncwarp();  // the queue is read before the next step fills it
}

// Drawing step `item` of a chunk: steps run over the chunk's half-sweeps, each in blocks of
// 32 G words.  The step that holds a sweep's first words also opens the sweep's (M, E) entry
// when several tiles will add their counts to it.
template <int G>
__device__ __forceinline__ void draw_item(const AheadLattice& d, uint32_t sweep0, int item, uint2* masks, DrawQueue& q,
                                          int lane)
{
    const int per = (d.words + 32 * G - 1) / (32 * G);
    const int hs = item / per, word0 = (item - hs * per) * 32 * G;
    const uint32_t sweep = sweep0 + (uint32_t)(hs >> 1);
    if (d.tiles > 1 && (hs & 1) == 0 && word0 == 0 && lane == 0) {
        const int64_t N = (int64_t)d.L * d.L;
        d.hist[2 * (int64_t)sweep] = -N;
        d.hist[2 * (int64_t)sweep + 1] = -2 * N;
    }
    draw_words<G>(d, sweep, hs & 1, word0, masks + (size_t)hs * d.words, q, lane);
}

// Named barriers of a tile's `threads` threads: of those that hold strips and those that count,
// at the end of a black half-sweep (the counting ones only arrive) and of a white one; and of
// all parts of the CTA.
constexpr int kBarBlack = 1, kBarWhite = 2, kBarTile = 3;

template <int ID>
__device__ __forceinline__ void tile_barrier(int threads)
{
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "r"(threads) : "memory");
}

template <int ID>
__device__ __forceinline__ void tile_arrive(int threads)
{
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "r"(threads) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sweep::smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void mbar_inval(uint64_t* bar)
{
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(sweep::smem_addr(bar)) : "memory");
}

// The neighbours of a thread's strip of K rows of one word column in the source colour:
// the words above and below the strip, and per row the word of horizontal neighbours.
template <int K>
struct StripNeighbours {
    uint32_t up, dn, hz[K];
};

// One colour's half of a sweep for a strip: t its target words, s its source words.
// Anti-aligned bits of the two vertical and of the two horizontal neighbours: the low bits of
// their sums do not depend on the target, and n >= 2 is two in one pair or one in each, so a
// word takes nine three-input operations.
template <int K>
__device__ __forceinline__ void update_strip(uint32_t (&t)[K], const uint32_t (&s)[K], const StripNeighbours<K>& nb,
                                             const uint2 (&m)[K])
{
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t u = k == 0 ? nb.up : s[k - 1], w = k == K - 1 ? nb.dn : s[k + 1];
        const uint32_t s1 = s[k] ^ nb.hz[k], both = (u ^ w) & s1, odd = u ^ w ^ s1;
        const uint32_t c0 = (t[k] ^ u) & (t[k] ^ w), c1 = (t[k] ^ s[k]) & (t[k] ^ nb.hz[k]);
        t[k] ^= (both | c0 | c1) | (odd & m[k].x) | (~odd & m[k].y);
    }
}

// Up spins of both colours and anti-aligned bonds of rows lo .. hi - 1 of a strip (each bond has
// one white end): n = odd + 2 (both + c0 + c1) for every white site.
template <int K>
__device__ __forceinline__ void count_strip(const uint32_t (&t)[K], const uint32_t (&s)[K],
                                            const StripNeighbours<K>& nb, int lo, int hi, uint32_t& ups,
                                            uint32_t& anti)
{
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t u = k == 0 ? nb.up : s[k - 1], w = k == K - 1 ? nb.dn : s[k + 1];
        const uint32_t s1 = s[k] ^ nb.hz[k], both = (u ^ w) & s1, odd = u ^ w ^ s1;
        const uint32_t c0 = (t[k] ^ u) & (t[k] ^ w), c1 = (t[k] ^ s[k]) & (t[k] ^ nb.hz[k]);
        const uint32_t keep = k >= lo && k < hi ? ~0u : 0u;
        ups += __popc(s[k] & keep) + __popc(t[k] & keep);
        anti += __popc(odd & keep) + 2u * __popc((both ^ c0 ^ c1) & keep) +
                4u * __popc(((both & c0) | (both & c1) | (c0 & c1)) & keep);
    }
}

// Where a tile lies and how its masks are staged: slots of `sps` sweeps, each half-sweep's
// masks the tile's rows one after the other.
struct TileAt {
    int first;             // its first row on the torus, 0 .. L - 1
    int held, before;      // rows it holds; of them up to the torus's seam
    uint32_t half_bytes;   // masks of one half-sweep
    int sps, slots;
};

template <int K>
__device__ __forceinline__ TileAt tile_at(const AheadLattice& d, int tile)
{
    TileAt a;
    a.first = d.tiles == 1 ? 0 : tile * d.rows - d.halo;
    if (a.first < 0) a.first += d.L;
    a.held = d.groups * K;
    a.before = min(a.held, d.L - a.first);
    a.half_bytes = (uint32_t)(a.held * d.W) * 8u;
    a.sps = max(1, (int)(kRingBytes / 4 / (2 * a.half_bytes)));
    a.slots = min(kMaxSlots, (int)(kRingBytes / (2 * a.half_bytes * a.sps)));
    return a;
}

// The fetching warp's part of a tile: one lane keeps the ring filled with the masks of the
// coming sweeps by bulk copies (a contiguous run of rows per half-sweep, two where the tile
// wraps round the torus; of a lattice of one tile all of a slot's half-sweeps at once).
__device__ __forceinline__ void fetch_masks(const AheadLattice& d, const AheadStep& st, const TileAt& a, SharedAhead& sh)
{
    const int n = st.upd_n;
    uint32_t phase = 1;  // of the slots' empty barriers: the first round finds them free
    for (int s = 0, slot = 0; s < n; s += a.sps) {
        if (s >= a.sps * a.slots && !mbar_wait_bounded(&sh.empty[slot], phase, kWaitLimitCycles)) {
            atomicExch(d.status, kStatusTimeout);
            return;
        }
        const int now = min(a.sps, n - s);
        unsigned char* dst = sh.ring + (size_t)slot * a.sps * 2 * a.half_bytes;
        const uint2* src = d.masks[st.upd_buf] + (size_t)(2 * s) * d.words;
        fence_proxy_async_smem();
        mbar_expect_tx(&sh.full[slot], 2u * (uint32_t)now * a.half_bytes);
        if (d.tiles == 1) {
            bulk_copy_g2s(dst, src, 2u * (uint32_t)now * a.half_bytes, &sh.full[slot]);
        } else {
            const uint32_t head = (uint32_t)(a.before * d.W) * 8u;
            for (int h = 0; h < 2 * now; ++h) {
                bulk_copy_g2s(dst, src + (size_t)a.first * d.W, head, &sh.full[slot]);
                if (head < a.half_bytes) bulk_copy_g2s(dst + head, src, a.half_bytes - head, &sh.full[slot]);
                dst += a.half_bytes;
                src += d.words;
            }
        }
        if (++slot == a.slots) {
            slot = 0;
            phase ^= 1u;
        }
    }
}

// The part of a tile that a thread of the first two groups works on: the words of column tx in
// the K rows from row ty * K of the tile.  Neighbour words' places in a plane's buffer.
struct StripAt {
    int t;                       // the strip's first word
    int above, below, left, right;  // the words above and below the strip, and beside its first row
    int row;                     // its first row in the tile
};

template <int K>
__device__ __forceinline__ StripAt strip_at(const AheadLattice& d, int t)
{
    StripAt p;
    const int W = d.W, ty = t / W, tx = t - ty * W;
    const bool whole = d.tiles == 1;
    p.t = t;
    p.row = ty * K;
    // where a tile with halo rows ends, any word will do: those rows are stale by then and never
    // reach an own row
    p.above = ty > 0 ? (K - 1) * kStrips + t - W : (whole ? (K - 1) * kStrips + (d.groups - 1) * W + tx : t);
    p.below = ty + 1 < d.groups ? t + W : (whole ? tx : t);
    p.right = tx + 1 == W ? t - tx : t + 1;
    p.left = tx == 0 ? t + W - 1 : t - 1;
    return p;
}

// The neighbours of a strip with source words s, from the source plane's buffer.  Strips start
// on even rows: row k's horizontal neighbour is to the right iff k + COLOUR is odd.
template <int K, int COLOUR>
__device__ __forceinline__ StripNeighbours<K> load_neighbours(const uint32_t* plane, const StripAt& p,
                                                              const uint32_t (&s)[K])
{
    StripNeighbours<K> nb;
    nb.up = plane[p.above];
    nb.dn = plane[p.below];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const bool right = ((k + COLOUR) & 1) != 0;
        const uint32_t side = plane[(right ? p.right : p.left) + k * kStrips];
        nb.hz[k] = right ? __funnelshift_r(s[k], side, 1) : __funnelshift_l(side, s[k], 1);
    }
    return nb;
}

template <int K>
__device__ __forceinline__ void load_strip(const uint32_t* plane, const StripAt& p, uint32_t (&v)[K])
{
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = plane[p.t + k * kStrips];
}

template <int K>
__device__ __forceinline__ void store_strip(uint32_t* plane, const StripAt& p, const uint32_t (&v)[K])
{
#pragma unroll
    for (int k = 0; k < K; ++k) plane[p.t + k * kStrips] = v[k];
}

// Updates one tile through the chunk's sweeps.  A CTA's warps have three parts:
//  - the first `active` threads hold the tile's spins, a strip each and both colours, in
//    registers; they go through shared memory only for the neighbours above, below and beside,
//    with one barrier per half-sweep;
//  - as many threads of the second group count the own rows' (M, E) of a sweep while the
//    first already runs the next one: they take the words from shared memory between the
//    barriers that end the sweep and the next black half-sweep (the black plane has a second
//    buffer for that);
//  - a lane of the last warp keeps the ring of masks filled (fetch_masks).
template <int K>
__device__ void update_tile(const AheadLattice& d, const AheadStep& st, int tile, SharedAhead& sh)
{
    const int W = d.W, L = d.L, active = d.groups * W;
    const int threads = (active + 31) & ~31, part = threadIdx.x / kStrips, tid = threadIdx.x % kStrips;
    const bool fetcher = part == 2;
    if (tid >= threads && !fetcher) return;
    const TileAt a = tile_at<K>(d, tile);
    const int n = st.upd_n, everyone = 2 * threads + 32;
    if (threadIdx.x == 0 && !st.alone) {
        for (int k = 0; k < a.slots; ++k) {
            mbar_init(&sh.full[k], 1);
            mbar_init(&sh.empty[k], (uint32_t)threads / 32u);
        }
        fence_mbarrier_init();
    }
    const bool on = tid < active;
    const StripAt p = strip_at<K>(d, on ? tid : active - 1);  // a lane past the end follows the last one and keeps nothing
    const int column = p.t % W;
    // own rows of the strip: k with lo <= k < hi
    const bool whole = d.tiles == 1;
    const int lo = !on ? K : (whole ? 0 : max(0, d.halo - p.row));
    const int hi = !on ? 0 : (whole ? K : min(d.halo + min(d.rows, L - tile * d.rows) - p.row, K));
    auto word_at = [&](int k) {  // row k's word in the planes
        int i = a.first + p.row + k;
        if (i >= L) i -= L;
        return (size_t)i * W + column;
    };
    uint32_t b[K], w[K];
    if (part == 0) {
        const uint32_t* src = st.src < 0 ? d.home : d.copy + (size_t)st.src * 2 * d.words;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const size_t at = word_at(k);
            b[k] = src[at];
            w[k] = src[d.words + at];
        }
        if (on) store_strip<K>(sh.planes[2], p, w);
        for (int k = tid; k < 2 * n; k += threads) sh.sums[k] = 0u;
    }
    tile_barrier<kBarTile>(everyone);

    if (part == 0) {
        bool dead = false;  // a wait ran out: the launch reports it and its results are not used
        int slot = 0;
        uint32_t phase = 0;
        const unsigned char* mp = sh.ring + (size_t)(p.row * W + column) * 8;
        auto load_masks = [&](uint2 (&m)[K]) {
#pragma unroll
            for (int k = 0; k < K; ++k) m[k] = *reinterpret_cast<const uint2*>(mp + k * (W * 8));
            mp += a.half_bytes;
        };
        auto one_sweep = [&](uint32_t* black) {
            uint2 m[K];
            {
                const StripNeighbours<K> nb = load_neighbours<K, 0>(sh.planes[2], p, w);
                load_masks(m);
                update_strip<K>(b, w, nb, m);
                if (on) store_strip<K>(black, p, b);
                tile_barrier<kBarBlack>(2 * threads);
            }
            {
                const StripNeighbours<K> nb = load_neighbours<K, 1>(black, p, b);
                load_masks(m);
                update_strip<K>(w, b, nb, m);
                if (on) store_strip<K>(sh.planes[2], p, w);
                tile_barrier<kBarWhite>(2 * threads);
            }
        };
        const int per_slot = st.alone ? n : a.sps;
        int odd = 0;  // sweeps done, modulo 2: the black buffer in use
        for (int s = 0; s < n; s += per_slot) {
            if (!st.alone && !dead && !mbar_wait_bounded(&sh.full[slot], phase, kWaitLimitCycles)) {
                dead = true;
                atomicExch(d.status, kStatusTimeout);
            }
            int left = min(per_slot, n - s);
            if (odd) {
                one_sweep(sh.planes[1]);
                odd = 0;
                --left;
            }
            for (; left >= 2; left -= 2) {
                one_sweep(sh.planes[0]);
                one_sweep(sh.planes[1]);
            }
            if (left) {
                one_sweep(sh.planes[0]);
                odd = 1;
            }
            if (!st.alone) {
                // this warp has read the slot
                __syncwarp();
                if ((tid & 31) == 0) mbar_arrive(&sh.empty[slot]);
                if (++slot == a.slots) {
                    slot = 0;
                    phase ^= 1u;
                    mp -= (size_t)a.slots * a.sps * 2 * a.half_bytes;
                }
            }
        }
        uint32_t* dst = st.dst < 0 ? d.home : d.copy + (size_t)st.dst * 2 * d.words;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k >= lo && k < hi) {
                const size_t at = word_at(k);
                dst[at] = b[k];
                dst[d.words + at] = w[k];
            }
    } else if (part == 1) {
        tile_arrive<kBarBlack>(2 * threads);
        for (int s = 0; s < n; ++s) {
            tile_barrier<kBarWhite>(2 * threads);
            const uint32_t* black = sh.planes[s & 1];
            load_strip<K>(sh.planes[2], p, w);
            load_strip<K>(black, p, b);
            const StripNeighbours<K> nb = load_neighbours<K, 1>(black, p, b);
            if (s + 1 < n) tile_arrive<kBarBlack>(2 * threads);
            uint32_t ups = 0, anti = 0;
            if (whole) {
                count_strip<K>(w, b, nb, 0, K, ups, anti);
                if (!on) ups = anti = 0u;
            } else {
                count_strip<K>(w, b, nb, lo, hi, ups, anti);
            }
            // a lane has at most 64 K <= 1024 up spins and 128 K <= 2048 bonds: a warp's sums fit
            // 16 bits for strips of up to 8 rows
            uint32_t u, v;
            if (K <= 8) {
                const uint32_t both = __reduce_add_sync(0xffffffffu, ups | (anti << 16));
                u = both & 0xffffu;
                v = both >> 16;
            } else {
                u = __reduce_add_sync(0xffffffffu, ups);
                v = __reduce_add_sync(0xffffffffu, anti);
            }
            if ((tid & 31) == 0) {
                atomicAdd(&sh.sums[2 * s], u);
                atomicAdd(&sh.sums[2 * s + 1], v);
            }
        }
    } else if (threadIdx.x == 2 * kStrips && !st.alone) {
        fetch_masks(d, st, a, sh);
    }
    tile_barrier<kBarTile>(everyone);
    if (part == 1) {
        const int64_t N = (int64_t)L * L;
        for (int s = tid; s < n; s += threads) {
            int64_t* entry = d.hist + 2 * (int64_t)(st.upd_sweep + (uint32_t)s);
            const int64_t M = 2 * (int64_t)sh.sums[2 * s], E = 2 * (int64_t)sh.sums[2 * s + 1];
            if (whole) {
                entry[0] = M - N;
                entry[1] = E - 2 * N;
            } else {
                atomicAdd(reinterpret_cast<unsigned long long*>(entry), (unsigned long long)M);
                atomicAdd(reinterpret_cast<unsigned long long*>(entry + 1), (unsigned long long)E);
            }
        }
    }
    if (threadIdx.x == 0 && !st.alone)
        for (int k = 0; k < a.slots; ++k) {
            mbar_inval(&sh.full[k]);
            mbar_inval(&sh.empty[k]);
        }
    // the next tile clears the sums and sets up the barriers again
    tile_barrier<kBarTile>(everyone);
}

// K: rows of a thread's strip.
template <int K>
__global__ void __launch_bounds__(kNT, 1) ahead_kernel(const __grid_constant__ AheadLattice d, const AheadStep st)
{
    extern __shared__ __align__(16) unsigned char smem_ahead[];
    SharedAhead& sh = *reinterpret_cast<SharedAhead*>(smem_ahead);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (st.alone) {
        // a short run of a lattice of one tile: this CTA draws the masks it needs itself, into
        // the ring's slots
        const int items = 2 * st.upd_n * ((d.words + 31) / 32);
        for (int item = warp; item < items; item += kWarps)
            draw_item<1>(d, st.upd_sweep, item, reinterpret_cast<uint2*>(sh.ring), sh.queue[warp], lane);
        __syncthreads();
    }
    if (st.upd_n > 0)
        for (int tile = (int)blockIdx.x; tile < d.tiles; tile += (int)gridDim.x) update_tile<K>(d, st, tile, sh);
    if (st.fill >= 0) {
        // the first launch of a call: the copy of the planes that the first update reads
        const size_t total = 2 * (size_t)d.words;
        for (size_t k = (size_t)blockIdx.x * kNT + threadIdx.x; k < total; k += (size_t)gridDim.x * kNT)
            d.copy[(size_t)st.fill * total + k] = d.home[k];
    }
    // the other buffer's ticket is the next launch's, and this launch's own is the next
    // call's once nothing is drawn any more
    if (!st.alone && blockIdx.x == 0 && threadIdx.x == 0) {
        d.ticket[st.gen_buf ^ 1] = 0;
        if (st.gen_n == 0) d.ticket[st.gen_buf] = 0;
    }
    if (st.gen_n > 0) {
        const int items = 2 * st.gen_n * ((d.words + kItemWords - 1) / kItemWords);
        for (;;) {
            int item = 0;
            if (lane == 0) item = atomicAdd(&d.ticket[st.gen_buf], 1);
            item = __shfl_sync(0xffffffffu, item, 0);
            if (item >= items) break;
            draw_item<4>(d, st.gen_sweep, item, d.masks[st.gen_buf], sh.queue[warp], lane);
        }
    }
}

template <int K>
cudaError_t launch_k(const AheadLattice& d, const AheadStep& st, int grid, cudaStream_t s)
{
    ahead_kernel<K><<<grid, kNT, sizeof(SharedAhead), s>>>(d, st);
    return cudaGetLastError();
}

cudaError_t launch_step(const AheadLattice& d, const AheadStep& st, cudaStream_t s)
{
    const int64_t items = 2 * (int64_t)st.gen_n * ((d.words + kItemWords - 1) / kItemWords);
    const int64_t want = (st.upd_n > 0 ? d.tiles : 0) + (items + kWarps - 1) / kWarps;
    const int64_t grid = std::min<int64_t>(sm_count(), std::max<int64_t>(want, 1));
    switch (d.strip) {
    case 2:
        return launch_k<2>(d, st, (int)grid, s);
    case 4:
        return launch_k<4>(d, st, (int)grid, s);
    case 8:
        return launch_k<8>(d, st, (int)grid, s);
    default:
        return launch_k<16>(d, st, (int)grid, s);
    }
}

}  // namespace

int ahead_max_L() { return 8192; }

AheadPlan ahead_plan(int64_t L)
{
    AheadPlan p;
    const int W = (int)(L / 64);
    if (L < 64 || L % 64 || L > ahead_max_L()) return p;
    const int64_t words = L * W, per_sweep = words * 2 * (int64_t)sizeof(uint2);
    if (L <= 320) {
        // one tile: the whole lattice in one CTA, two, four or eight rows a thread
        p.strip = 2;
        while (words > (int64_t)p.strip * kStrips) p.strip *= 2;
        p.groups = (int)L / p.strip;
        p.rows = (int)L;
        p.halo = 0;
        p.tiles = 1;
        p.chunk = (int)std::min<int64_t>(kMaxChunk, (8ll << 20) / per_sweep);
    } else {
        p.strip = L <= 1024 ? 4 : (L <= 2048 ? 8 : 16);
        p.groups = kStrips / W;
        const int held = p.groups * p.strip;  // rows a CTA holds
        p.chunk = std::min(16, held / 8);
        p.halo = 2 * p.chunk;
        p.rows = held - 2 * p.halo;
        p.tiles = (int)((L + p.rows - 1) / p.rows);
    }
    p.mask_bytes = per_sweep * p.chunk;
    p.copy_bytes = p.tiles > 1 ? 2 * 2 * words * (int64_t)sizeof(uint32_t) : 0;
    return p;
}

cudaError_t ahead_configure(const AheadPlan& p)
{
    const void* k = p.strip == 2   ? (const void*)ahead_kernel<2>
                    : p.strip == 4 ? (const void*)ahead_kernel<4>
                    : p.strip == 8 ? (const void*)ahead_kernel<8>
                                   : (const void*)ahead_kernel<16>;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SharedAhead));
}

// Up to two drawing steps of 32 words for each warp: a few microseconds less than a launch for
// the drawing alone.
bool ahead_alone(const AheadLattice& d, int64_t n)
{
    return d.tiles == 1 && n <= kWarps && 2 * n * ((d.words + 31) / 32) <= 2 * kWarps;
}

cudaError_t launch_ahead_sweeps(const AheadLattice& d, int chunk, uint32_t sweep, int64_t n, cudaStream_t s)
{
    AheadStep st;
    st.upd_n = st.gen_n = 0;
    st.upd_buf = st.gen_buf = 0;
    st.src = st.dst = st.fill = -1;
    st.alone = 0;
    if (ahead_alone(d, n)) {
        st.alone = 1;
        st.upd_sweep = sweep;
        st.upd_n = (int)n;
        return launch_step(d, st, s);
    }
    // chunk k is drawn into buffer k & 1 by the launch that updates chunk k - 1.  Of a lattice
    // of one tile the first chunk is short, as nothing is updated while it is drawn.
    int64_t drawn = 0, updated = 0;
    int in_flight = 0, k = 0;
    while (updated < n) {
        int next = (int)std::min<int64_t>(n - drawn, drawn == 0 && d.tiles == 1 ? std::min(chunk, 64) : chunk);
        st.upd_sweep = sweep + (uint32_t)updated;
        st.upd_n = in_flight;
        st.upd_buf = (k & 1) ^ 1;
        st.gen_sweep = sweep + (uint32_t)drawn;
        st.gen_n = next;
        st.gen_buf = k & 1;
        if (d.tiles > 1) {
            st.fill = k == 0 ? 0 : -1;
            st.src = (k & 1) ^ 1;
            st.dst = updated + in_flight == n ? -1 : (k & 1);
        }
        cudaError_t e = launch_step(d, st, s);
        if (e != cudaSuccess) return e;
        updated += in_flight;
        drawn += next;
        in_flight = next;
        ++k;
    }
    return cudaSuccess;
}

}  // namespace ising
