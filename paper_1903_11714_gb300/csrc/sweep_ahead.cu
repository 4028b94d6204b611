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
// to the other copy.  Small cubes go the same way, with slices in the place of rows.
#include <algorithm>
#include <type_traits>

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
constexpr int kMaxBatchChunk = 32;
constexpr int kMaxStrip = 16;       // rows of a thread's strip at most
constexpr int kItemWords = 128;     // plane words of one drawing step of a warp: four a lane

// Words with sites still undecided, per warp: the next call each needs is in the entry, so that
// a drain draws one call for 32 words that all need it.  31 may be left over when the words of a
// pair of lanes' steps are pushed.
constexpr int kQueueWords = 31 + 2 * 32 + 1;
struct DrawQueue {
    uint4 e[kQueueWords];    // undecided against T_2, against T_4, below T_2 so far, below T_4
    uint2 at[kQueueWords];   // lattice << kWordBits | word; half-sweep of the chunk << 3 | next call
};
constexpr int kWordBits = 20;  // a plane has at most 2^20 words (L = 8,192)
constexpr uint32_t kWordMask = (1u << kWordBits) - 1u;

struct SharedAhead {
    alignas(128) unsigned char ring[kRingBytes];
    uint64_t full[kMaxSlots];         // a ring slot's masks have arrived
    uint64_t empty[kMaxSlots];        // every warp has read them
    DrawQueue queue[kWarps];
    uint32_t planes[3][kMaxStrip * kStrips];  // the tile's spins, word of thread t's k-th row at [k * kStrips + t]:
                                              // black after even and after odd sweeps, white
    union {
        uint4 bits[16];               // the thresholds' bits as masks: [c] T_2's in call c's planes, [8 + c] T_4's
        struct {                      // batches: the tile's lattice and what to do with it
            AheadLattice lattice;
            AheadStep step;
        } now;
    };
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

// What drawing needs of a lattice.
struct DrawLattice {
    uint64_t key;
    uint32_t t2, t4, all2, all4;
    int words;
    uint32_t sweep0;   // the chunk's first sweep
    uint2* masks;      // of half-sweep hs at hs * words: (U < T_2, U < T_4)
};

// A drawing warp's queue.
struct DrawState {
    DrawQueue* q;
    int qn;            // entries queued (the same in every lane)
    int lane;
};

// One call for the top n queue entries, a word per lane; words still undecided go back.
// `lattice` gives an entry's lattice, `bits` the thresholds' bits of a call's four planes.
template <typename Lattice, typename Bits>
__device__ __forceinline__ void drain_draws(DrawState& w, int n, Lattice lattice, Bits bits)
{
    const bool act = w.lane < n;
    uint4 e = make_uint4(0u, 0u, 0u, 0u);
    uint2 at = make_uint2(0u, 2u);
    if (act) {
        e = w.q->e[w.qn - n + w.lane];
        at = w.q->at[w.qn - n + w.lane];
    }
    w.qn -= n;
    __syncwarp();  // entries read before any goes back
    const uint32_t word = at.x & kWordMask, c = at.y & 7u, hs = at.y >> 3;
    const DrawLattice d = lattice((int)(at.x >> kWordBits));
    const PhiloxWordConsts pc = philox_consts(d.key, 0u, d.sweep0 + (hs >> 1), hs & 1u);
    const uint32_t base[1] = {8u * word ^ pc.x0k};
    uint32_t o[1][4];
    philox_calls<1>(base, c, pc, d.key, o);
    uint32_t l2 = 0u, l4 = 0u, e2 = e.x, e4 = e.y;
    uint4 b2, b4;
    bits(d, c, b2, b4);
    compare_plane(o[0][3], b2.w, l2, e2);
    compare_plane(o[0][2], b2.z, l2, e2);
    compare_plane(o[0][1], b2.y, l2, e2);
    compare_plane(o[0][0], b2.x, l2, e2);
    compare_plane(o[0][3], b4.w, l4, e4);
    compare_plane(o[0][2], b4.z, l4, e4);
    compare_plane(o[0][1], b4.y, l4, e4);
    compare_plane(o[0][0], b4.x, l4, e4);
    e.z |= e.x & l2;
    e.w |= e.y & l4;
    // a site still tied after all 32 planes has U equal to min(T, 2^32 - 1): below only if T = 2^32
    if (c == 7u) {
        e.z |= e2 & d.all2;
        e.w |= e4 & d.all4;
    }
    const bool pend = (e2 | e4) != 0u && c < 7u;
    if (act && !pend) d.masks[(size_t)hs * d.words + word] = make_uint2(e.z, e.w);
    const uint32_t bal = __ballot_sync(0xffffffffu, pend);
    if (pend) {
        const int slot = w.qn + __popc(bal & ((1u << w.lane) - 1u));
        w.q->e[slot] = make_uint4(e2, e4, e.z, e.w);
        w.q->at[slot] = make_uint2(at.x, at.y + 1u);
    }
    w.qn += __popc(bal);
}

// Draws words word0 + lane + 32 j (j < G) of one half-sweep (FULL: all of them exist).  Two
// calls (planes 7..4, then 3..0) for every word, side by side: they decide about 78 % of the
// words for all 32 sites and both thresholds; the others finish from the warp's queue, a word per
// lane.  K2, K4: the thresholds' bits of the first eight planes as masks.
template <int G, bool FULL, typename Lattice, typename Bits, typename Then>
__device__ __forceinline__ void draw_words(DrawState& w, const DrawLattice& d, int index, const PhiloxWordConsts& pc, int hs,
                                           int word0, const uint32_t (&K2)[8], const uint32_t (&K4)[8], Lattice lattice,
                                           Bits bits, Then then)
{
    uint32_t base[G], lt2[G], lt4[G], eq2[G], eq4[G];
#pragma unroll
    for (int j = 0; j < G; ++j) {
        base[j] = 8u * (uint32_t)(word0 + w.lane + 32 * j) ^ pc.x0k;
        lt2[j] = lt4[j] = 0u;
        eq2[j] = eq4[j] = ~0u;
    }
#pragma unroll
    for (int c = 1; c >= 0; --c) {
        uint32_t o[G][4];
        philox_calls<G>(base, (uint32_t)c, pc, d.key, o);
#pragma unroll
        for (int m = 3; m >= 0; --m)
#pragma unroll
            for (int j = 0; j < G; ++j) {
                compare_plane(o[j][m], K2[4 * c + m], lt2[j], eq2[j]);
                compare_plane(o[j][m], K4[4 * c + m], lt4[j], eq4[j]);
            }
    }
    then();
    uint2* const out = d.masks + (size_t)hs * d.words + word0 + w.lane;
#pragma unroll
    for (int j = 0; j < G; ++j) {
        const int word = word0 + w.lane + 32 * j;
        const bool valid = FULL || word < d.words;
        const bool pend = valid && (eq2[j] | eq4[j]) != 0u;
        if (valid && !pend) out[32 * j] = make_uint2(lt2[j], lt4[j]);
        const uint32_t bal = __ballot_sync(0xffffffffu, pend);
        if (pend) {
            const int slot = w.qn + __popc(bal & ((1u << w.lane) - 1u));
            w.q->e[slot] = make_uint4(eq2[j], eq4[j], lt2[j], lt4[j]);
            w.q->at[slot] = make_uint2((uint32_t)index << kWordBits | (uint32_t)word, (uint32_t)hs << 3 | 2u);
        }
        w.qn += __popc(bal);
        if ((j & 1) || j == G - 1)
            while (w.qn >= 32) {
                __syncwarp();  // pushes visible to the draining lanes
                drain_draws(w, 32, lattice, bits);
            }
    }
}

// One drawing step: words first .. first + ITEM - 1 (as far as they exist) of half-sweep hs.
template <int G, int ITEM, typename Lattice, typename Bits, typename Then>
__device__ __forceinline__ void draw_step(DrawState& w, const DrawLattice& d, int index, int hs, int first,
                                          const uint32_t (&K2)[8], const uint32_t (&K4)[8], Lattice lattice, Bits bits, Then then)
{
    const PhiloxWordConsts pc = philox_consts(d.key, 0u, d.sweep0 + (uint32_t)(hs >> 1), (uint32_t)(hs & 1));
    if (first + ITEM <= d.words) {
        static_assert(ITEM == 32 * G, "a step is one group");
        draw_words<G, true>(w, d, index, pc, hs, first, K2, K4, lattice, bits, then);
    } else {
        then();
#pragma unroll 1
        for (int word0 = first; word0 < d.words; word0 += 32)
            draw_words<1, false>(w, d, index, pc, hs, word0, K2, K4, lattice, bits, [] {});
    }
}

// Opens the (M, E) entry of a sweep of N sites in dim dimensions to which several tiles will add their counts.
__device__ __forceinline__ void open_entry(int64_t* hist, uint32_t sweep, int64_t N, int dim = 2)
{
    hist[2 * (int64_t)sweep] = -N;
    hist[2 * (int64_t)sweep + 1] = -dim * N;
}

// The thresholds' bits as masks, for the drains; formed by one warp of the CTA.
__device__ __forceinline__ void form_bits(const AheadLattice& d, SharedAhead& sh, int lane)
{
    uint32_t* b = reinterpret_cast<uint32_t*>(sh.bits);
    b[lane] = plane_mask(d.t2, lane);
    b[32 + lane] = plane_mask(d.t4, lane);
}

// A warp's part of drawing a chunk of one lattice: drawing steps of up to ITEM words of one
// half-sweep each, `take` giving the next (in lane 0).  One at a time and only when the step in
// hand is done: a step takes a warp about 4 us, so a warp that holds one it has not begun, or
// several, keeps the launch waiting at its end (L = 1,024: 1.45 us a sweep taking one step
// ahead, 1.30 so).  The step that holds a sweep's first words also opens the sweep's (M, E)
// entry when several tiles will add their counts to it.
template <int G, int ITEM, typename Take>
__device__ void draw_chunk(const AheadLattice& d, uint32_t sweep0, int sweeps, uint2* masks, SharedAhead& sh, int warp,
                           int lane, Take take)
{
    DrawState w{&sh.queue[warp], 0, lane};
    const DrawLattice one{d.key, d.t2, d.t4, d.all2, d.all4, d.words, sweep0, masks};
    auto lattice = [&](int) { return one; };
    auto bits = [&](const DrawLattice&, uint32_t c, uint4& b2, uint4& b4) {
        b2 = sh.bits[c];
        b4 = sh.bits[8 + c];
    };
    // held in registers (the opaque move keeps the compiler from forming them again for every step)
    uint32_t K2[8], K4[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        K2[k] = plane_mask(d.t2, k);
        K4[k] = plane_mask(d.t4, k);
        asm volatile("mov.b32 %0, %0;" : "+r"(K2[k]));
        asm volatile("mov.b32 %0, %0;" : "+r"(K4[k]));
    }
    const int per = (d.words + ITEM - 1) / ITEM, items = 2 * sweeps * per;
    for (;;) {
        const int item = __shfl_sync(0xffffffffu, take(), 0);
        if (item >= items) break;
        const int hs = item / per, first = (item - hs * per) * ITEM;
        if (d.tiles > 1 && (hs & 1) == 0 && first == 0 && lane == 0)
            open_entry(d.hist, sweep0 + (uint32_t)(hs >> 1), (int64_t)d.L * d.L);
        draw_step<G, ITEM>(w, one, 0, hs, first, K2, K4, lattice, bits, [] {});
    }
    while (w.qn > 0) {
        __syncwarp();
        drain_draws(w, min(w.qn, 32), lattice, bits);
    }
    __syncwarp();
}

// Named barriers: of all parts of a tile, and, one pair for even and one for odd sweeps, of the
// threads that hold strips and those that count the sweep, at the end of its white half (kBarWhite
// + parity) and of the next sweep's black half (kBarBlack + the next one's parity; the counting
// threads only arrive).
constexpr int kBarTile = 1, kBarBlack = 2, kBarWhite = 4;

__device__ __forceinline__ void tile_barrier(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

template <int ID>
__device__ __forceinline__ void tile_barrier(int threads)
{
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "r"(threads) : "memory");
}

__device__ __forceinline__ void tile_arrive(int id, int threads)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
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

// ---- cubes.  A tile is a run of slices instead of rows: a strip is one word column of K
// consecutive slices, so the neighbours i - 1 and i + 1 are the strip's own words, and the four in
// the slice (rows j - 1 and j + 1, and the word's own row) come from shared memory.  The three
// decisions of a site (U < T_2, T_4, T_6, each implying the ones before) are two bits: x = U < T_4,
// y = U < (x ? T_6 : T_2).

struct CubeStripAt {
    int t, above, below, left, right, north, south;
    bool odd;   // of an odd row j: the horizontal neighbours' side is the other one
    int row;    // its first slice in the tile
};

template <int K>
__device__ __forceinline__ CubeStripAt cube_strip_at(const AheadLattice& d, int t)
{
    CubeStripAt p;
    const int S = d.W, R = d.row_words, ty = t / S, tx = t - ty * S, j = tx / R, w = tx - j * R;
    const bool whole = d.tiles == 1;
    p.t = t;
    p.row = ty * K;
    p.above = ty > 0 ? (K - 1) * kStrips + t - S : (whole ? (K - 1) * kStrips + (d.groups - 1) * S + tx : t);
    p.below = ty + 1 < d.groups ? t + S : (whole ? tx : t);
    p.right = w + 1 == R ? t - w : t + 1;
    p.left = w == 0 ? t + R - 1 : t - 1;
    p.north = j == 0 ? t + (d.L - 1) * R : t - R;
    p.south = j + 1 == d.L ? t - (d.L - 1) * R : t + R;
    p.odd = (j & 1) != 0;
    return p;
}

// The neighbour count of one word of a strip (bits b0, b1, b2 of the number of +1 neighbours, 0..6).
// COLOUR, k: the word's horizontal neighbour is to the right iff k + COLOUR + j is odd.
template <int COLOUR>
__device__ __forceinline__ void cube_count(const uint32_t* plane, const CubeStripAt& p, int k, uint32_t up, uint32_t dn,
                                           uint32_t same, uint32_t& b0, uint32_t& b1, uint32_t& b2)
{
    const uint32_t no = plane[p.north + k * kStrips], so = plane[p.south + k * kStrips];
    const bool right = (((k + COLOUR) & 1) != 0) != p.odd;
    const uint32_t side = plane[(right ? p.right : p.left) + k * kStrips];
    const uint32_t hz = __funnelshift_r(right ? same : side, right ? side : same, right ? 1 : 31);
    const uint32_t s1 = up ^ dn ^ no, c1 = (up & dn) | (no & (up | dn));
    const uint32_t s2 = so ^ same ^ hz, c2 = (so & same) | (hz & (so | same));
    const uint32_t c3 = s1 & s2;
    b0 = s1 ^ s2;
    b1 = c1 ^ c2 ^ c3;
    b2 = (c1 & c2) | (c3 & (c1 | c2));
}

// One colour's half of a sweep for a strip: t its target words, s its source words (in `plane`), m
// the masks at mp, K words `stride` bytes apart.
template <int K, int COLOUR>
__device__ __forceinline__ void update_cube_strip(uint32_t (&t)[K], const uint32_t (&s)[K], const uint32_t* plane,
                                                  const CubeStripAt& p, const unsigned char* mp, int stride)
{
    const uint32_t above = plane[p.above], below = plane[p.below];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        uint32_t b0, b1, b2;
        cube_count<COLOUR>(plane, p, k, k == 0 ? above : s[k - 1], k == K - 1 ? below : s[k + 1], s[k], b0, b1, b2);
        const uint2 m = *reinterpret_cast<const uint2*>(mp + k * stride);
        // n anti-aligned neighbours: c or 6 - c of the c that are +1.  n < 3: c > 3 for a +1, c < 3
        // for a -1; n odd iff c is; n = 2 rather than 0 iff b1 differs from the spin.
        const uint32_t h = b2 | (b1 & b0);
        const uint32_t low = (t[k] & b2) | (~t[k] & ~h);
        const uint32_t z = b1 ^ t[k];
        const uint32_t even = (m.x & m.y) | (z & (m.x | m.y));  // n = 2: U < T_2 = x | y; n = 0: U < T_6 = x & y
        const uint32_t acc = (b0 & m.x) | (~b0 & even);         // n = 1: U < T_4 = x
        t[k] ^= ~low | acc;
    }
}

// Up spins of both colours and anti-aligned bonds of slices lo .. hi - 1 of a strip, from its white
// words t.
template <int K>
__device__ __forceinline__ void count_cube_strip(const uint32_t (&t)[K], const uint32_t (&s)[K], const uint32_t* plane,
                                                 const CubeStripAt& p, int lo, int hi, uint32_t& ups, uint32_t& anti)
{
    const uint32_t above = plane[p.above], below = plane[p.below];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        uint32_t b0, b1, b2;
        cube_count<1>(plane, p, k, k == 0 ? above : s[k - 1], k == K - 1 ? below : s[k + 1], s[k], b0, b1, b2);
        const uint32_t keep = k >= lo && k < hi ? ~0u : 0u;
        // bits of n = 6 - c for a +1, c for a -1
        const uint32_t n1 = (t[k] & ~(b1 ^ b0)) | (~t[k] & b1), n2 = (t[k] & ~(b2 | (b1 & b0))) | (~t[k] & b2);
        ups += __popc(s[k] & keep) + __popc(t[k] & keep);
        anti += __popc(b0 & keep) + 2u * __popc(n1 & keep) + 4u * __popc(n2 & keep);
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

template <int K, typename At>
__device__ __forceinline__ void load_strip(const uint32_t* plane, const At& p, uint32_t (&v)[K])
{
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = plane[p.t + k * kStrips];
}

template <int K, typename At>
__device__ __forceinline__ void store_strip(uint32_t* plane, const At& p, const uint32_t (&v)[K])
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
//    buffer for that).  Tiles of at most half the strips have two such groups, a sweep each in
//    turn, as counting takes longer than updating (L = 128: 300 ns a sweep counted by the
//    first group, 237 by one group beside it, 180 by two; L = 64: 154);
//  - a lane of the last warp keeps the ring of masks filled (fetch_masks).
template <int K, bool CUBE = false>
__device__ void update_tile(const AheadLattice& d, const AheadStep& st, int tile, SharedAhead& sh)
{
    const int W = d.W, L = d.L, active = d.groups * W;  // (of a cube, W: a slice's words)
    const int threads = (active + 31) & ~31, part = threadIdx.x / kStrips;
    // tiles of at most half the strips are counted by two groups in turn, a sweep each
    const int turns = threads <= kStrips / 2 ? 2 : 1;
    const int turn = turns == 2 && part == 1 ? threadIdx.x % kStrips / (kStrips / 2) : 0;
    const int tid = threadIdx.x % kStrips - turn * (kStrips / 2);
    const bool fetcher = part == 2;
    if (tid >= threads && !fetcher) return;
    const TileAt a = tile_at<K>(d, tile);
    const int n = st.upd_n, everyone = (1 + turns) * threads + 32;
    if (threadIdx.x == 0 && !st.alone) {
        for (int k = 0; k < a.slots; ++k) {
            mbar_init(&sh.full[k], 1);
            mbar_init(&sh.empty[k], (uint32_t)threads / 32u);
        }
        fence_mbarrier_init();
    }
    const bool on = tid < active;
    // a lane past the end follows the last one and keeps nothing
    const std::conditional_t<CUBE, CubeStripAt, StripAt> p = [&] {
        if constexpr (CUBE)
            return cube_strip_at<K>(d, on ? tid : active - 1);
        else
            return strip_at<K>(d, on ? tid : active - 1);
    }();
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
        auto one_sweep = [&](auto which) {
            constexpr int parity = decltype(which)::value;
            uint32_t* const black = sh.planes[parity];
            if constexpr (CUBE) {
                update_cube_strip<K, 0>(b, w, sh.planes[2], p, mp, W * 8);
                mp += a.half_bytes;
                if (on) store_strip<K>(black, p, b);
                tile_barrier<kBarBlack + parity>(2 * threads);
                update_cube_strip<K, 1>(w, b, black, p, mp, W * 8);
                mp += a.half_bytes;
                if (on) store_strip<K>(sh.planes[2], p, w);
                tile_barrier<kBarWhite + parity>(2 * threads);
            } else {
                uint2 m[K];
                {
                    const StripNeighbours<K> nb = load_neighbours<K, 0>(sh.planes[2], p, w);
                    load_masks(m);
                    update_strip<K>(b, w, nb, m);
                    if (on) store_strip<K>(black, p, b);
                    tile_barrier<kBarBlack + parity>(2 * threads);
                }
                {
                    const StripNeighbours<K> nb = load_neighbours<K, 1>(black, p, b);
                    load_masks(m);
                    update_strip<K>(w, b, nb, m);
                    if (on) store_strip<K>(sh.planes[2], p, w);
                    tile_barrier<kBarWhite + parity>(2 * threads);
                }
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
                one_sweep(std::integral_constant<int, 1>());
                odd = 0;
                --left;
            }
            for (; left >= 2; left -= 2) {
                one_sweep(std::integral_constant<int, 0>());
                one_sweep(std::integral_constant<int, 1>());
            }
            if (left) {
                one_sweep(std::integral_constant<int, 0>());
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
        const bool strips = whole || (d.halo % K == 0 && d.rows % K == 0 && L % d.rows % K == 0);  // own rows are whole strips
        // a warp whose strips are all halo rows only keeps the barriers' count
        const bool any_own = __any_sync(0xffffffffu, lo < hi);
        // (for the first black half-sweep, which has no sweep before it)
        if (turn == turns - 1) tile_arrive(kBarBlack, 2 * threads);
        for (int s = turn; s < n; s += turns) {
            tile_barrier(kBarWhite + (s & 1), 2 * threads);
            if (!any_own) {
                if (s + 1 < n) tile_arrive(kBarBlack + ((s + 1) & 1), 2 * threads);
                continue;
            }
            const uint32_t* black = sh.planes[s & 1];
            load_strip<K>(sh.planes[2], p, w);
            // of what the next black half-sweep's end allows to be overwritten, this was all
            // (arriving after the other loads is still faster by 5 % at L = 128)
            if (CUBE && s + 1 < n) tile_arrive(kBarBlack + ((s + 1) & 1), 2 * threads);
            load_strip<K>(black, p, b);
            uint32_t ups = 0, anti = 0;
            if constexpr (CUBE) {
                count_cube_strip<K>(w, b, black, p, lo, hi, ups, anti);
            } else {
                const StripNeighbours<K> nb = load_neighbours<K, 1>(black, p, b);
                if (s + 1 < n) tile_arrive(kBarBlack + ((s + 1) & 1), 2 * threads);
                if (strips) {
                    count_strip<K>(w, b, nb, 0, K, ups, anti);
                    if (lo >= hi) ups = anti = 0u;
                } else {
                    count_strip<K>(w, b, nb, lo, hi, ups, anti);
                }
            }
            // a lane has at most 64 K <= 1024 up spins and 128 K <= 2048 bonds (a cube's 192 K): a
            // warp's sums fit 16 bits for strips of up to 8 rows
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
        const int64_t N = CUBE ? (int64_t)L * L * L : (int64_t)L * L;
        for (int s = turn * threads + tid; s < n; s += turns * threads) {
            int64_t* entry = d.hist + 2 * (int64_t)(st.upd_sweep + (uint32_t)s);
            const int64_t M = 2 * (int64_t)sh.sums[2 * s], E = 2 * (int64_t)sh.sums[2 * s + 1];
            if (whole) {
                entry[0] = M - N;
                entry[1] = E - (CUBE ? 3 : 2) * N;
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

// K: rows (slices of a cube) of a thread's strip.
template <int K, bool CUBE = false>
__global__ void __launch_bounds__(kNT, 1) ahead_kernel(const __grid_constant__ AheadLattice d, const AheadStep st)
{
    extern __shared__ __align__(16) unsigned char smem_ahead[];
    SharedAhead& sh = *reinterpret_cast<SharedAhead*>(smem_ahead);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_launch_next();
    if (warp == 0) form_bits(d, sh, lane);
    __syncthreads();
    grid_wait();
    if (!CUBE && st.alone) {
        // a short run of a lattice of one tile: this CTA draws the masks it needs itself, into
        // the ring's slots
        int next = warp - kWarps;
        draw_chunk<1, 32>(d, st.upd_sweep, st.upd_n, reinterpret_cast<uint2*>(sh.ring), sh, warp, lane,
                          [&] { return next += kWarps; });
        __syncthreads();
    }
    if (st.upd_n > 0)
        for (int tile = (int)blockIdx.x; tile < d.tiles; tile += (int)gridDim.x) update_tile<K, CUBE>(d, st, tile, sh);
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
    if (CUBE && st.gen_n > 0)
        draw_cube_chunk(d, st.gen_sweep, st.gen_n, d.masks[st.gen_buf], sh, warp, lane,
                        [&] { return lane == 0 ? atomicAdd(&d.ticket[st.gen_buf], 1) : 0; });
    if (!CUBE && st.gen_n > 0)
        draw_chunk<4, kItemWords>(d, st.gen_sweep, st.gen_n, d.masks[st.gen_buf], sh, warp, lane,
                                  [&] { return lane == 0 ? atomicAdd(&d.ticket[st.gen_buf], 1) : 0; });
}

// ---- drawing for cubes: the same with three thresholds and the two-bit decisions.  An entry of the
// queue is (undecided against T_2, T_4, T_6; below each so far; word; half-sweep << 3 | next call)
// in the room of a 2D queue, checked after every word.
constexpr int kCubeQueueWords = 64;
static_assert(kCubeQueueWords * 32 <= (int)sizeof(DrawQueue), "a cube's queue fits");

__device__ __forceinline__ uint2 cube_decisions(uint32_t lt2, uint32_t lt4, uint32_t lt6)
{
    return make_uint2(lt4, (lt4 & lt6) | (~lt4 & lt2));
}

__device__ __forceinline__ void drain_cube_draws(const AheadLattice& d, uint32_t sweep0, uint2* masks, uint4* q, int& qn,
                                                 int n, int lane)
{
    uint4 e = make_uint4(0u, 0u, 0u, 0u), f = make_uint4(0u, 0u, 0u, 2u);
    if (lane < n) {
        e = q[2 * (qn - n + lane)];
        f = q[2 * (qn - n + lane) + 1];
    }
    qn -= n;
    __syncwarp();  // entries read before any goes back
    const uint32_t c = f.w & 7u, hs = f.w >> 3;
    const PhiloxWordConsts pc = philox_consts(d.key, 0u, sweep0 + (hs >> 1), hs & 1u);
    const uint32_t base[1] = {8u * f.z ^ pc.x0k};
    uint32_t o[1][4];
    philox_calls<1>(base, c, pc, d.key, o);
    uint32_t l2 = 0u, l4 = 0u, l6 = 0u, e2 = e.x, e4 = e.y, e6 = e.z;
    const uint32_t t2 = d.t2 << (4u * c), t4 = d.t4 << (4u * c), t6 = d.t6 << (4u * c);
#pragma unroll
    for (int m = 3; m >= 0; --m) {
        compare_plane(o[0][m], plane_mask(t2, m), l2, e2);
        compare_plane(o[0][m], plane_mask(t4, m), l4, e4);
        compare_plane(o[0][m], plane_mask(t6, m), l6, e6);
    }
    uint32_t lt2 = e.w | (e.x & l2), lt4 = f.x | (e.y & l4), lt6 = f.y | (e.z & l6);
    if (c == 7u) {  // U equal to min(T, 2^32 - 1): below only if T = 2^32
        lt2 |= e2 & d.all2;
        lt4 |= e4 & d.all4;
        lt6 |= e6 & d.all6;
    }
    const bool pend = (e2 | e4 | e6) != 0u && c < 7u;
    if (lane < n && !pend) masks[(size_t)hs * d.words + f.z] = cube_decisions(lt2, lt4, lt6);
    const uint32_t bal = __ballot_sync(0xffffffffu, pend);
    if (pend) {
        const int slot = qn + __popc(bal & ((1u << lane) - 1u));
        q[2 * slot] = make_uint4(e2, e4, e6, lt2);
        q[2 * slot + 1] = make_uint4(lt4, lt6, f.z, f.w + 1u);
    }
    qn += __popc(bal);
}

// A warp's part of drawing a chunk of a cube, 64 words a step (a plane's words are a multiple).
template <typename Take>
__device__ void draw_cube_chunk(const AheadLattice& d, uint32_t sweep0, int sweeps, uint2* masks, SharedAhead& sh,
                                int warp, int lane, Take take)
{
    constexpr int G = 2;
    uint4* q = reinterpret_cast<uint4*>(&sh.queue[warp]);
    int qn = 0;
    const int per = d.words / (32 * G), items = 2 * sweeps * per;
    for (;;) {
        const int item = __shfl_sync(0xffffffffu, take(), 0);
        if (item >= items) break;
        const int hs = item / per, word0 = (item - hs * per) * 32 * G + lane;
        if (d.tiles > 1 && (hs & 1) == 0 && item == hs * per && lane == 0)
            open_entry(d.hist, sweep0 + (uint32_t)(hs >> 1), (int64_t)d.L * d.L * d.L, 3);
        const PhiloxWordConsts pc = philox_consts(d.key, 0u, sweep0 + (uint32_t)(hs >> 1), (uint32_t)(hs & 1));
        uint32_t base[G], lt2[G], lt4[G], lt6[G], eq2[G], eq4[G], eq6[G];
#pragma unroll
        for (int j = 0; j < G; ++j) {
            base[j] = 8u * (uint32_t)(word0 + 32 * j) ^ pc.x0k;
            lt2[j] = lt4[j] = lt6[j] = 0u;
            eq2[j] = eq4[j] = eq6[j] = ~0u;
        }
#pragma unroll
        for (int c = 1; c >= 0; --c) {
            uint32_t o[G][4];
            philox_calls<G>(base, (uint32_t)c, pc, d.key, o);
#pragma unroll
            for (int m = 3; m >= 0; --m) {
                const uint32_t K2 = plane_mask(d.t2, 4 * c + m), K4 = plane_mask(d.t4, 4 * c + m),
                               K6 = plane_mask(d.t6, 4 * c + m);
#pragma unroll
                for (int j = 0; j < G; ++j) {
                    compare_plane(o[j][m], K2, lt2[j], eq2[j]);
                    compare_plane(o[j][m], K4, lt4[j], eq4[j]);
                    compare_plane(o[j][m], K6, lt6[j], eq6[j]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < G; ++j) {
            const int word = word0 + 32 * j;
            const bool pend = (eq2[j] | eq4[j] | eq6[j]) != 0u;
            if (!pend) masks[(size_t)hs * d.words + word] = cube_decisions(lt2[j], lt4[j], lt6[j]);
            const uint32_t bal = __ballot_sync(0xffffffffu, pend);
            if (pend) {
                const int slot = qn + __popc(bal & ((1u << lane) - 1u));
                q[2 * slot] = make_uint4(eq2[j], eq4[j], eq6[j], lt2[j]);
                q[2 * slot + 1] = make_uint4(lt4[j], lt6[j], (uint32_t)word, (uint32_t)hs << 3 | 2u);
            }
            qn += __popc(bal);
            while (qn >= 32) {
                __syncwarp();  // pushes visible to the draining lanes
                drain_cube_draws(d, sweep0, masks, q, qn, 32, lane);
            }
        }
    }
    while (qn > 0) {
        __syncwarp();
        drain_cube_draws(d, sweep0, masks, q, qn, min(qn, 32), lane);
    }
    __syncwarp();
}

// ---- batches: the same for many lattices of a batch, in common launches.  The geometry of each
// lattice's tiles follows from its side and the batch's chunk, and its places in the mask
// buffers, the copies of the planes and the launch's tables from the plane words of the
// lattices before it, so a change of the batch costs three small tables.

// dense: the batch has work for every SM throughout a launch, so tiles are as tall as strips of
// 16 rows make them (few halo rows) and lattices of up to 512 are one tile; else they are low,
// for short half-sweeps.
__host__ __device__ inline bool batch_whole(int W, int dense) { return W <= 3 || (dense && W <= 8); }

__host__ __device__ inline void batch_geometry(int W, int chunk, int dense, AheadPlan& p)
{
    const int L = 64 * W, most = kStrips / W;  // strips one above the other
    p.strip = 2;
    if (batch_whole(W, dense)) {
        while (L > most * p.strip) p.strip *= 2;
        p.groups = L / p.strip;
        p.rows = L;
        p.halo = 0;
        p.tiles = 1;
        return;
    }
    // not dense: the shortest strips that leave a tile at least as many own rows as halo rows
    while (p.strip < kMaxStrip && (dense || most * p.strip < 8 * chunk)) p.strip *= 2;
    p.groups = most;
    p.halo = 2 * chunk;
    p.rows = p.groups * p.strip - 2 * p.halo;
    p.tiles = (L + p.rows - 1) / p.rows;
}

// Entry of a table of prefix sums that holds `at`.
__device__ __forceinline__ int find_entry(const int32_t* start, int count, int at)
{
    int lo = 0, hi = count;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (start[mid] <= at)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// Sweeps of a run of `total` that lattice d takes part in: up to its own limit.
__device__ __forceinline__ int sweeps_of(const LatticeDesc& d, int total)
{
    if (!d.active || d.sweep >= d.target) return 0;
    const uint32_t left = d.target - d.sweep;
    return left < (uint32_t)total ? (int)left : total;
}

__device__ __forceinline__ AheadLattice batch_lattice(const AheadBatch& b, const LatticeDesc& d, int word_start)
{
    AheadPlan p;
    batch_geometry(d.W, b.chunk, b.dense, p);
    AheadLattice a;
    a.home = d.plane[0];
    a.copy = b.copy + 4 * (size_t)word_start;
    a.masks[0] = b.masks[0] + 2 * (size_t)b.chunk * word_start;
    a.masks[1] = b.masks[1] + 2 * (size_t)b.chunk * word_start;
    a.ticket = nullptr;
    a.hist = d.hist;
    a.status = b.status;
    a.key = d.key;
    a.t2 = d.t2;
    a.t4 = d.t4;
    a.all2 = d.all2;
    a.all4 = d.all4;
    a.L = d.L;
    a.W = d.W;
    a.words = d.L * d.W;
    a.strip = p.strip;
    a.groups = p.groups;
    a.rows = p.rows;
    a.halo = p.halo;
    a.tiles = p.tiles;
    return a;
}

__global__ void __launch_bounds__(kNT, 1) ahead_batch_kernel(const __grid_constant__ AheadBatch b, const AheadBatchStep st)
{
    extern __shared__ __align__(16) unsigned char smem_ahead[];
    SharedAhead& sh = *reinterpret_cast<SharedAhead*>(smem_ahead);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    grid_launch_next();
    grid_wait();
    // the tables behind the few sums that a chunk needs
    int32_t* const tile_start = reinterpret_cast<int32_t*>(sh.sums) + 2 * kMaxBatchChunk;
    int32_t* const step_start = tile_start + b.count + 1;
    int32_t* const word_start = step_start + b.count + 1;
    for (int k = threadIdx.x; k < 3 * (b.count + 1); k += kNT) tile_start[k] = b.tables[k];
    __syncthreads();

    if (st.upd_n > 0 || st.fill)
        for (int tile = (int)blockIdx.x; tile < b.tiles; tile += (int)gridDim.x) {
            const int l = find_entry(tile_start, b.count, tile);
            const int local = tile - tile_start[l];
            if (threadIdx.x == 0) {
                const LatticeDesc& ld = b.desc[l];
                const int mine = sweeps_of(ld, st.total);
                AheadLattice& d = sh.now.lattice;
                AheadStep& s = sh.now.step;
                d = batch_lattice(b, ld, word_start[l]);
                s.upd_n = st.fill ? mine : max(0, min(mine - st.upd_off, st.upd_n));
                s.upd_sweep = ld.sweep + (uint32_t)st.upd_off;
                s.upd_buf = st.upd_buf;
                s.src = d.tiles > 1 ? st.src : -1;
                s.dst = d.tiles > 1 && st.upd_off + s.upd_n < mine ? st.src ^ 1 : -1;
                s.alone = 0;
            }
            __syncthreads();
            const AheadLattice& d = sh.now.lattice;
            const AheadStep& s = sh.now.step;
            if (s.upd_n == 0) {
            } else if (st.fill) {
                // the first launch of a run: the copy of the planes that the first update reads
                const int from = local * d.rows * d.W, n = d.tiles > 1 ? min(d.rows * d.W, d.words - from) : 0;
                for (int k = threadIdx.x; k < n; k += kNT) {
                    d.copy[from + k] = d.home[from + k];
                    d.copy[d.words + from + k] = d.home[d.words + from + k];
                }
            } else if (d.strip == 2) {
                update_tile<2>(d, s, local, sh);
            } else if (d.strip == 4) {
                update_tile<4>(d, s, local, sh);
            } else if (d.strip == 8) {
                update_tile<8>(d, s, local, sh);
            } else {
                update_tile<16>(d, s, local, sh);
            }
            __syncthreads();
        }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        b.ticket[st.gen_buf ^ 1] = 0;
        if (st.gen_n == 0) b.ticket[st.gen_buf] = 0;
    }
    if (st.gen_n == 0) return;

    DrawState w{&sh.queue[warp], 0, lane};
    uint2* const masks = b.masks[st.gen_buf];
    auto lattice = [&](int l) {
        const LatticeDesc& d = b.desc[l];
        return DrawLattice{d.key, d.t2, d.t4, d.all2, d.all4, d.L * d.W, d.sweep + (uint32_t)st.gen_off,
                           masks + 2 * (size_t)b.chunk * word_start[l]};
    };
    auto bits = [&](const DrawLattice& d, uint32_t c, uint4& b2, uint4& b4) {
        const uint32_t t2 = d.t2 << (4u * c), t4 = d.t4 << (4u * c);
        b2 = make_uint4(plane_mask(t2, 0), plane_mask(t2, 1), plane_mask(t2, 2), plane_mask(t2, 3));
        b4 = make_uint4(plane_mask(t4, 0), plane_mask(t4, 1), plane_mask(t4, 2), plane_mask(t4, 3));
    };
    const int per = step_start[b.count], items = 2 * st.gen_n * per;
    auto take = [&] { return lane == 0 ? atomicAdd(&b.ticket[st.gen_buf], 1) : 0; };
    int taken = take();
    for (;;) {
        const int item = __shfl_sync(0xffffffffu, taken, 0);
        if (item >= items) break;
        const int hs = item / per, r = item - hs * per;
        const int l = find_entry(step_start, b.count, r);
        const LatticeDesc& ld = b.desc[l];
        if (st.gen_off + (hs >> 1) >= sweeps_of(ld, st.total)) {
            taken = take();
            continue;
        }
        const int first = (r - step_start[l]) * kItemWords;
        const DrawLattice d = lattice(l);
        if (!batch_whole(ld.W, b.dense) && (hs & 1) == 0 && first == 0 && lane == 0) 
            open_entry(ld.hist, d.sweep0 + (uint32_t)(hs >> 1), (int64_t)ld.L * ld.L);
        uint32_t K2[8], K4[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            K2[k] = plane_mask(d.t2, k);
            K4[k] = plane_mask(d.t4, k);
        }
        draw_step<4, kItemWords>(w, d, l, hs, first, K2, K4, lattice, bits, [&] { taken = take(); });
    }
    while (w.qn > 0) {
        __syncwarp();
        drain_draws(w, min(w.qn, 32), lattice, bits);
    }
}

template <int K, bool CUBE = false>
cudaError_t launch_k(const AheadLattice& d, const AheadStep& st, int grid, cudaStream_t s)
{
    return launch_following(ahead_kernel<K, CUBE>, dim3(grid), dim3(kNT), sizeof(SharedAhead), s, d, st);
}

cudaError_t launch_step(const AheadLattice& d, const AheadStep& st, cudaStream_t s)
{
    const int64_t items = 2 * (int64_t)st.gen_n * ((d.words + kItemWords - 1) / kItemWords);
    const int64_t want = (st.upd_n > 0 ? d.tiles : 0) + (items + kWarps - 1) / kWarps;
    const int64_t grid = std::min<int64_t>(sm_count(), std::max<int64_t>(want, 1));
    if (d.cube) return launch_k<16, true>(d, st, (int)grid, s);
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

// Sides up to 4,096 (longer rows leave a tile too few own rows) and as many lattices as the
// tables in shared memory hold.
int ahead_batch_max_L() { return 4096; }
int ahead_batch_max_count() { return (2 * kMaxChunk - 2 * kMaxBatchChunk) / 3 - 1; }

// Sweeps of a launch for a batch whose longest side is L: the tallest tile that W words a row
// allow is four times as high as its halo.
int ahead_batch_chunk(int64_t L)
{
    const int held = kStrips / (int)(L / 64) * kMaxStrip;
    return std::max(1, std::min(16, held / 8));
}

int32_t ahead_batch_tiles(int64_t L, int chunk, int dense)
{
    AheadPlan p;
    batch_geometry((int)(L / 64), chunk, dense, p);
    return p.tiles;
}

int32_t ahead_batch_steps(int64_t L) { return (int32_t)((L * (L / 64) + kItemWords - 1) / kItemWords); }

cudaError_t ahead_batch_configure()
{
    return cudaFuncSetAttribute(ahead_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SharedAhead));
}

cudaError_t launch_ahead_batch(const AheadBatch& b, int64_t steps, int64_t n, cudaStream_t s, int64_t* launched)
{
    // chunk k is drawn by the launch that updates chunk k - 1, as for a single lattice
    int64_t drawn = 0, updated = 0;
    int in_flight = 0, k = 0;
    AheadBatchStep st;
    st.total = (int32_t)n;
    while (updated < n) {
        const int next = (int)std::min<int64_t>(n - drawn, b.chunk);
        st.upd_off = (int32_t)updated;
        st.upd_n = in_flight;
        st.upd_buf = (k & 1) ^ 1;
        st.gen_off = (int32_t)drawn;
        st.gen_n = next;
        st.gen_buf = k & 1;
        st.src = (k & 1) ^ 1;
        st.fill = k == 0;
        const int64_t want = std::max<int64_t>(b.tiles, 0) + (2 * next * steps + kWarps - 1) / kWarps;
        const int grid = (int)std::min<int64_t>(sm_count(), want);
        const cudaError_t e = launch_following(ahead_batch_kernel, dim3(grid), dim3(kNT), sizeof(SharedAhead), s, b, st);
        if (e != cudaSuccess) return e;
        ++*launched;
        updated += in_flight;
        drawn += next;
        in_flight = next;
        ++k;
    }
    return cudaSuccess;
}

int ahead_max_L() { return 8192; }

AheadPlan ahead_plan(int64_t L)
{
    AheadPlan p;
    const int W = (int)(L / 64);
    if (L < 64 || L % 64 || L > ahead_max_L()) return p;
    const int64_t words = L * W, per_sweep = words * 2 * (int64_t)sizeof(uint2);
    if (W <= 3) {
        // one tile: the whole lattice in one CTA, two or four rows a thread
        p.strip = words <= 2 * kStrips ? 2 : 4;
        p.groups = (int)L / p.strip;
        p.rows = (int)L;
        p.halo = 0;
        p.tiles = 1;
        p.chunk = (int)std::min<int64_t>(kMaxChunk, (8ll << 20) / per_sweep);
    } else {
        // Several tiles.  A launch costs about 4 us beyond its half-sweeps, which asks for long
        // chunks; their halo rows are updated (and their masks fetched) by two tiles, which
        // asks for short ones, the more so the more the drawing of the own rows' masks takes.
        // us a sweep: L = 256: 0.59 in one tile, 0.48 and 0.46 with strips of 2 and chunks of 24 and
        // 28; 320: 0.81 / 0.54 (20); 512: strips of 4 0.65 (24), 0.63 (28), of 2 0.64 (14); 1,024: strips
        // of 4 0.93 (10), 0.88 (12), 1.13 (14), of 8 1.08 (20); 1,344: strips of 8 1.19 (16), of
        // 16 2.0; 2,048: strips of 8 2.15 (8), of 16 1.71 (16), 1.77 (20); 4,096: 6.70 (6), 6.42 (8),
        // 6.80 (10); 8,192: 26.7 (2), 25.9 (3), 26.8 (4)
        p.strip = W <= 6 ? 2 : (W <= 16 ? 4 : (W <= 28 ? 8 : 16));
        p.groups = kStrips / W;
        const int held = p.groups * p.strip;  // rows a CTA holds
        p.chunk = W <= 8    ? std::min(32, held * 7 / 32)
                  : W <= 28 ? held * 3 / 16
                  : W <= 64 ? held / 8
                            : held * 3 / 32;
        p.halo = 2 * p.chunk;
        p.rows = held - 2 * p.halo;
        p.tiles = (int)((L + p.rows - 1) / p.rows);
    }
    p.mask_bytes = per_sweep * p.chunk;
    p.copy_bytes = p.tiles > 1 ? 2 * 2 * words * (int64_t)sizeof(uint32_t) : 0;
    return p;
}

// Cubes whose slice (L * L/64 words) is one thread's word each: L = 64 in one tile, L = 128 in tiles
// of 16 slices.
AheadPlan ahead_plan3(int64_t L)
{
    AheadPlan p;
    if (L != 64 && L != 128) return p;
    const int S = (int)(L * (L / 64));
    const int64_t per_sweep = L * S * 2 * (int64_t)sizeof(uint2);
    p.cube = 1;
    p.strip = kMaxStrip;
    p.groups = kStrips / S;
    if (L == 64) {
        p.rows = (int)L;
        p.halo = 0;
        p.tiles = 1;
        p.chunk = (int)((8ll << 20) / per_sweep);
    } else {
        p.chunk = 3;
        p.halo = 2 * p.chunk;
        p.rows = p.groups * p.strip - 2 * p.halo;
        p.tiles = (int)((L + p.rows - 1) / p.rows);
        p.copy_bytes = 2 * 2 * L * S * (int64_t)sizeof(uint32_t);
    }
    p.mask_bytes = per_sweep * p.chunk;
    return p;
}

cudaError_t ahead_configure(const AheadPlan& p)
{
    const void* k = p.cube         ? (const void*)ahead_kernel<16, true>
                    : p.strip == 2 ? (const void*)ahead_kernel<2>
                    : p.strip == 4 ? (const void*)ahead_kernel<4>
                    : p.strip == 8 ? (const void*)ahead_kernel<8>
                                   : (const void*)ahead_kernel<16>;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SharedAhead));
}

// Up to two drawing steps of 32 words for each warp: a few microseconds less than a launch for
// the drawing alone.
bool ahead_alone(const AheadLattice& d, int64_t n)
{
    return !d.cube && d.tiles == 1 && n <= kWarps && 2 * n * ((d.words + 31) / 32) <= 2 * kWarps;
}

cudaError_t launch_ahead_sweeps(const AheadLattice& d, int chunk, uint32_t sweep, int64_t n, cudaStream_t s,
                                int64_t* launched)
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
        ++*launched;
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
        ++*launched;
        updated += in_flight;
        drawn += next;
        in_flight = next;
        ++k;
    }
    return cudaSuccess;
}

}  // namespace ising
