// Internal declarations shared by the library's translation units.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "ising_device.cuh"

namespace ising {

// Launches a kernel that starts with grid_wait() so that its start overlaps the end of the
// stream's work before it.
template <typename... P, typename... A>
cudaError_t launch_following(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// The same for a kernel known by its handle (compiled at run time), with its argument array.
inline cudaError_t launch_following_c(const void* kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t s, void** args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, kernel, args);
}

// Launchers (return cudaError_t of the launch).  extra_tx > 0 makes every tile
// barrier expect bytes that never arrive: only the timeout self-test uses it.
// one != nullptr: a launch over that single lattice, whose descriptor (with the
// sweep index the host knows) is passed by value; tt is then not read.  Not for
// graph capture, since the sweep index is baked into the launch.  blocks: some
// lattice of tt may have column-block tiles (tile_words < W).  fixed: an instance
// compiled for the thresholds (jit_sweep_kernel) of that lattice (with one) or of
// every lattice of tt (without), launched instead of the built-in one.
cudaError_t launch_packed_half_sweep(const TileTable& tt, int colour, int step, int* status, int grid,
                                     int threads, int smem_stage_bytes, cudaStream_t s,
                                     long long wait_limit = kWaitLimitCycles, uint32_t extra_tx = 0,
                                     const LatticeDesc* one = nullptr, bool blocks = false,
                                     const void* fixed = nullptr);
// Allows launches of a fixed-threshold kernel with `smem` bytes of dynamic shared
// memory (never less than two full stages) and gives its resident CTAs per SM.
cudaError_t packed_fixed_configure(const void* fixed, size_t smem, int threads, int* blocks_per_sm);
// Sweeps with the random numbers drawn ahead of the update (sweep_ahead.cu), for one packed
// lattice of side L <= ahead_max_L().  A plan's tiles = 0: no plan.
struct AheadPlan {
    int strip = 0;             // rows of a thread's strip
    int groups = 0;            // strips one above the other in a tile (with its halo)
    int rows = 0, halo = 0;    // a tile's own rows, and extra rows above and below them
    int tiles = 0;
    int chunk = 0;             // most sweeps of one launch
    int cube = 0;              // a cube: slices in the place of rows
    int64_t mask_bytes = 0;    // one buffer of acceptance masks (two are needed)
    int64_t copy_bytes = 0;    // both copies of the planes (0: the lattice is one tile)
};
struct AheadLattice {
    uint32_t* home;            // both planes, black then white
    uint32_t* copy;            // two copies of them (lattices of several tiles)
    uint2* masks[2];           // per half-sweep of a chunk and word: U < T_2, U < T_4
    int* ticket;               // drawing steps taken of each buffer's chunk (two, zero between calls)
    int64_t* hist;             // (M, E) pairs indexed by sweep number
    int* status;               // set when a bounded wait runs out
    uint64_t key;
    uint32_t t2, t4, all2, all4;  // thresholds as in LatticeDesc
    int32_t L, W, words;       // words: of one plane (W: of a row, of a cube's slice)
    uint32_t t6, all6;         // cubes
    int32_t cube, row_words;   // cubes: 1, words of a row
    int32_t strip, groups, rows, halo, tiles;  // the plan's
};
// What one launch does: update upd_n sweeps from upd_sweep on from masks buffer upd_buf, reading
// the planes at src (-1: home, else a copy) and writing them at dst; draw the masks of gen_n
// sweeps from gen_sweep on into buffer gen_buf; fill >= 0: copy home there first.  alone:
// draw the update's masks in the same launch (a lattice of one tile, one CTA).
struct AheadStep {
    uint32_t upd_sweep, gen_sweep;
    int32_t upd_n, upd_buf, src, dst;
    int32_t gen_n, gen_buf, fill, alone;
};
// The same for the lattices of a batch (sides up to ahead_batch_max_L(), at most
// ahead_batch_max_count() slots): every lattice's masks, copies and tiles in common launches.
struct AheadBatch {
    const LatticeDesc* desc;   // count slots
    const int32_t* tables;     // prefix sums over the slots, count + 1 entries each: tiles, drawing
                               // steps of a half-sweep, plane words
    uint2* masks[2];           // each 2 * chunk uint2 for every plane word
    uint32_t* copy;            // four words for every plane word
    int* ticket;               // two, zero between runs
    int* status;
    int32_t count, chunk, tiles;
    int32_t dense;             // work for every SM: tall tiles
};
struct AheadBatchStep {
    int32_t total;             // sweeps of the run; a lattice stops at its own limit
    int32_t upd_off, upd_n, upd_buf, src;
    int32_t gen_off, gen_n, gen_buf, fill;
};
int ahead_batch_max_L();
int ahead_batch_max_count();
int ahead_batch_chunk(int64_t L);               // sweeps of a launch, for the batch's longest side
int32_t ahead_batch_tiles(int64_t L, int chunk, int dense);
int32_t ahead_batch_steps(int64_t L);
cudaError_t ahead_batch_configure();
// Enqueues a run of n sweeps; steps: drawing steps of a half-sweep of all lattices.  Adds its
// launches to *launched.
cudaError_t launch_ahead_batch(const AheadBatch& b, int64_t steps, int64_t n, cudaStream_t s, int64_t* launched);
int ahead_max_L();
AheadPlan ahead_plan(int64_t L);
AheadPlan ahead_plan3(int64_t L);  // of a cube
cudaError_t ahead_configure(const AheadPlan& p);
// Whether n sweeps are one launch of one CTA that draws its own masks (no workspace needed).
bool ahead_alone(const AheadLattice& d, int64_t n);
// Enqueues n sweeps, numbered from `sweep` on, in launches of at most `chunk` sweeps, added to *launched.
cudaError_t launch_ahead_sweeps(const AheadLattice& d, int chunk, uint32_t sweep, int64_t n, cudaStream_t s,
                                int64_t* launched);
// One small lattice (L <= packed_resident_max_L()) swept nsweeps times by a single
// CTA holding both planes in shared memory; writes hist[d.sweep .. +nsweeps).
int packed_resident_max_L();
cudaError_t launch_packed_resident(const LatticeDesc& d, int nsweeps, cudaStream_t s);
cudaError_t launch_packed_advance(LatticeDesc* desc, const int32_t* count, int max_count, int steps,
                                  cudaStream_t s);
// Cluster-resident sweeps (sweep_cluster.cu): lattices of one side L <= cluster_max_L()
// kept in the shared memory of one thread-block cluster of C CTAs each (threads per
// CTA, dynamic shared memory per CTA).  cluster_plan gives the plan for `count`
// lattices (C = 0: none fits); the launch runs nsweeps sweeps of every live lattice of
// desc[0..count), each stopping at its limit.
struct ClusterPlan {
    int C = 0;
    int threads = 0;
    size_t smem = 0;
};
int cluster_max_L();
ClusterPlan cluster_plan(int64_t L, int count);
cudaError_t launch_cluster_sweeps(const LatticeDesc* desc, int count, int64_t L, const ClusterPlan& p, int nsweeps,
                                  cudaStream_t s);
// Parameter blocks of the by-value updates (each under the 4 KB kernel-parameter limit).
struct TileChunk {
    static constexpr int kMax = 960;
    int32_t first, n, count;  // entries first .. first+n-1; count >= 0: also set the lattice count
    int32_t v[kMax];
};
struct GatherChunk {
    static constexpr int kMax = 960;
    int32_t n;
    int32_t idx[kMax];
};
// Enqueue a descriptor write, a tile-table write (n entries and the lattice count), and
// the (sweeps, M, E) gather of batch slots idx[0..n) into out[3n] (device-accessible);
// none waits for the stream's earlier work and the host arrays may change on return.
cudaError_t launch_set_desc(LatticeDesc* dst, const LatticeDesc& d, cudaStream_t s);
cudaError_t launch_set_tiles(int32_t* tile_start, int32_t* count_dst, const int32_t* v, int32_t n, int32_t count,
                             cudaStream_t s);
cudaError_t launch_gather(const LatticeDesc* desc, const int32_t* idx, int32_t n, int64_t* out, cudaStream_t s);
cudaError_t launch_packed_init(uint32_t* black, uint32_t* white, int64_t L, uint64_t key, int start,
                               cudaStream_t s);
cudaError_t launch_packed_observe(const uint32_t* black, const uint32_t* white, int64_t L, int64_t* ME,
                                  cudaStream_t s);
// Layout conversion of rows [row0, row0 + nrows); `lat` points at row row0.
cudaError_t launch_pack(const int8_t* lat, uint32_t* black, uint32_t* white, int64_t L, int64_t row0,
                        int64_t nrows, cudaStream_t s);
cudaError_t launch_unpack(const uint32_t* black, const uint32_t* white, int8_t* lat, int64_t L, int64_t row0,
                          int64_t nrows, cudaStream_t s);

cudaError_t launch_int8_init(int8_t* lat, int64_t L, uint64_t key, int start, cudaStream_t s);
cudaError_t launch_int8_half_sweep(int8_t* lat, int64_t L, uint64_t key, uint32_t t2, uint32_t t4, uint32_t all2,
                                   uint32_t all4, uint32_t sweep, int colour, int64_t* hist_slot,
                                   cudaStream_t s);
cudaError_t launch_int8_observe(const int8_t* lat, int64_t L, int64_t* ME, cudaStream_t s);

// Exact moments over hist[first .. first+count), or of the batch lattice desc over its samples from
// `first` on: writes 6 doubles (abs_m, m2, m4, e, e2, binder) and the exact sums (see
// moments.cu), nothing where there is no sample; report[0] = *status (0 for null), report[1] = the
// sweep count.
cudaError_t launch_moments(const LatticeDesc* desc, const int64_t* hist, int64_t first, int64_t count, int64_t N,
                           double* out6, uint64_t* sums, const int* status, int64_t* report, cudaStream_t s);

cudaError_t launch_philox_words(uint64_t key, const uint32_t* ctr4, int64_t n, uint32_t* out, cudaStream_t s);

int sm_count();

// Sets the thread-local message that ising_last_error() returns (api.cu).
void set_last_error(const char* msg);

// Packed sweep kernel configuration helpers (sweep_packed.cu).
int packed_smem_header_bytes(int threads);
// Allows launches with up to max(bytes, header + 2 stages of kStageCapBytes) of dynamic
// shared memory on every instance of the sweep kernel for `threads`.  The limit is
// per kernel, shared by every engine of the process, so it is never set below the
// largest launch any engine can make.
cudaError_t packed_set_smem_limit(int threads, size_t bytes);
// Resident CTAs per SM of the sweep kernel: the single-lattice instance (one) or
// the general one, which the two launch bounds give different register budgets.
cudaError_t packed_occupancy(int threads, size_t smem, int* blocks_per_sm, bool one = false);

}  // namespace ising
