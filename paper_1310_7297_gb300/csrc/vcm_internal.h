// vcm_internal.h -- structures shared by the host runtime (vcm_api.cpp) and
// the sm_103a kernels (vcm_kernels.cu).  Not part of the public C ABI.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/vcm.h"

#ifdef __CUDACC__
#define VCM_HD __host__ __device__
#else
#define VCM_HD
#endif

namespace vcm {

constexpr int kWarps = 4;                 // warps per block of the tile kernel
constexpr int kThreads = kWarps * 32;
constexpr int kPassCap = 2 * kThreads;       // cells listed per round of the grid walk
constexpr int kDistClasses = 128;            // distance classes of the candidate counting sort
// Launches whose requests all have this many patches look at recorded blockers
// before a tile's cull.  What decides is how much of the map one box hides, which
// the host does not know: 33.5 M viewpoints, 100,000 boxes and 64 x 32 patches
// took 1.47 ms without and 1.28 with them where nearly all is hidden, 2.05 and
// 2.04 where more is seen.  The line keeps them from the maps they were slower
// for: 512^2 x 5 viewpoints, 5,000 boxes, 32 x 16 patches 80.0 -> 81.6 us, with
// bits 146.5 -> 149.5.
constexpr int kTileCheckMinPatches = 1024;
constexpr float kBand = 1e-6f;            // FP32 slab margin that is re-decided exactly
constexpr int kMaxBoxCap = 5000;          // candidate boxes a tile stages in shared memory
constexpr int kRowCap = 256;              // patch rows a warp stages for the measure
constexpr int kWarpBoxes = 64;            // boxes of a chunk's list a warp stages
constexpr int kTileBlocks = 8;            // blocks per SM of the tile pass
constexpr long long kTileWaves = 3;         // waves of resident blocks below which a launch's tiles shrink
constexpr int kNodeBoxes = 64;             // nearest candidates that the tile's nodes test
#ifndef VCM_CHECKED
constexpr int kPublishMax = 1 << 20;      // longest list a tile publishes (x 8 blocks x 152 SMs < 2^31)
constexpr int kWideIds = 1 << 24;         // boxes from which a spill region's ids take 4 bytes, not 3
#else   // the checked build's small scenes reach both sides of either limit
constexpr int kPublishMax = 300;
constexpr int kWideIds = 600;
#endif
constexpr int kKeptWarps = 2;             // warps that sweep the viewpoints a tile keeps
constexpr int kSweepBlocks = 6;           // blocks per SM of the second pass
constexpr int kPartsPerWarp = 2;          // parts of chunks the second pass wants per warp
constexpr int kMaxTileViewpoints = 1024;  // viewpoints in one tile (tile_x * tile_y)
constexpr int kClaimRounds = 4096;        // bounded retries of a spill-region claim (2 us pauses)

// Work sharing of the persistent tile kernel, in two passes.  In the first,
// the tiles publish the viewpoints their checks leave open, kChunkVp at a time,
// as chunks; in the second, k_sweep's warps sweep parts of the chunks.
// The work buffer of a launch holds kWorkHeader counters (next tile, and for
// each round records, chunks published, parts taken, id-pool ints used) and
// then the arena:
//   chunk[kChunkCap][kChunkInts]     32 x record index + count, viewpoints (x + 256 y in the tile, 16 bits each)
//   record[kRecCap][kRecInts]        request, candidate count, offset of its ids in the pool, layer, tile origin
//   pool[kPoolInts]                  the records' candidate box ids, in the owner's order
//   blocker[kBlockerCap]             per tile position of each request (many-patch
//                                    launches): a box id that blocked a tile there, or -1
// A launch with many more viewpoints than the arena holds runs in rounds of
// both passes.  A tile whose publication would pass a cap keeps its viewpoints.
constexpr int kChunkVp = 16;
constexpr int kChunkInts = 1 + kChunkVp / 2;
constexpr int kChunkCap = 800000;
constexpr int kRecCap = 131072;
constexpr int kRecInts = 8;
constexpr int kPoolInts = 8 << 20;
constexpr int kBlockerCap = 1 << 20;
constexpr int kWorkHeader = 64;   // ints before the arena (256 bytes)
constexpr int kMaxRounds = 15;    // rounds of a launch: 1 + 4 x 15 counters fit the header
// Where the parts of an arena lie (in ints, after the header).  The defaults are
// those of a work buffer of kWorkBytes; vcm_compute_static lays out a smaller
// one.
struct Arena {
    int chunk_cap = kChunkCap, rec_cap = kRecCap, pool_ints = kPoolInts;
    VCM_HD size_t rec_off() const { return (size_t)chunk_cap * kChunkInts; }
    VCM_HD size_t pool_off() const { return rec_off() + (size_t)rec_cap * kRecInts; }
    VCM_HD size_t blocker_off() const { return pool_off() + (size_t)pool_ints; }
};
constexpr size_t kArenaInts = (size_t)kChunkCap * kChunkInts + (size_t)kRecCap * kRecInts + (size_t)kPoolInts +
                              (size_t)kBlockerCap;
constexpr size_t kWorkBytes = (kWorkHeader + kArenaInts) * sizeof(int);

// Bytes per id of a spill region, and of a block's region (a multiple of 4).
int spill_id_bytes(int n_boxes);
VCM_HD inline size_t spill_region_bytes(int n_boxes, int id_bytes)
{
    return ((size_t)(n_boxes > 0 ? n_boxes : 1) * id_bytes + 3) & ~(size_t)3;
}

// Dynamic shared memory of the tile kernel: box_cap staged boxes, and the ids
// of list_cap candidates.
inline size_t tiles_smem_bytes(int box_cap, int list_cap) { return (size_t)box_cap * 32 + (size_t)list_cap * 4; }

// Device view of the scene and its uniform-grid index.  Boxes are sorted by
// grid cell; `boxes[perm]` holds the same boxes with their coordinates
// permuted into one of the six (u, n, w) target frames, two float4 per box
// (lo.xyz, hi.xyz).  Permutation 0 is the world frame (x, y, z).
struct DevScene {
    const float4 *boxes[6];
    int n_boxes;
    int dims;
    const int *cell_start;     // [n_cells + 1] into the sorted box order
    const float4 *cell_lo;     // [n_cells] bounds of each cell's boxes (world)
    const float4 *cell_hi;
    float gx0, gy0;            // grid origin (world x, y)
    float cell, inv_cell;
    int gnx, gny;
    float overhang;            // how far a cell's bounds reach past the cell
};

// One canonicalised request (host-computed, lattice-exact coordinates).
// Target frame: axis 0 = u (patch columns), 1 = n (normal), 2 = w (rows).
struct DevRequest {
    int dims;
    int au, an, aw;            // world axis of u, n, w
    int perm;                  // index of the box copy in that frame
    float sn;                  // +1 / -1: side of the normal
    float p_n;                 // patch coordinate along the normal axis
    int nu, nw, P, words;
    float measure;             // patch area (3D) or length (2D), metres
    int nx, ny, nl;            // viewpoint grid
    int tile_x, tile_y, tiles_x, tiles_y, n_tiles;
    int nuc, groups, col_passes, rows;   // lane mapping: columns and row groups of a pass, column passes, rows per lane
    int filter_stop;           // kept boxes at which a viewpoint's filter leaves its list to the passes
    float inv_row, row_dev;    // 1 / w step between a lane's rows; how far a row is off an even step
    int blk_base;                // offset of its tile positions in the blocker table, or -1
    const float *u_coord;      // [nu] patch centre coordinate along u
    const float *w_coord;      // [nw] along w (one 0 in 2D)
    const float *x_coord;      // [nx] viewpoint x
    const float *y_coord;      // [ny] viewpoint y
    const float *z_coord;      // [nl] layer heights (one 0 in 2D)
    float u_min, u_max, w_min, w_max;
    float *v_out;
    uint8_t *color_out;
    uint32_t *bits_out;
    vcm_stats *stats;
    float v_ref_given;
    int levels;
    unsigned flags;
    int cone;                  // 1: a field-of-view cone masks the patches
    float cone_c;              // cosine of its half-angle
    float cone_a[3];           // its unit axis, world x, y, z
};

// The rules that the checked build applies to what goes through the arena: the
// places a tile publishes at, and what a chunk's first word, a record (its list's
// ids and its layer among them) and a viewpoint of the chunk name.
VCM_HD inline bool publication_in_bounds(const Arena &a, int rec, int chunk, int chunks, int ids, int n_ids)
{
    return rec >= 0 && rec < a.rec_cap && chunk >= 0 && chunks >= 0 && chunk <= a.chunk_cap - chunks && ids >= 0 &&
           n_ids >= 0 && ids <= a.pool_ints - n_ids;
}
VCM_HD inline bool chunk_in_bounds(const Arena &a, int word)
{
    return word >= 0 && (word >> 5) < a.rec_cap && (word & 31) <= kChunkVp;
}
VCM_HD inline bool record_in_bounds(const Arena &a, const int *rec, const DevRequest *reqs, int n_req, int n_boxes)
{
    return rec[0] >= 0 && rec[0] < n_req && rec[1] >= 0 && rec[1] <= n_boxes && rec[2] >= 0 &&
           rec[2] <= a.pool_ints - rec[1] && rec[3] >= 0 && rec[3] < reqs[rec[0]].nl;
}
VCM_HD inline bool viewpoint_in_bounds(const DevRequest &R, int ix, int iy)
{
    return ix >= 0 && ix < R.nx && iy >= 0 && iy < R.ny;
}

// Launch helpers implemented in vcm_kernels.cu.  All are asynchronous on
// `stream` and return the launch status.
cudaError_t launch_grid_build(const float *d_lo_world, const float *d_hi_world, int n, int dims,
                              float gx0, float gy0, float cell, int gnx, int gny,
                              int *d_cell_of, int *d_count, int *d_order,
                              int *d_cell_start, float4 *const *d_perm_boxes, float4 *d_cell_lo,
                              float4 *d_cell_hi, unsigned *d_overhang_bits, cudaStream_t stream);

// The tile kernel over `n_req` requests (their tiles concatenated,
// `d_tile_prefix` = exclusive prefix of tiles, n_req + 1 entries).  Persistent
// by default: grid_blocks blocks draw tiles from `d_work` (zeroed by the
// caller).  With one_tile, one block per tile, so concurrent launches
// interleave block by block; grid_blocks must then be at least the number of
// blocks that can be resident at once, and `d_spill_busy` (grid_blocks ints,
// all zero between launches) hands out the spill regions.  `d_spill` holds
// grid_blocks regions of spill_region_bytes for candidate lists longer than box_cap.
// `extra` must be set when any request is two-sided or has a field-of-view
// cone: it selects the tile kernel's instantiation that handles them.
// `tile_check` selects the instantiation that looks at recorded blockers (any
// launch may use either; it pays when every request has many patches).
// `share` (persistent launches only): d_work holds `arena` behind its header
// (kWorkBytes for the default one), and a second
// kernel on all sm_count SMs works the open viewpoints that expensive tiles of
// the first published there.
// `total_vp`: the requests' viewpoints, from which the number of rounds follows;
// 0: one round (vcm_compute_static: its arena is small, and rounds that find
// nothing left would cost 8 us each).
// `list_cap` > box_cap: the ids of candidates past the staged boxes are kept in
// shared memory, which must then hold every box of the scene (d_spill is not
// used); otherwise they spill.
// `overlap` false: the tile kernel is not launched ahead of the end of what is
// before it on the stream (k_sweep and the other kernels of a call are).
// `claim_rounds` (1..kClaimRounds) bounds the retries of a one-tile block's
// spill-region claim; a block that gives up runs without a region and sets
// its request's vcm_stats.error to VCM_DEVERR_SPILL_WAIT if its candidate
// list needs one.
cudaError_t launch_tiles(const DevScene &sc, const DevRequest *d_reqs, const int *d_tile_prefix,
                         int n_req, int total_tiles, long long total_vp, int *d_work, int *d_spill, int grid_blocks,
                         int box_cap, bool extra, bool tile_check, int sm_count, cudaStream_t stream,
                         bool one_tile = false,
                         int *d_spill_busy = nullptr, bool share = false, int claim_rounds = kClaimRounds,
                         const Arena &arena = Arena(), int list_cap = 0, bool overlap = true);
// Colors and edge counts for all viewpoints of n_req requests (grid over the
// concatenated viewpoints, `d_vp_prefix` = exclusive prefix, n_req + 1).
cudaError_t launch_quantise(const DevRequest *d_reqs, const long long *d_vp_prefix, int n_req,
                            long long total_vp, cudaStream_t stream);

// Values of one request (d_req[0]) recomputed from the occlusion bits its
// bits_out points at (read only); colors then come from launch_quantise.
// n_rows: its patch rows.  d_list: n_vp ints of scratch for the viewpoints that
// need a measure, and d_n_list their count, 0 before (n_vp <= INT_MAX).
cudaError_t launch_recolor(const DevRequest *d_req, long long n_vp, int n_rows, int sm_count, int *d_list, int *d_n_list,
                           cudaStream_t stream);

// Zero the work counters (d_work[0..kWorkHeader)) and every request's vcm_stats, and set
// n_blockers entries of the blocker table to -1.
cudaError_t launch_prologue(const DevRequest *d_reqs, int n_req, int *d_work, int *d_blockers, long long n_blockers,
                            cudaStream_t stream);
// The same, and write the descriptors (host memory, consumed before the call
// returns; `bytes` at most kDescParamBytes) to d_desc, 16-byte aligned.
constexpr int kDescParamBytes = 32512;   // a kernel's parameters hold 32,764 bytes
cudaError_t launch_prologue_desc(const void *h_desc, size_t bytes, void *d_desc, int n_req, int *d_work, int *d_blockers,
                                 long long n_blockers, cudaStream_t stream);

// Blocks of the tile kernel that fit on one SM for this shared-memory size.
int tiles_blocks_per_sm(int box_cap, int list_cap = 0);

// One-time per-device setup (kernel attributes); must run before any launch is
// captured into a graph.
cudaError_t init_device();

// Device address and size of the file-scope scratch array used by
// vcm_compute_static on the current device (looked up once per device).
cudaError_t static_scratch(void **ptr, size_t *bytes);

}  // namespace vcm
