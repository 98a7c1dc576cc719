// Internal declarations shared by the bridge's translation units (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "emc2_bridge.h"
#include "rules.cuh"

namespace emc2 {

constexpr int kTile = 256;           // points per CTA tile in the per-point kernels
constexpr int kThreads = 256;

// Threads of the kernels that move feature rows when Cf/4 = cf4 is not one of the compiled widths: as many whole
// rows of cf4 columns as 512 threads hold (at least 256: one per point of a tile), so that every thread keeps its
// column and no index is divided inside the loop.  Rows wider than that take the divide.  Rows of an odd number of
// columns are half a sector off at every other row: up to 1 KB an even number of them is taken, so that a CTA's
// stores stay on sectors (132 channels, 1,800 tiles: project_gather 47.7 -> 44.7 us; 36: 23.1 -> 22.0; 52: 27.2 -> 25.1).
constexpr int kMaxRowThreads = 512;
inline int row_threads(int cf4) {
    if (cf4 > kTile) return kThreads;
    const int rows = kMaxRowThreads / cf4;
    return (cf4 <= 64 && (cf4 & 1) ? rows & ~1 : rows) * cf4;
}
// The cell stores.  Large grids: 16-byte units of 96 cell bits and the rank of the unit's first voxel, so that
// one 128-bit load answers a look-up and the scan streams 1.33 bits per cell (a {32 bits, rank} pair per 32
// cells streams 2: 75 instead of 50 MB for four frames of the nuScenes-shaped grid, and the scan is paid by
// the grid's volume).  Small grids: one word per cell.
constexpr uint32_t kUnitCells = 96;
constexpr size_t kScanTileBytes = 8192;   // of the store; the ranking pass takes eighths of them
constexpr uint32_t kBitmapTileCells = (uint32_t)(kScanTileBytes / 16) * kUnitCells;
constexpr uint32_t kTableTileCells = (uint32_t)(kScanTileBytes / 4);
constexpr int kMaxTableCells = 1 << 24;  // a word per cell up to 16 Mi cells per batch (64 MB)
constexpr uint32_t kOverCap = 0x80000000u;  // table word / list entry of a cell over the cap
constexpr int kCursorStride = 8;         // ints between list cursors: one 32-byte sector each

// Kernel kinds, for the launch counters and the optional event timing.
enum KernelKind {
    K_VOX_MARK = 0,
    K_VOX_COUNT,
    K_VOX_RANK,
    K_VOX_ACCUM,
    K_VOX_OVER_FIND,
    K_VOX_OVER_FILL,
    K_VOX_FINALIZE,
    K_ARM_KEYS,
    K_ARM_SORT,
    K_ARM_HASH,
    K_ARM_RANK,
    K_PROJECT_GATHER,
    K_PROJECT_ROUTE,
    K_GATHER_SCATTER,
    K_ROUTE_HIST,
    K_ROUTE_SCAN,
    K_DISPATCH_SCATTER,
    K_SCENE_ROUTE,
    K_POOL_FEATURES,
    K_VIF_SCAN,
    K_VIF_FILL,
    K_VIF_MEAN,
    K_VIF_SAMPLE,
    K_OCCL_FILL,
    K_OCCL_SPLAT,
    K_OCCL_TEST,
    K_CHANNELS_LAST,
    K_RB_MARK,
    K_RB_COUNT,
    K_RB_SCAN,
    K_RB_FILL,
    K_RB_CLEAR,
    K_KINDS
};

enum ScaleMode { MODE_BITMAP = 0, MODE_TABLE = 1 };

// Division of any 32-bit unsigned number by a fixed divisor with a multiply and two shifts
// (Granlund and Montgomery, "Division by invariant integers using multiplication", 1994).
struct FastDiv {
    uint32_t d, m, s1, s2;
#ifdef __CUDACC__
    __device__ __forceinline__ void divmod(uint32_t n, uint32_t& q, uint32_t& r) const {
        const uint32_t t = __umulhi(m, n);
        const uint32_t qq = (t + ((n - t) >> s1)) >> s2;
        r = n - qq * d;
        q = qq;
    }
#endif
};

inline FastDiv make_fast_div(uint32_t d) {
    FastDiv f;
    uint32_t L = 0;
    while (L < 32 && ((uint64_t)1 << L) < d) ++L;
    f.d = d;
    f.m = (uint32_t)((((uint64_t)1 << 32) * (((uint64_t)1 << L) - d)) / d + 1);
    f.s1 = L < 1 ? L : 1;
    f.s2 = L > 0 ? L - 1 : 0;
    return f;
}

// Per-scale grid description and scratch pointers, passed to kernels by value.
struct ScaleDev {
    float mn[3];
    float vs[3];
    float inv[3];           // 1 / vs in fp32 (NaN where that is not a normal number) and how far from an integer
    float margin[3];        // a product with it decides the cell without a divide, see cell_by_product
    int dims[3];            // Gx, Gy, Gz
    FastDiv div[3];         // division by Gx, Gy, Gz
    int cap;                // 0 = none
    int mode;               // ScaleMode
    uint32_t cells;         // cells per frame
    uint32_t tiles;         // 8 KB tiles of `store` for the largest batch, a multiple of kCountTiles
    uint32_t max_ovf;       // most cells that can exceed the cap
    uint32_t max_list;      // entries of acc / cell_list / ovf_list: the most points of a call
    uint32_t* store;        // bitmap: 16-byte units {96 cell bits, rank}; table: one word per cell, its point
                            // count while marking, then its rank or kOverCap | index among the cells over the
                            // cap.  All zero between calls
    int acc_f4;             // float4 per accumulator: 1 or 2, see accumulator_f4
    float4* acc;            // [max voxels][acc_f4] per-voxel accumulators
    uint32_t* cell_list;    // [max voxels] cell id of each unique voxel (table stores: bit 31 = over the cap)
    int* ovf_off;           // per cell over the cap j: start of its points in ovf_list
    int* ovf_cursor;        // per cell over the cap j: points appended so far, at [j * kCursorStride]
    uint32_t* ovf_cell;     // per cell over the cap j: its cell id
    int* ovf_vox;           // per cell over the cap j: its row m in the unique list
    int* ovf_list;          // global point indices of the points in cells over the cap
    int design;             // dedup design of this scale: 0 = this direct-addressed store, 1 = hash, 2 = sort
                            // (dedup_arms.cu); with 1 or 2 the store is not used and rows come from point_rank
    const int* point_rank;  // design != 0: [points of the call] row of every point's voxel, -1 if outside
    int* totals;            // [0] voxels, [1] not 0: the lists of cells over the cap are not used (refuse_lists),
                            // [2] points in cells over the cap, [3] cells over the cap (one 64-bit ticket counter)
};

// Routing tables as the kernels take them (Sec. 3.2 distance rule, per point with visibility).
struct RouteParams {
    int T, E;
    float thr2[EMC2_MAX_THRESHOLDS];    // squared thresholds
    uint8_t lut[16];                    // [visible ? 8 : 0] + number of thresholds reached -> expert
};

// State of the rank scan.
constexpr int kTilesPerGroup = 128;
constexpr int kCountTiles = 4;  // tiles per CTA of the counting pass
struct ScanState {
    uint32_t* tile_voxels[2];   // [tiles] voxels per tile
    uint4* tile_parts[2];       // [tiles] voxels per eighth of a tile, 16 bits each
    uint32_t* group_voxels[2];  // [ceil(tiles / 128)] per group of tiles; zero when the scan begins
    uint32_t* listed;           // parts in `list`; zero when the scan begins
    uint32_t* list;             // [8 * tiles of both scales] parts that hold voxels, in any order: 8 * tile + part; bit 31: scale 1
    uint32_t* marked[2];        // a bit per tile of a store: a cell of it was marked; kNoteCopies of them, zero between calls
    uint32_t note_stride;       // words from one copy of the notes to the next
    int words[2];               // words of `marked` to clear, 0 where the marking pass does not keep it
};

// Where the marking pass notes the tiles that it touches (see keeps_tile_marks and kNoteCopies), or null.
struct TileMarks {
    uint32_t* marked[2];
    uint32_t stride;                        // words from one copy to the next
    uint16_t word0[2][EMC2_MAX_BATCH];      // first word of `marked` that has tiles of the frame, per scale (a store has at most
    uint16_t words[2][EMC2_MAX_BATCH];      // 2,731 words), and how many
};

// What of it is zeroed when a call begins, by whichever kernel marks the cells.
struct ScanReset {
    uint32_t* words;            // group_voxels of both scales and `listed`, side by side
    int n;
    int* totals[2];             // null: nothing to reset (second half of a split batch)
};

// Scratch of the alternative dedup designs (allocated when one is first selected).
struct DedupArm {
    void* slab = nullptr;
    size_t bytes = 0;
    uint32_t* keys[2] = {nullptr, nullptr};     // sort buffers (ping-pong): cell ids ...
    uint32_t* vals[2] = {nullptr, nullptr};     // ... and point indices (hash design: the unique ids)
    int* counts = nullptr;                      // [256][tiles] digit counts of a radix pass
    int* row_tot = nullptr;                     // [256] totals per digit
    int* tile_tot = nullptr;                    // run heads per tile
    int* point_rank[2] = {nullptr, nullptr};    // per scale
    uint32_t* tab_keys = nullptr;               // hash table: cell ids ...
    int* tab_rows = nullptr;                    // ... and their rows
    int* d_total = nullptr;
    uint32_t slots = 0;
};

struct ProfRec {
    int kind;
    cudaEvent_t a, b;
};

}  // namespace emc2

struct emc2_bridge {
    emc2_config_t cfg;
    emc2::ScaleDev scale[2];
    float thr2[EMC2_MAX_THRESHOLDS];
    void* slab = nullptr;
    size_t slab_bytes = 0;
    int* d_status = nullptr;       // sticky device status word
    int* d_tile_counts = nullptr;  // [B, tiles per frame, E]
    int* d_tile_base = nullptr;    // same shape, exclusive bases
    emc2::ScanState scan = {};
    int scan_reset_words = 0;
    int* d_vif_start = nullptr;    // emc2_voxel_image: [max points] list starts, cursors, lists
    int* d_vif_cursor = nullptr;
    int* d_vif_list = nullptr;
    uint4* d_vif_recs = nullptr;   // emc2_voxel_image_sampled: [max points] tap records in list order
    int* d_vif_part = nullptr;     // list slots given out (64 bits, zero between calls), flag of bad counts
    uint32_t* d_rb_bits = nullptr;  // emc2_rulebook: [max points] neighbour bits per voxel
    int* d_rb_counts = nullptr;    // [13][voxel tiles] pairs per (offset, tile), and their prefix sums
    int* d_rb_base = nullptr;
    int max_tiles = 0;
    int tune[EMC2_TUNE_KNOBS] = {0, 1, 0, 0, 0};   // emc2_bridge_set_tuning
    emc2::DedupArm arm;
    int num_sms = 0;               // multiprocessors of the handle's device
    bool overlap = true;           // emc2_bridge_run uses `side` and `rows`
    cudaStream_t side = nullptr;   // stream of stage 1 inside emc2_bridge_run ...
    cudaStream_t rows = nullptr;   // ... or, in small calls, of the rows; of the maps' copy in emc2_bridge_run_host
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr, ev_half = nullptr, ev_copy = nullptr, ev_scan = nullptr;
    int last_cuda_error = 0;
    bool profiling = false;
    int64_t launches[emc2::K_KINDS] = {0};
    double ms[emc2::K_KINDS] = {0};
    std::vector<emc2::ProfRec> recs;
    std::vector<cudaEvent_t> event_pool;
};

namespace emc2 {

// Brackets a launch with events when profiling; always counts it.
struct LaunchScope {
    emc2_bridge* h;
    int kind;
    cudaStream_t st;
    cudaEvent_t a = nullptr, b = nullptr;
    LaunchScope(emc2_bridge* h_, int kind_, cudaStream_t st_);
    ~LaunchScope();
};

int check_cuda(emc2_bridge* h, cudaError_t e);

// `marked`: the cells of this batch are already marked and the BEV image zeroed (by the projection
// kernel of the one-call path); the marking pass is then skipped.  `chained`: that kernel is the call's previous work on
// `st`, see launch_chained.
int launch_voxelize(emc2_bridge* h, int B, int N, const float* d_points, int32_t* const d_coords[2],
                    int32_t* const d_counts[2], float* const d_mean[2], int32_t* const d_point_voxel[2],
                    const int32_t capacity[2], int32_t* d_num_voxels, float* d_bev, cudaStream_t st,
                    bool marked = false, bool chained = false);
int dedup_arm_alloc(emc2_bridge* h);
int launch_dedup_arm(emc2_bridge* h, int s, int design, int B, int N, const float* d_points, int capacity,
                     int32_t* d_num_voxels, cudaStream_t st);
int launch_project_gather(emc2_bridge* h, int B, int N, const float* d_points, const float* d_proj,
                          const float* d_feat, float* d_uvd, uint8_t* d_vis_mask, int8_t* d_cam,
                          float* d_gathered, cudaStream_t st);
int launch_route_dispatch(emc2_bridge* h, int B, int N, const float* d_points, const uint8_t* d_vis_mask,
                          const float* d_gathered, uint8_t* d_expert, int32_t* d_offsets, int32_t* d_perm,
                          float* d_points_out, float* d_feat_out, cudaStream_t st);

#ifdef __CUDACC__
// Launches a kernel that may be set up while its predecessor in the stream still drains (programmatic dependent
// launch); for kernels that follow another kernel of the same call on the same stream.  Every kernel launched this
// way calls await_predecessor() before it touches memory and, when its own work is done, release_successor().
// Such a kernel can be resident while its predecessor still writes: what a kernel of the same call writes is read
// through plain pointers, never through `const __restrict__` ones or __ldg, whose loads the compiler may move ahead
// of the wait.  The call's own inputs are complete before the first kernel of a call, which is launched plainly.
// Released earlier, the successor's CTAs would hold places on the SMs that the kernels of the other stream need.
// us per call queued behind others: one small frame 35 -> 30, stage calls with occlusion 155 -> 140, voxels and rulebooks
// 261 -> 239 (B200).  A call on an idle GPU gains less: there the host's enqueuing of its kernels and events sets the pace.
// `chained` false: an ordinary launch, for a kernel that follows a copy or an event wait, or that can be the first of
// its call.
template <typename... P, typename... A>
inline void launch_kernel(bool chained, void (*kernel)(P...), dim3 grid, unsigned threads, size_t shared, cudaStream_t st, const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = shared;
    cfg.stream = st;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = chained ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <typename... P, typename... A>
inline void launch_chained(void (*kernel)(P...), dim3 grid, unsigned threads, size_t shared, cudaStream_t st, const A&... args) {
    launch_kernel(true, kernel, grid, threads, shared, st, args...);
}
#endif

inline ScanReset scan_reset(const emc2_bridge* h) {
    ScanReset r;
    r.words = h->scan.group_voxels[0];
    r.n = h->scan_reset_words;
    for (int s = 0; s < 2; ++s) r.totals[s] = h->scale[s].totals;
    return r;
}

// Grid of a marking pass: `tiles` CTAs per frame, (tiles * frames of a group, groups); `group` divides by the frames of a group.
inline dim3 marking_grid(int tiles, int B, const FastDiv& group) { return dim3(tiles * group.d, (B + group.d - 1) / group.d); }

// Bytes of both stores of a frame.
inline uint64_t store_bytes(const emc2_bridge* h) {
    uint64_t bytes = 0;
    for (int s = 0; s < 2; ++s) {
        const ScaleDev& g = h->scale[s];
        if (!g.design) bytes += g.mode == MODE_BITMAP ? g.cells / kUnitCells * 16ull : g.cells * 4ull;
    }
    return bytes;
}

// Whether the marking pass of this call notes the tiles it touches; a handle's other dedup designs have no stores.
inline bool keeps_tile_marks(const emc2_bridge* h, int B, int N) {
    uint64_t words = 0;
    for (int s = 0; s < 2; ++s) {
        const ScaleDev& g = h->scale[s];
        if (g.design) return false;
        const bool bitmap = g.mode == MODE_BITMAP;
        words += most_frame_words(g.cells, bitmap ? kBitmapTileCells : kTableTileCells);
    }
    return keeps_frame_notes(store_bytes(h), words, B, N);
}

inline TileMarks tile_marks(const emc2_bridge* h, int B, int N) {
    TileMarks m = {};
    if (!keeps_tile_marks(h, B, N)) return m;
    m.stride = h->scan.note_stride;
    for (int s = 0; s < 2; ++s) {
        const ScaleDev& g = h->scale[s];
        const uint32_t per = g.mode == MODE_BITMAP ? kBitmapTileCells : kTableTileCells;
        m.marked[s] = h->scan.marked[s];
        for (int b = 0; b < B; ++b) {
            m.word0[s][b] = (uint16_t)frame_first_word((uint32_t)b, g.cells, per);
            m.words[s][b] = (uint16_t)frame_words((uint32_t)b, g.cells, per);
        }
    }
    return m;
}

// Whether the marking kernels zero a BEV image of n floats: whole float4, counted in 32 bits (a grid has far less than 2^30 threads).
inline bool bev_by_kernel(size_t n) { return (n & 3) == 0 && n >> 2 < (size_t)3 << 30; }

inline RouteParams route_params(const emc2_bridge* h) {
    RouteParams rp;
    rp.T = h->cfg.num_thresholds;
    rp.E = h->cfg.num_experts;
    for (int k = 0; k < EMC2_MAX_THRESHOLDS; ++k) rp.thr2[k] = h->thr2[k];
    for (int k = 0; k < 16; ++k) rp.lut[k] = h->cfg.lut[k >> 3][k & 7];
    return rp;
}

int launch_occlusion(emc2_bridge* h, int B, int N, const float* d_points, const float* d_proj,
                     const uint8_t* d_vis_mask, int cell, float margin, uint32_t* d_zbuf, uint8_t* d_occ_mask,
                     uint8_t* d_clear_mask, cudaStream_t st);
int launch_voxel_image(emc2_bridge* h, int B, int N, int capacity, const int32_t* d_point_voxel,
                       const int32_t* d_counts, const int32_t* d_num_voxels, const uint8_t* d_vis_mask,
                       const float* d_gathered, const float* d_uvd, const int8_t* d_cam, const float* d_feat,
                       float* d_vox_img, int32_t* d_vox_img_count, cudaStream_t st, int pool = 1);
int launch_rulebook(emc2_bridge* h, int scale, int capacity, const int32_t* d_coords, const int32_t* d_num_voxels,
                    int32_t* d_rule_offsets, int32_t* d_rule_in, int32_t* d_rule_out, long long pair_capacity,
                    cudaStream_t st);
int launch_channels_last(emc2_bridge* h, int B, const float* d_planar, float* d_feat, cudaStream_t st);
int launch_pool_features(emc2_bridge* h, int B, int p, const float* d_feat, float* d_pooled, cudaStream_t st);
int launch_scene_route(emc2_bridge* h, int B, const int32_t* d_offsets, const uint8_t* priority, int min_points,
                       int32_t* d_scene_expert, cudaStream_t st);
// Tile histograms (handle scratch) of frames [b0, b0 + B) -> d_offsets (of frame b0 on) and tile bases.
// `chained` (here and below): the call's previous work on `st` is one kernel, see launch_chained.
void launch_route_scan(emc2_bridge* h, int b0, int B, int tiles, int32_t* d_offsets, bool chained, cudaStream_t st);
// Stages 2 - 4 in one pass over the feature rows (the one-call path), in two parts: projection +
// routing per point (which, with `d_bev_to_zero`/`mark`, also marks the voxel cells of both scales
// and zeroes the BEV image, so that stage 1 reads the points once less), then, after launch_route_scan, the rows.
int launch_project_route(emc2_bridge* h, int b0, int B, int N, const float* d_points, const float* d_proj,
                         float* d_uvd, uint8_t* d_vis_mask, int8_t* d_cam, uint8_t* d_expert, bool mark,
                         float* d_bev_to_zero, int bev_frames, const TileMarks& marks, cudaStream_t st);
int launch_gather_scatter(emc2_bridge* h, int b0, int B, int N, const float* d_points, const float* d_feat,
                          const float* d_uvd, const int8_t* d_cam, float* d_gathered, const uint8_t* d_expert,
                          int32_t* d_perm, float* d_points_out, float* d_feat_out, bool chained, cudaStream_t st);

// ---------------------------------------------------------------- device helpers
#ifdef __CUDACC__

// See launch_chained.  What the predecessors in the stream wrote is visible after the first call; the second one
// lets the successor be set up (it waits for the end of this kernel all the same).
__device__ __forceinline__ void await_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void release_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Loads `nfloats` consecutive floats starting at a 16-byte aligned address into shared
// memory with 128-bit loads (scalar loads for a ragged tail).
__device__ __forceinline__ void load_tile_f32(const float* __restrict__ src, int nfloats, float* smem) {
    const int nvec = nfloats >> 2;
    const float4* s4 = reinterpret_cast<const float4*>(src);
    float4* d4 = reinterpret_cast<float4*>(smem);
    for (int i = threadIdx.x; i < nvec; i += blockDim.x) d4[i] = __ldg(s4 + i);
    for (int i = (nvec << 2) + threadIdx.x; i < nfloats; i += blockDim.x) smem[i] = __ldg(src + i);
}

// Cell id of a point inside the whole batch, or 0xFFFFFFFF if outside the grid.
__device__ __forceinline__ uint32_t cell_of(const ScaleDev& g, float x, float y, float z, int b) {
    int ix, iy, iz;
    if (!cell_xyz(g, x, y, z, ix, iy, iz)) return 0xFFFFFFFFu;
    return (((uint32_t)b * g.dims[2] + iz) * g.dims[1] + iy) * g.dims[0] + ix;
}

// Bit `cell` of a bitmap store: its unit and its place in it.
__device__ __forceinline__ uint32_t unit_of(uint32_t cell, uint32_t& pos) {
    const uint32_t u = cell / kUnitCells;
    pos = cell - u * kUnitCells;
    return u;
}

// Set bits of a unit below place `pos`.
__device__ __forceinline__ uint32_t bits_below(const uint4& q, uint32_t pos) {
    const uint32_t part = (1u << (pos & 31u)) - 1u;
    if (pos < 32u) return __popc(q.x & part);
    if (pos < 64u) return __popc(q.x) + __popc(q.y & part);
    return __popc(q.x) + __popc(q.y) + __popc(q.z & part);
}

// Marks the cells of one point in both scales' stores: one fire-and-forget reduction each (OR into
// the bit word, ADD into the cell's point count).  tile[]: their tiles of the stores, -1 where there is none.
__device__ __forceinline__ void mark_point(const ScaleDev& s0, const ScaleDev& s1, float x, float y, float z, int b,
                                           int tile[2]) {
#pragma unroll
    for (int sc = 0; sc < 2; ++sc) {
        const ScaleDev& g = sc ? s1 : s0;
        tile[sc] = -1;
        if (g.design) continue;                   // another dedup design: no store to mark
        const uint32_t cell = cell_of(g, x, y, z, b);
        if (cell == 0xFFFFFFFFu) continue;
        // Results unused: these compile to reductions, which the thread does not wait for.
        if (g.mode == MODE_BITMAP) {
            uint32_t pos;
            const uint32_t u = unit_of(cell, pos);
            atomicOr(&g.store[4 * (size_t)u + (pos >> 5)], 1u << (pos & 31u));
            tile[sc] = (int)(u / (kBitmapTileCells / kUnitCells));
        } else {
            atomicAdd(&g.store[cell], 1u);
            tile[sc] = (int)(cell / kTableTileCells);
        }
    }
}

// ---- the tiles of the stores that a CTA of a marking pass touches, all of one frame
struct FrameTiles {
    __align__(16) uint8_t seen[kMarkWords * 32];        // a byte per tile, scale 1 behind scale 0
};

// Shared memory for them where the kernel keeps notes.
template <bool kNote>
__device__ __forceinline__ FrameTiles* frame_tiles() {
    if constexpr (kNote) {
        __shared__ FrameTiles tiles;
        return &tiles;
    } else {
        return nullptr;
    }
}

// The caller synchronises the CTA before the first note_tiles and before publish_tiles.
__device__ __forceinline__ void begin_tiles(FrameTiles& f) {
    if (threadIdx.x < kMarkWords * 2) reinterpret_cast<uint4*>(f.seen)[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
}

__device__ __forceinline__ void note_tiles(FrameTiles& f, const TileMarks& to, int b, const int tile[2]) {
    if (tile[0] >= 0) f.seen[tile[0] - 32 * (int)to.word0[0][b]] = 1;
    if (tile[1] >= 0) f.seen[tile[1] - 32 * ((int)to.word0[1][b] - (int)to.words[0][b])] = 1;
}

// One fire-and-forget reduction per word, in copy `copy` % kNoteCopies of the notes of frame b.
__device__ __forceinline__ void publish_tiles(const FrameTiles& f, const TileMarks& to, int b, uint32_t copy) {
    const uint32_t t = threadIdx.x, n0 = to.words[0][b];
    if (t >= n0 + to.words[1][b]) return;
    const uint4* bytes = reinterpret_cast<const uint4*>(f.seen) + 2 * t;
    const uint4 p = bytes[0], q = bytes[1];
    const uint32_t mine = bits_of_bytes(p.x) | bits_of_bytes(p.y) << 4 | bits_of_bytes(p.z) << 8 | bits_of_bytes(p.w) << 12 |
                          bits_of_bytes(q.x) << 16 | bits_of_bytes(q.y) << 20 | bits_of_bytes(q.z) << 24 | bits_of_bytes(q.w) << 28;
    uint32_t* w = t < n0 ? to.marked[0] + to.word0[0][b] + t : to.marked[1] + to.word0[1][b] + (t - n0);
    if (mine) atomicOr(w + (copy % kNoteCopies) * to.stride, mine);
}

// By one CTA.
__device__ __forceinline__ void reset_scan(const ScanReset& r) {
    for (int i = threadIdx.x; i < r.n; i += blockDim.x) r.words[i] = 0u;
    if (threadIdx.x == 0 && r.totals[0]) {
        *reinterpret_cast<int4*>(r.totals[0]) = make_int4(0, 0, 0, 0);
        *reinterpret_cast<int4*>(r.totals[1]) = make_int4(0, 0, 0, 0);
    }
}

// Spread over the whole grid.
__device__ __forceinline__ void zero_bev(float4* bev, uint32_t n4) {
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t step = gridDim.x * gridDim.y * blockDim.x;
    for (uint32_t i = (blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x; i < n4; i += step) __stcs(bev + i, zero);
}

__device__ __forceinline__ int warp_sum(int v) { return __reduce_add_sync(0xFFFFFFFFu, v); }

// ---- stable order of a 256-point tile by expert (used by every kernel that dispatches rows)
template <int C>
struct TileOrder {
    int dest[kTile];                                  // row of every point in the frame's output
    int wcnt[kTile / 32][EMC2_MAX_EXPERTS];           // points of expert k in warp w
    int base[EMC2_MAX_EXPERTS];                       // first row of the tile's points of expert k
    float pts[C == 4 ? 1 : kTile * C];                // five floats per point: the point rows in expert order ...
    int to[C == 4 ? 1 : kTile];                       // ... and the rows they go to
};

template <int C>
struct TilePoint {
    int e;                                            // expert, -1 past the tile
    float f[C];
};

// What a thread needs of point i0 + t, requested before anything waits.  `tile_base`: the tile's E bases.
template <int C>
__device__ __forceinline__ TilePoint<C> load_tile_point(TileOrder<C>& s, const float* __restrict__ pts, const uint8_t* expert,
                                                        const int* tile_base, size_t g0, int npts, int E) {
    const int t = threadIdx.x, k = t - ((int)blockDim.x - EMC2_MAX_EXPERTS);
    if (k >= 0) s.base[k] = k < E ? tile_base[k] : 0;
    TilePoint<C> p;
    p.e = -1;
    if (t < npts) {
        p.e = (int)expert[g0 + t];
        const float* q = pts + (g0 + t) * C;
        if (C == 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(q));
            p.f[0] = v.x; p.f[1] = v.y; p.f[2] = v.z; p.f[3] = v.w;
        } else {
#pragma unroll
            for (int c = 0; c < C; ++c) p.f[c] = __ldg(q + c);
        }
    }
    return p;
}

// Fills s.dest, writes the permutation and moves the point rows; f0: first row of the frame, i0: first point of
// the tile.  At least kTile threads, all of which call it; s.dest is ready on return.
// Scattered a float at a time the rows of five floats cost 16 us of the 188 that gather_scatter_kernel took on four
// nuScenes-shaped frames.  They are put into expert order in shared memory instead, where the rows of one expert
// are one contiguous run of the output, and leave as whole sectors; a row of four floats is one 16-byte store.
template <int C>
__device__ __forceinline__ void order_tile(TileOrder<C>& s, const TilePoint<C>& p, int32_t* perm, float* pts_out, size_t f0,
                                           int i0, int npts, int E) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int rank = 0;
    if (t < kTile) {
        for (int k = 0; k < E; ++k) {
            const unsigned m = __ballot_sync(0xFFFFFFFFu, p.e == k);
            if (p.e == k) rank = __popc(m & ((1u << lane) - 1u));
            if (lane == 0) s.wcnt[warp][k] = __popc(m);
        }
    }
    __syncthreads();
    if (t < kTile) {
        // Lane k: the tile's points of expert k in earlier warps, and (five floats) those of smaller experts.
        int before = 0, all = 0, start = 0;
        if (lane < E) {
#pragma unroll
            for (int w = 0; w < kTile / 32; ++w) {
                const int n = s.wcnt[w][lane];
                if (w < warp) before += n;
                all += n;
            }
        }
        if (C != 4) {
            int inc = all;
#pragma unroll
            for (int d = 1; d < EMC2_MAX_EXPERTS; d <<= 1) {
                const int y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
                if (lane >= d) inc += y;
            }
            start = __shfl_sync(0xFFFFFFFFu, inc - all, max(p.e, 0));
        }
        rank += __shfl_sync(0xFFFFFFFFu, before, max(p.e, 0));
        if (t < npts) {
            const int d = s.base[p.e] + rank;
            s.dest[t] = d;
            perm[f0 + d] = i0 + t;
            if (C == 4) {
                float* dst = pts_out + (f0 + d) * C;      // the caller's buffer may have any alignment
                if ((reinterpret_cast<uintptr_t>(pts_out) & 15) == 0) {
                    *reinterpret_cast<float4*>(dst) = make_float4(p.f[0], p.f[1], p.f[2], p.f[3]);
                } else {
#pragma unroll
                    for (int c = 0; c < C; ++c) dst[c] = p.f[c];
                }
            } else {
#pragma unroll
                for (int c = 0; c < C; ++c) s.pts[(start + rank) * C + c] = p.f[c];
                s.to[start + rank] = d;
            }
        }
    }
    __syncthreads();
    if (C != 4) {
        float* dst = pts_out + f0 * C;
        for (int i = t; i < npts * C; i += blockDim.x) {
            const int r = i / C, c = i - r * C;
            dst[(size_t)s.to[r] * C + c] = s.pts[i];
        }
    }
}

// ---- bilinear sampling of the channels-last feature maps (used by every kernel that blends rows)
constexpr uint32_t kZeroRow = 0xFFFFFFFFu;

__device__ __forceinline__ float4 blend(const float4& f00, const float4& f01, const float4& f10, const float4& f11,
                                        float wx, float wy) {
    const float ax = 1.0f - wx, ay = 1.0f - wy;
    float4 o;
    o.x = ay * (ax * f00.x + wx * f01.x) + wy * (ax * f10.x + wx * f11.x);
    o.y = ay * (ax * f00.y + wx * f01.y) + wy * (ax * f10.y + wx * f11.y);
    o.z = ay * (ax * f00.z + wx * f01.z) + wy * (ax * f10.z + wx * f11.z);
    o.w = ay * (ax * f00.w + wx * f01.w) + wy * (ax * f10.w + wx * f11.w);
    return o;
}

// Tap record of a point seen by camera `cam` of frame b at pixel (u, v): {float4 index of tap
// (y0, x0), clamp flags, wx, wy}; kZeroRow in .x for a point no camera sees.
__device__ __forceinline__ uint4 tap_record(int b, int cam, float u, float v, int K, int Hf, int Wf, int cf4,
                                            float inv_stride, float offset) {
    uint4 rec = make_uint4(kZeroRow, 0u, 0u, 0u);
    if (cam >= 0 && cam < K) {
        // Texel coordinates: one fp32 subtraction, then an exact scaling (the stride is a power of
        // two).  Taps are clamped to the map on every side.
        const float fx = __fsub_rn(u, offset) * inv_stride, fy = __fsub_rn(v, offset) * inv_stride;
        const float flx = floorf(fx), fly = floorf(fy);
        int x0 = (int)flx, y0 = (int)fly;
        const int x1 = max(min(x0 + 1, Wf - 1), 0), y1 = max(min(y0 + 1, Hf - 1), 0);
        x0 = max(min(x0, Wf - 1), 0);
        y0 = max(min(y0, Hf - 1), 0);
        const uint32_t map = ((uint32_t)b * K + cam) * Hf;
        rec.x = ((map + y0) * Wf + x0) * (uint32_t)cf4;
        rec.y = (uint32_t)(x1 - x0) | ((uint32_t)(y1 - y0) << 1);
        rec.z = __float_as_uint(fx - flx);
        rec.w = __float_as_uint(fy - fly);
    }
    return rec;
}

// Blended feature column c of the row described by `rec` (zeros for kZeroRow).
__device__ __forceinline__ float4 gather_column(const float4* __restrict__ feat, const uint4& rec, int c, uint32_t cf4,
                                                uint32_t row_stride) {
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    if (rec.x != kZeroRow) {
        const float4* p = feat + rec.x + c;
        const uint32_t dx = (rec.y & 1u) ? cf4 : 0u, dy = (rec.y & 2u) ? row_stride : 0u;
        const float4 f00 = __ldg(p), f01 = __ldg(p + dx), f10 = __ldg(p + dy), f11 = __ldg(p + dy + dx);
        o = blend(f00, f01, f10, f11, __uint_as_float(rec.z), __uint_as_float(rec.w));
    }
    return o;
}


#endif  // __CUDACC__

}  // namespace emc2
