// Stage 1 of the bridge: two-scale voxelization, dedup in canonical order, per-voxel counts
// and means, BEV scatter (Sec. 3.1 preprocessing; BEV for the 2D expert of Sec. 3.3).
//
// Dedup is direct-addressed, with no sort and no hash probing.  Large grids keep one bit per
// cell: the store is an array of units {96 cell bits, rank} in cell order.  Grids small enough
// keep one word per cell, its point count.  "Rank" is the number of occupied cells before this
// unit / cell in ascending (b, z, y, x) order, which is the canonical voxel order, so a point finds
// its voxel row with ONE 16- or 4-byte load plus a popcount, and no sort is ever needed.
//
//   vox_mark      every point marks its two cells with one fire-and-forget reduction each;
//                 the same launch zeroes the BEV image.
//   vox_count,    the rank scan, two launches: voxels per tile of the store and eighth of it (of the tiles that the marking
//                 pass noted, where it notes them), then the exclusive prefix
//   vox_rank      sums (the parallel prefix-sum index search of Sec. 3.6) are written into the rank
//                 fields and the occupied cell ids listed in that order; the bookkeeping of cells over
//                 the cap is laid out.
//   vox_accum     every point looks its rank up, writes point_voxel and adds itself to its
//                 voxels' accumulators with one or two fp32 vector reductions (offsets from the cell
//                 corner, the other channels).  Points are counted in the words of a table store while they are
//                 marked; on a bitmap scale here, in the caller's array (four channels, no cap) or in the accumulator.
//                 Points of cells over the cap go to per-cell lists instead.
//   vox_finalize  a warp per 32 consecutive voxels: coordinates from the listed cell id, count,
//                 mean and BEV cell, with contiguous row traffic, and the store back to zero; in the same launch
//                 one warp per cell over the cap keeps the
//                 `cap` lowest point indices (keep-first-by-index) and sums them in fp64.
//
// Writes and reductions that land in one 32-byte sector are served one after another by the
// L2 (about 10 ns each on B200), so nothing here funnels many points into a shared flag or
// counter: the contended words are the cells themselves and the notes of their tiles.  The cost of a call follows the
// occupied tiles, not the grid volume, except for one streaming read of the store where no notes are kept.
#include "bridge_internal.cuh"

namespace emc2 {
namespace {

constexpr int kStatusCapacity = 1;
// The cell store held more than one call's points can set, or a cell that none of them marked.  A call that keeps notes looks
// at the noted tiles only: what two calls on one handle at once left in another tile stays there until some call marks a
// cell of that tile, and is found, reported (on a bitmap scale, by its missing points) and cleared then.
constexpr int kStatusDirtyStore = 8;

// Where a point's cell sits in the unique list.
struct Slot {
    int m;      // row in the unique list, -1 if the point is outside the grid
    int j;      // rank among cells over the cap, -1 if the cell is not over it
};

__device__ __forceinline__ Slot slot_of(const ScaleDev& g, uint32_t cell, long long point) {
    Slot s;
    s.m = -1; s.j = -1;
    if (cell == 0xFFFFFFFFu) return s;
    if (g.design) {                               // hash / sort design: the row was computed per point
        s.m = g.point_rank[point];
        return s;
    }
    if (g.mode == MODE_BITMAP) {
        uint32_t pos;
        const uint32_t u = unit_of(cell, pos);
        const uint4 q = reinterpret_cast<const uint4*>(g.store)[u];
        s.m = (int)(q.w + bits_below(q, pos));
    } else {
        const uint32_t w = g.store[cell];
        if (w & kOverCap) s.j = (int)(w & ~kOverCap);
        else s.m = (int)w;
    }
    return s;
}

// A bitmap scale with accumulators of 16 bytes: the points of every voxel are counted in the caller's array.
__device__ __forceinline__ bool counts_in_output(const ScaleDev& g) { return g.mode == MODE_BITMAP && g.acc_f4 == 1; }

// Lower corner of cell i along one axis; both per-point and per-voxel code use this value.
__device__ __forceinline__ float cell_corner(float mn, float vs, int i) { return __fmaf_rn((float)i, vs, mn); }

// ------------------------------------------------------------------ pass 1: mark cells
// See marking_grid; tiles never straddle frames.
template <int C>
__global__ void __launch_bounds__(kThreads)
vox_mark_kernel(const float* __restrict__ pts, int B, int N, const FastDiv group, const __grid_constant__ ScaleDev s0, const __grid_constant__ ScaleDev s1,
                float4* bev, uint32_t bev_n4, ScanReset reset, TileMarks marks) {
    __shared__ FrameTiles tiles;
    uint32_t tile, in_group;
    group.divmod(blockIdx.x, tile, in_group);
    const int b = (int)(blockIdx.y * group.d + in_group);
    const int i = (int)(tile * kThreads + threadIdx.x);
    if (b >= B) N = 0;                            // the last group can have fewer frames
    float x = 0.f, y = 0.f, z = 0.f;
    if (i < N) {
        const float* p = pts + ((size_t)b * N + i) * C;
        if (C == 4) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(p));
            x = q.x; y = q.y; z = q.z;
        } else {
            x = __ldg(p); y = __ldg(p + 1); z = __ldg(p + 2);
        }
    }
    if (marks.marked[0] && b < B) {
        begin_tiles(tiles);
        __syncthreads();
    }
    if (i < N) {
        int tile[2];
        mark_point(s0, s1, x, y, z, b, tile);
        if (marks.marked[0]) note_tiles(tiles, marks, b, tile);
    }
    if (blockIdx.x + blockIdx.y == 0) reset_scan(reset);
    // The BEV image is zeroed here, spread over the whole grid, so it costs no extra launch.
    if (bev) zero_bev(bev, bev_n4);
    if (marks.marked[0] && b < B) {
        __syncthreads();
        publish_tiles(tiles, marks, b, tile);
    }
    release_successor();
}

// ------------------------------------------------------------------ pass 2: ranks
struct ScanArgs {
    ScaleDev s[2];
    int capacity[2];
    int32_t* counts[2];         // the caller's: written for a table store, cleared where vox_accum counts in them
    int32_t* num_voxels;
    int* status;
    int tiles[2];               // 8 KB tiles covering this call's B frames
    ScanState st;
};

// Two launches.
//   vox_count   voxels per 8 KB tile of the store and per eighth of it (a part: 32 sectors), their sum per 128 tiles, and a
//               list of the parts that hold any (most of a fine grid is empty space).  One kernel streams the whole store, a CTA
//               per four tiles; another, where the marking pass keeps notes (see keeps_frame_notes), reads the noted tiles only.
//   vox_rank    a warp per listed part finds the voxels before it (groups of tiles before its group, tiles of the group
//               and parts of the tile before it: a load each), ranks its units or cells and lists the
//               occupied cells in rank order.
// The counting is bound by the read of the store or of the noted tiles, vox_rank by the latency of
// its three dependent round trips and by the parts on the ground plane that hold most voxels: a lane
// has one sector of 32 bytes, and a warp lists the cells of its 32 sectors together.  Nothing in its loop waits for another
// warp.  By events, us, with a CTA per listed tile and three barriers each / now: tiny frame 12.8 / 11.5, eight KITTI-shaped
// frames 33.7 / 26.1, four nuScenes-shaped 33.0 / 28.2, 32 KITTI-shaped frames of 262,144 points 146.8 / 99.7, of 524,288, which take
// more tickets for cells over the cap, 210 / 143.  (As it was first, cells listed by sectors and accumulators of 32 bytes, the
// second to fourth of these took 28.3, 30.6 and 125, with a warp for the empty parts of the listed tiles too 32.7, 30.8 and 137,
// with the next part's sectors requested ahead 29.9, 30.3 and 125.)
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
        if (lane >= d) x += y;
    }
    return x;
}

// Occupied cells of a sector: two units or eight cells.
__device__ __forceinline__ uint32_t sector_voxels(bool bitmap, const uint4& p, const uint4& q) {
    if (bitmap) return __popc(p.x) + __popc(p.y) + __popc(p.z) + __popc(q.x) + __popc(q.y) + __popc(q.z);
    return (p.x != 0u) + (p.y != 0u) + (p.z != 0u) + (p.w != 0u) + (q.x != 0u) + (q.y != 0u) + (q.z != 0u) + (q.w != 0u);
}

constexpr int kScanSectors = (int)(kScanTileBytes / 32);          // 32-byte sectors per tile
static_assert(kScanSectors == kThreads, "vox_count_kernel gives a thread one sector of each of its tiles");

// Voxels of the kCountTiles tiles from tile0 on; `which`: those to look at, a bit each.
__device__ __forceinline__ void count_tiles(const ScanArgs& a, uint32_t (*s_warp)[kThreads / 32], int sc, int tile0, uint32_t which) {
    constexpr int kWarps = kThreads / 32;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const ScaleDev& g = a.s[sc];
    const uint4* p = reinterpret_cast<const uint4*>(g.store) + ((size_t)tile0 * kScanSectors + t) * 2;
    uint4 x[kCountTiles][2];
#pragma unroll
    for (int u = 0; u < kCountTiles; ++u) {
        x[u][0] = x[u][1] = make_uint4(0u, 0u, 0u, 0u);
        if (which >> u & 1u) {
            x[u][0] = p[u * kScanSectors * 2];
            x[u][1] = p[u * kScanSectors * 2 + 1];
        }
    }
#pragma unroll
    for (int u = 0; u < kCountTiles; ++u) {
        const uint32_t n = __reduce_add_sync(0xFFFFFFFFu, sector_voxels(g.mode == MODE_BITMAP, x[u][0], x[u][1]));
        if (lane == 0) s_warp[u][warp] = n;
    }
    __syncthreads();
    if (t < kCountTiles) {
        uint32_t n = 0, pair[kWarps / 2];
#pragma unroll
        for (int w = 0; w < kWarps; w += 2) {
            n += s_warp[t][w] + s_warp[t][w + 1];
            pair[w / 2] = s_warp[t][w] | s_warp[t][w + 1] << 16;          // a part holds at most 32 * 192 voxels
        }
        a.st.tile_voxels[sc][tile0 + t] = n;
        a.st.tile_parts[sc][tile0 + t] = make_uint4(pair[0], pair[1], pair[2], pair[3]);
        // One ticket per CTA: tickets on one address are served one after another (about 10 ns each).
        constexpr unsigned kAll = (1u << kCountTiles) - 1u;
        uint32_t held = 0u;                                       // a bit per part that holds voxels
#pragma unroll
        for (int w = 0; w < kWarps; ++w) held |= s_warp[t][w] != 0u ? 1u << w : 0u;
        const uint32_t mine = __popc(held);
        uint32_t at = mine;
#pragma unroll
        for (int d = 1; d < kCountTiles; d <<= 1) {
            const uint32_t y = __shfl_up_sync(kAll, at, d);
            if (t >= d) at += y;
        }
        const uint32_t sum = __reduce_add_sync(kAll, n);          // the CTA's tiles are all in one group
        uint32_t first = 0;
        if (t == kCountTiles - 1 && at) {
            atomicAdd(&a.st.group_voxels[sc][tile0 / kTilesPerGroup], sum);
            first = atomicAdd(a.st.listed, at);
        }
        at += __shfl_sync(kAll, first, kCountTiles - 1) - mine;
        for (uint32_t entry = (sc ? 0x80000000u : 0u) | (uint32_t)(tile0 + t) << 3; held; held &= held - 1u)
            a.st.list[at++] = entry | (uint32_t)__ffs(held) - 1u;
    }
}

__global__ void __launch_bounds__(kThreads) vox_count_kernel(const __grid_constant__ ScanArgs a) {
    await_predecessor();
    __shared__ uint32_t s_warp[kCountTiles][kThreads / 32];
    int tile0 = (int)blockIdx.x * kCountTiles;
    const int sc = tile0 < a.tiles[1] ? 1 : 0;
    if (!sc) tile0 -= a.tiles[1];
    count_tiles(a, s_warp, sc, tile0, 15u);
    release_successor();
}

// The same where the marking pass noted the tiles it touched: only those are looked at (vox_rank clears the notes).  A
// fixed grid of CTAs, each with at most kThreads groups of four tiles.  us by events, without / with notes: eight KITTI-shaped
// frames (127 MB of stores) 28.5 / 16.8, and project_route, which does the marking, 32.3 / 33.2; four nuScenes-shaped ones 16.9 / 11.5
// and 35.4 / 37.4; 32 KITTI-shaped ones of 262,144 points 88.5 / 50.0 and 154 / 161.  See keeps_frame_notes for whole calls.
__global__ void __launch_bounds__(kThreads) vox_count_marked_kernel(const __grid_constant__ ScanArgs a) {
    await_predecessor();
    __shared__ uint32_t s_warp[kCountTiles][kThreads / 32], s_which[kThreads];
    const int t = threadIdx.x, words1 = a.tiles[1] / kCountTiles, words = words1 + a.tiles[0] / kCountTiles;
    const int mine = (int)blockIdx.x + t * (int)gridDim.x;
    uint32_t which = 0u;
    if (mine < words) {
        const int sc = mine < words1 ? 1 : 0, w = sc ? mine : mine - words1;
#pragma unroll
        for (uint32_t r = 0; r < kNoteCopies; ++r) which |= a.st.marked[sc][w / 8 + r * a.st.note_stride];
        which = which >> (w % 8 * 4) & 15u;
        if (!which) *reinterpret_cast<uint4*>(a.st.tile_voxels[sc] + w * kCountTiles) = make_uint4(0u, 0u, 0u, 0u);
    }
    s_which[t] = which;
    __syncthreads();
    for (int k = 0, w = (int)blockIdx.x; w < words; ++k, w += (int)gridDim.x) {
        const uint32_t these = s_which[k];
        if (!these) continue;
        const int sc = w < words1 ? 1 : 0;
        count_tiles(a, s_warp, sc, (sc ? w : w - words1) * kCountTiles, these);
        __syncthreads();                                  // s_warp is used again
    }
    release_successor();
}

// More cells over the cap, or more points in them, than a call's points allow: the store was not all zero when the
// call began.  The scale's lists are not used then; vox_finalize reports no voxels for it.
__device__ __forceinline__ void refuse_lists(const ScaleDev& g, int* status) {
    atomicOr(&g.totals[1], 1);
    atomicOr(status, kStatusDirtyStore);
}

// A part whose sectors hold few voxels each is listed by its lanes, a sector each; in any other the warp would wait for the lane
// with most, and its words are shared out.  vox_rank by events, us, by words only / by sectors up to four voxels / by sectors only:
// two frames of 33,333 uniform points 18.7 / 16.7 / 16.7, 32 KITTI-shaped frames of 4,000 points 32.0 / 28.0 / 27.2, eight of 16,384
// 20.8 / 18.8 / 18.7, of 120,000 26.4 / 25.6 / 28.5, 32 of 262,144 101 / 98.6 / 113, four nuScenes-shaped ones 28.2 / 28.3 / 30.6.  Up to
// two voxels instead of four the same, up to ten 26.8 for eight of 120,000 and 106 for 32 of 262,144.
constexpr uint32_t kFewVoxels = 4;

constexpr int kRankThreads = 256, kRankCtas = 6;
static_assert(0xFFFFFF00u / kBitmapTileCells / kTilesPerGroup < 3 * kRankThreads, "a thread has up to three groups of tiles of a scale, see validate");
static_assert(kScanSectors == 8 * 32, "a tile has eight parts, one sector for each lane of a warp");

__global__ void __launch_bounds__(kRankThreads, kRankCtas) vox_rank_kernel(const __grid_constant__ ScanArgs a) {
    await_predecessor();
    constexpr int kWarps = kRankThreads / 32;
    extern __shared__ uint32_t s_groups[];                // [groups of both scales]
    __shared__ uint32_t s_sum[2][kWarps], s_words[kWarps][6 * 32];    // words of a part that have a bit
    const uint32_t groups0 = (uint32_t)(a.tiles[0] + kTilesPerGroup - 1) / kTilesPerGroup;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t listed = *a.st.listed, step = gridDim.x * kWarps;
#pragma unroll
    for (int v = 0; v < 2; ++v)                           // vox_count has read the notes
        for (int i = blockIdx.x * kRankThreads + t; i < a.st.words[v]; i += gridDim.x * kRankThreads)
#pragma unroll
            for (uint32_t r = 0; r < kNoteCopies; ++r) a.st.marked[v][i + r * a.st.note_stride] = 0u;
    uint32_t k = (uint32_t)warp * gridDim.x + blockIdx.x, next = 0u;
    uint32_t entry = k < listed ? a.st.list[k] : 0u;
    // Voxels before every group of tiles, and of both scales.
    uint32_t all[2] = {0u, 0u};
    {
        uint32_t n[2][3], inc[2], sum[2];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
#pragma unroll
            for (int i = 0; i < 3; ++i) n[v][i] = (3 * t + i) * kTilesPerGroup < a.tiles[v] ? a.st.group_voxels[v][3 * t + i] : 0u;
        }
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            sum[v] = n[v][0] + n[v][1] + n[v][2];
            inc[v] = warp_incl_scan(sum[v]);
            if (lane == 31) s_sum[v][warp] = inc[v];
        }
        __syncthreads();
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const uint32_t own = lane < kWarps ? s_sum[v][lane] : 0u;
            all[v] = __reduce_add_sync(0xFFFFFFFFu, own);
            uint32_t run = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? own : 0u) + inc[v] - sum[v];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                if ((3 * t + i) * kTilesPerGroup < a.tiles[v]) s_groups[v * groups0 + 3 * t + i] = run;
                run += n[v][i];
            }
        }
        __syncthreads();
    }
    if (blockIdx.x == 0 && t < 2 && !a.s[t].design) {
        // More voxels than a call's points allow: the store was not all zero when the call began (two
        // calls on one handle at once).  The scale is then not ranked and reports no voxels, and the
        // handle's status becomes an internal error.
        const ScaleDev& g = a.s[t];
        const uint32_t n = t ? all[1] : all[0];
        const bool dirty = !voxels_possible(n, g.max_list);
        g.totals[0] = (int)voxels_ranked(n, g.max_list);
        a.num_voxels[t] = (int)voxels_ranked(n, g.max_list);
        if (dirty) atomicOr(a.status, kStatusDirtyStore);
        else if ((int)n > a.capacity[t]) atomicOr(a.status, kStatusCapacity);
    }
    // The listed parts, a warp each; the warps of a CTA are far apart in the list.
    for (; k < listed; k += step, entry = next) {
        if (k + step < listed) next = a.st.list[k + step];
        const int sc = (int)(entry >> 31), tile = (int)(entry >> 3 & 0x0FFFFFFFu), part = (int)(entry & 7u);
        const ScaleDev& g = a.s[sc];
        if (!voxels_possible(sc ? all[1] : all[0], g.max_list)) continue;
        const bool bitmap = g.mode == MODE_BITMAP;
        const uint32_t sector = (uint32_t)tile * kScanSectors + part * 32 + lane;
        uint4* const at = reinterpret_cast<uint4*>(g.store) + (size_t)sector * 2;
        uint4 p = at[0], q = at[1];
        // Voxels before the part: groups before its group, tiles of its group before its tile, parts of its tile before it.
        const int in_group = tile % kTilesPerGroup, k0 = 4 * lane;
        uint4 four = make_uint4(0u, 0u, 0u, 0u);
        if (k0 < in_group) four = *reinterpret_cast<const uint4*>(a.st.tile_voxels[sc] + (tile - in_group) + k0);
        uint32_t before = lane < part ? reinterpret_cast<const uint16_t*>(a.st.tile_parts[sc] + tile)[lane] : 0u;
        before += (k0 < in_group ? four.x : 0u) + (k0 + 1 < in_group ? four.y : 0u) + (k0 + 2 < in_group ? four.z : 0u) +
                  (k0 + 3 < in_group ? four.w : 0u);
        before = __reduce_add_sync(0xFFFFFFFFu, before) + s_groups[sc * groups0 + tile / kTilesPerGroup];
        const uint32_t c = sector_voxels(bitmap, p, q);
        const uint32_t inc = warp_incl_scan(c);
        uint32_t m = before + inc - c;
        if (bitmap) {
            const uint32_t w[6] = {p.x, p.y, p.z, q.x, q.y, q.z};
            if (c != 0u) {
                p.w = m;
                q.w = m + __popc(p.x) + __popc(p.y) + __popc(p.z);
                at[0] = p;
                at[1] = q;
            }
            if (__reduce_max_sync(0xFFFFFFFFu, c) <= kFewVoxels) {
                uint32_t cell = sector * (2u * kUnitCells);
#pragma unroll
                for (int i = 0; i < 6; ++i, cell += 32u) {
                    for (uint32_t bits = w[i]; bits; bits &= bits - 1u, ++m)
                        if (m < g.max_list) g.cell_list[m] = cell + (uint32_t)__ffs(bits) - 1u;
                }
                continue;
            }
            // The words with voxels side by side in shared memory, {voxels of the part before it, number, lane that has it}, then a
            // lane per word.
            uint32_t some = 0u;
#pragma unroll
            for (int i = 0; i < 6; ++i) some += w[i] != 0u;
            uint32_t to = warp_incl_scan(some), rel = inc - c;
            const uint32_t words = __shfl_sync(0xFFFFFFFFu, to, 31);
            to -= some;
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                if (w[i] == 0u) continue;
                s_words[warp][to++] = rel << 8 | i << 5 | lane;
                rel += __popc(w[i]);
            }
            __syncwarp();
            const uint32_t cell0 = (sector - lane) * (2u * kUnitCells);
            for (uint32_t i0 = 0u; i0 < words; i0 += 32u) {
                const uint32_t word = i0 + lane < words ? s_words[warp][i0 + lane] : 7u << 5;
                const uint32_t number = word >> 5 & 7u, from = word & 31u;
                uint32_t bits = 0u;
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    const uint32_t theirs = __shfl_sync(0xFFFFFFFFu, w[i], from);
                    if (number == i) bits = theirs;
                }
                const uint32_t cell = cell0 + from * (2u * kUnitCells) + number * 32u;
                for (uint32_t row = before + (word >> 8); bits; bits &= bits - 1u, ++row)
                    if (row < g.max_list) g.cell_list[row] = cell + (uint32_t)__ffs(bits) - 1u;
            }
            __syncwarp();                                 // the words are used again
            continue;
        }
        // Cells over the cap take the next places among such cells, and their points the next slots of
        // the index list, in any order: one ticket per part.
        uint32_t n[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
        uint32_t j = 0, off = 0, cells = 0, points = 0;
        bool list_over = false;
        if (g.cap > 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (n[i] > (uint32_t)g.cap) { cells += 1; points += clamp_points(n[i]); }
        }
        if (__any_sync(0xFFFFFFFFu, cells != 0)) {
            points = clamp_points(points);
            const uint32_t ic = warp_incl_scan(cells), ip = warp_incl_scan(points);
            unsigned long long first = 0;
            bool fits = false;
            if (lane == 31) {
                fits = ip <= g.max_list;
                if (fits) {
                    first = atomicAdd(reinterpret_cast<unsigned long long*>(g.totals + 2), (unsigned long long)over_ticket(ic, ip));
                    fits = over_fits(first, ic, ip, g.max_ovf, g.max_list);
                }
                if (!fits) refuse_lists(g, a.status);
            }
            list_over = __shfl_sync(0xFFFFFFFFu, fits ? 1 : 0, 31) != 0;
            j = __shfl_sync(0xFFFFFFFFu, (uint32_t)(first >> 32), 31) + ic - cells;
            off = __shfl_sync(0xFFFFFFFFu, (uint32_t)first, 31) + ip - points;
        }
        if (c != 0u) {
            const uint32_t cell = sector * 8u;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (n[i] == 0u) continue;
                const bool over = list_over && n[i] > (uint32_t)g.cap;
                if (m < (uint32_t)a.capacity[sc]) a.counts[sc][m] = over ? g.cap : (int)n[i];
                if (m < g.max_list) g.cell_list[m] = over ? (cell + i) | kOverCap : cell + i;
                if (over) {
                    g.ovf_vox[j] = (int)m; g.ovf_off[j] = (int)off; g.ovf_cell[j] = cell + i;
                    g.ovf_cursor[(size_t)j * kCursorStride] = 0;
                    off += n[i];
                    n[i] = kOverCap | j++;
                } else {
                    n[i] = m;
                }
                ++m;
            }
            at[0] = make_uint4(n[0], n[1], n[2], n[3]);
            at[1] = make_uint4(n[4], n[5], n[6], n[7]);
        }
    }
    // This CTA's share of the accumulators of the voxels cleared: a few tiles hold most of the voxels, so the clearing is
    // not tied to the tiles.  Done here, just before they are added to, it also brings
    // them into L2 (cleared after use by vox_finalize, vox_accum took 48 instead of 43 us on four nuScenes-shaped
    // frames and vox_finalize 40 instead of 37).
    const uint32_t thread = blockIdx.x * kRankThreads + t, threads = gridDim.x * kRankThreads;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        const ScaleDev& g = a.s[v];
        const uint32_t voxels = voxels_ranked(all[v], g.max_list);
        for (size_t i = thread; i < (size_t)voxels * g.acc_f4; i += threads) g.acc[i] = zero;
        if (counts_in_output(g))
            for (uint32_t i = thread; i < min(voxels, (uint32_t)a.capacity[v]); i += threads) a.counts[v][i] = 0;
    }
    release_successor();
}

// ------------------------------------------------------------------ pass 3: accumulate
struct AccumArgs {
    ScaleDev s[2];
    int capacity[2];            // at most max_list
    int32_t* coords[2];
    int32_t* counts[2];
    int32_t* point_voxel[2];
    float* mean[2];
    float* bev;
    uint32_t frames;            // B
    int32_t* num_voxels;
    int* status;
};

// Per-voxel accumulator, 32 bytes of fp32: {sum dx, sum dy, sum dz, sum ch3}, {sum ch4, count, -, -},
// where d* are offsets from the cell's lower corner, so that those sums stay small.  Two vector
// reductions per point and scale; a table store's voxels have their counts already, so there the second
// one only adds ch4, and with four channels there is neither a second reduction nor a second half.  A bitmap scale with four
// channels and no cap counts its points in the caller's array instead of a second half: as many reductions, but 20 bytes
// per voxel to clear, add to and read where it were 32 and the counts besides (32 frames of 262,144 points: vox_rank 125 ->
// 117 us, vox_accum 175 -> 159, vox_finalize 147 -> 140, the call 1,793 -> 1,761).  A sum of n terms carries a relative error of at most n * 2^-24
// (far less in practice, since the roundings do not line up).
// Every thread loads its own point: staged in shared memory first, as five floats or four, the points cost a barrier
// before the look-ups (eight KITTI-shaped frames 25.2 -> 24.4 us, four nuScenes-shaped ones 43.4 -> 41.0; the marking pass
// of the latter 28.5 -> 27.1).  What remains is the rate of scattered L2 requests: two look-ups and three or four
// reductions per point.
template <int C>
__global__ void __launch_bounds__(kThreads)
vox_accum_kernel(const float* __restrict__ pts, long long total, int N, const __grid_constant__ AccumArgs a) {
    await_predecessor();
    const long long g = (long long)blockIdx.x * kThreads + threadIdx.x;
    if (g >= total) return;
    float f[C];
    if (C == 4) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(pts) + g);
        f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
    } else {
#pragma unroll
        for (int k = 0; k < C; ++k) f[k] = __ldg(pts + g * C + k);
    }
    const int b = (int)((uint32_t)g / (uint32_t)N);       // at most 2^24 points
    // Both look-ups first, so that the thread has its loads in flight together.
    Slot slot[2];
    int c[2][3];
#pragma unroll
    for (int sc = 0; sc < 2; ++sc) {
        const ScaleDev& s = a.s[sc];
        uint32_t cell = 0xFFFFFFFFu;
        if (cell_xyz(s, f[0], f[1], f[2], c[sc][0], c[sc][1], c[sc][2]))
            cell = (((uint32_t)b * s.dims[2] + c[sc][2]) * s.dims[1] + c[sc][1]) * s.dims[0] + c[sc][0];
        slot[sc] = slot_of(s, cell, g);
    }
#pragma unroll
    for (int sc = 0; sc < 2; ++sc) {
        const ScaleDev& s = a.s[sc];
        int32_t* pv = a.point_voxel[sc];
        const Slot at = slot[sc];
        if (at.j >= 0) {
            // Which of this cell's points survive the cap is decided per cell in
            // vox_finalize_kernel, which also writes their point_voxel entries.
            if ((uint32_t)at.j < s.max_ovf) {         // always, unless the store was dirty
                const int tk = atomicAdd(&s.ovf_cursor[(size_t)at.j * kCursorStride], 1);
                const uint32_t pos = (uint32_t)(s.ovf_off[at.j] + tk);
                if (pos < s.max_list) s.ovf_list[pos] = (int)g;
            }
            continue;
        }
        if (pv) pv[g] = at.m;
        if (at.m < 0 || at.m >= a.capacity[sc]) continue;
        const float dx = __fsub_rn(f[0], cell_corner(s.mn[0], s.vs[0], c[sc][0]));
        const float dy = __fsub_rn(f[1], cell_corner(s.mn[1], s.vs[1], c[sc][1]));
        const float dz = __fsub_rn(f[2], cell_corner(s.mn[2], s.vs[2], c[sc][2]));
        float4* row = s.acc + (size_t)at.m * s.acc_f4;
        atomicAdd(row, make_float4(dx, dy, dz, f[3]));
        // A scale that was not ranked reports no voxels, whatever its store holds, and the caller's counts stay as they were.  The
        // total is read here and not with the look-ups, where it cost eight KITTI-shaped frames 22.4 -> 23.2 us (here 22.5).
        if (counts_in_output(s)) { if (at.m < s.totals[0]) atomicAdd(a.counts[sc] + at.m, 1); }
        else if (s.mode == MODE_BITMAP) atomicAdd(reinterpret_cast<float2*>(row + 1), make_float2(C > 4 ? f[C - 1] : 0.0f, 1.0f));
        else if (C > 4) atomicAdd(reinterpret_cast<float*>(row + 1), f[C - 1]);
    }
    release_successor();
}

// ------------------------------------------------------------------ per-voxel cap on a bitmap scale
// A bitmap store keeps no per-cell point count, so a voxel over its cap is only known once the points
// are accumulated.  Two small passes then build what the table path gets from the rank scan:
//   vox_over_find   a thread per voxel row: count > cap -> the voxel takes the next place j among the
//                   over-cap voxels and the next `count` slots of the index list (warp-aggregated
//                   tickets), and remembers j + 1 in the spare word of its accumulator;
//   vox_over_fill   a thread per point: if its voxel is over the cap, the point's index goes into the
//                   voxel's list.
// vox_finalize then keeps the `cap` lowest indices of every list exactly as for a table scale.
__global__ void __launch_bounds__(kThreads) vox_over_find_kernel(AccumArgs a, int sc) {
    await_predecessor();
    const ScaleDev& g = a.s[sc];
    const int lane = threadIdx.x & 31;
    const int M = min(g.totals[0], a.capacity[sc]);
    for (int m0 = (blockIdx.x * kThreads + threadIdx.x) & ~31; m0 < M; m0 += gridDim.x * kThreads) {
        const int m = m0 + lane;
        const int n = m < M ? (int)g.acc[2 * (size_t)m + 1].y : 0;
        const bool over = n > g.cap;
        const unsigned who = __ballot_sync(0xFFFFFFFFu, over);
        if (!who) continue;
        int inc = over ? n : 0;                   // inclusive scan of the over-cap counts
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        int j0 = 0, off0 = 0;
        if (lane == 31) {                         // sums of at most 32 counts of at most 2^24
            const uint32_t cells = (uint32_t)__popc(who), points = (uint32_t)inc;
            unsigned long long at = 0;
            bool fits = points <= g.max_list;
            if (fits) {
                at = atomicAdd(reinterpret_cast<unsigned long long*>(g.totals + 2), (unsigned long long)over_ticket(cells, points));
                fits = over_fits(at, cells, points, g.max_ovf, g.max_list);
            }
            if (!fits) refuse_lists(g, a.status);     // never with this batch's own counts
            j0 = fits ? (int)(at >> 32) : -1; off0 = (int)(uint32_t)at;
        }
        j0 = __shfl_sync(0xFFFFFFFFu, j0, 31);
        off0 = __shfl_sync(0xFFFFFFFFu, off0, 31);
        if (!over || j0 < 0) continue;
        const int j = j0 + __popc(who & ((1u << lane) - 1u));
        const int off = off0 + inc - n;
        g.ovf_vox[j] = m; g.ovf_off[j] = off; g.ovf_cell[j] = g.cell_list[m];
        g.ovf_cursor[(size_t)j * kCursorStride] = 0;
        reinterpret_cast<uint32_t*>(g.acc + 2 * (size_t)m + 1)[2] = (uint32_t)j + 1u;
    }
    release_successor();
}

template <int C>
__global__ void __launch_bounds__(kThreads)
vox_over_fill_kernel(const float* __restrict__ pts, long long total, int N, AccumArgs a, int sc) {
    await_predecessor();
    const ScaleDev& g = a.s[sc];
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < total; i += (long long)gridDim.x * kThreads) {
        const float* p = pts + i * C;
        const Slot s = slot_of(g, cell_of(g, p[0], p[1], p[2], (int)(i / N)), i);
        if (s.m < 0 || s.m >= a.capacity[sc]) continue;
        const uint32_t tag = reinterpret_cast<const uint32_t*>(g.acc + 2 * (size_t)s.m + 1)[2];
        if (tag == 0u || tag > g.max_ovf) continue;
        const int j = (int)tag - 1;
        const int tk = atomicAdd(&g.ovf_cursor[(size_t)j * kCursorStride], 1);
        const uint32_t pos = (uint32_t)(g.ovf_off[j] + tk);
        if (pos < g.max_list) g.ovf_list[pos] = (int)i;
    }
    release_successor();
}

// ------------------------------------------------------------------ pass 4: rows, BEV, cleanup
// What the output rows of n <= 32 voxels with consecutive rows mb, mb+1, ... are made from, as loaded: lane i holds the cell-list
// entry of row mb + i, and of the accumulators either row mb + i or, where they have two halves, float4 i and i + 32.
struct VoxelBatch {
    uint32_t entry;
    int count;
    float4 lo, hi;
};

__device__ __forceinline__ VoxelBatch load_batch(const AccumArgs& a, int v, int nb0, int tot0, int tot1) {
    const int lane = threadIdx.x & 31, sc = v >= nb0 ? 1 : 0;
    const int mb = (sc ? v - nb0 : v) << 5, n = min(32, (sc ? tot1 : tot0) - mb), rows = min(n, a.capacity[sc] - mb);
    const ScaleDev& g = a.s[sc];
    VoxelBatch b;
    b.entry = lane < n ? g.cell_list[mb + lane] : 0u;
    b.count = 1;
    b.lo = b.hi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (g.acc_f4 == 2) {
        const float4* src = g.acc + 2 * (size_t)mb;
        if (lane < 2 * rows) b.lo = __ldcg(src + lane);
        if (lane + 32 < 2 * rows) b.hi = __ldcg(src + lane + 32);
    } else if (lane < rows) {
        b.lo = __ldcg(g.acc + mb + lane);
    }
    if ((g.mode == MODE_TABLE || g.acc_f4 == 1) && lane < rows) b.count = a.counts[sc][mb + lane];   // by the rank scan or the accumulation
    return b;
}

// Writes the output rows of a batch; `stage` is 1 KB of the warp's own shared memory.  Accumulators are read and mean rows written as
// contiguous blocks through shared memory, so the warp issues full-sector requests only.
template <int C>
__device__ __forceinline__ void write_batch(const AccumArgs& a, int sc, int mb, int n, const VoxelBatch& b, float4* stage) {
    const ScaleDev& g = a.s[sc];
    const int lane = threadIdx.x & 31;
    n = min(n, a.capacity[sc] - mb);              // rows past the caller's capacity are not written
    if (n <= 0) return;
    const bool active = lane < n;
    const bool table = g.mode == MODE_TABLE, counted = table || counts_in_output(g);
    const uint32_t entry = b.entry;
    int cnt = b.count;
    float4 a0 = b.lo, a1 = b.hi;
    if (g.acc_f4 == 2) {
        stage[lane] = a0;
        stage[lane + 32] = a1;
        __syncwarp();
        a0 = stage[2 * lane]; a1 = stage[2 * lane + 1];
        __syncwarp();
    }
    const uint32_t cell = table ? (entry & ~kOverCap) : entry;
    // Over the cap: a table store flags the cell in its list entry; a bitmap store has no per-cell count,
    // there vox_over_find_kernel left the voxel's place among the over-cap voxels (+ 1) in a spare word.
    const bool over = active && (table ? (entry & kOverCap) != 0u : __float_as_uint(a1.z) != 0u);   // a1 0: no such voxels
    uint32_t r = cell, x, y, z;
    g.div[0].divmod(r, r, x);
    g.div[1].divmod(r, r, y);
    g.div[2].divmod(r, r, z);
    if (!counted) cnt = over ? g.cap : (int)a1.y;
    if (!table && active && cnt == 0) atomicOr(a.status, kStatusDirtyStore);     // no point of this call marked the cell
    // Offsets are below one cell size, so fp32 keeps the mean to a few 1e-7 of that size.
    const float inv = __frcp_rn((float)cnt);
    float mu[C];
    mu[0] = __fadd_rn(cell_corner(g.mn[0], g.vs[0], (int)x), a0.x * inv);
    mu[1] = __fadd_rn(cell_corner(g.mn[1], g.vs[1], (int)y), a0.y * inv);
    mu[2] = __fadd_rn(cell_corner(g.mn[2], g.vs[2], (int)z), a0.z * inv);
    mu[3] = __fdiv_rn(a0.w, (float)cnt);
    if (C > 4) mu[4] = __fdiv_rn(a1.x, (float)cnt);
    if (active) {
        reinterpret_cast<int4*>(a.coords[sc])[mb + lane] = make_int4((int)r, (int)z, (int)y, (int)x);
        if (!counted) a.counts[sc][mb + lane] = cnt;
    }
    // Mean rows: the n * C floats of rows mb .. mb+n-1 are contiguous.  The row of a cell over the
    // cap is written by that cell's own warp, so a batch holding one writes its rows one by one.
    float* rows = a.mean[sc] + (size_t)mb * C;
    if (!__any_sync(0xFFFFFFFFu, over)) {
        float* st = reinterpret_cast<float*>(stage);
#pragma unroll
        for (int k = 0; k < C; ++k) st[lane * C + k] = mu[k];
        __syncwarp();
        for (int i = lane; i < n * C; i += 32) rows[i] = st[i];
        __syncwarp();
    } else if (active && !over) {
#pragma unroll
        for (int k = 0; k < C; ++k) rows[lane * C + k] = mu[k];
    }
    if (sc == 1 && a.bev && active && !over && frame_in_call(r, a.frames)) {
        const size_t plane = (size_t)g.dims[1] * g.dims[0];
        float* dst = a.bev + (size_t)r * C * plane + (size_t)y * g.dims[0] + x;
#pragma unroll
        for (int k = 0; k < C; ++k) dst[(size_t)k * plane] = mu[k];
    }
}

// CTAs [0, ovf_blocks) serve cells over the cap, one warp per cell: the `cap` lowest point
// indices are kept (keep-first-by-index), summed in fp64 and written as the voxel's mean; all of
// the cell's points get their point_voxel entry.  The other CTAs write the voxel rows.  Six CTAs per SM, 40
// registers: with 47, five, four nuScenes-shaped frames took 39.4 instead of 37.8 us.
// A warp takes some twenty steps to bisect a cell's indices, each of which waited for the list to come from L2 again: it
// keeps the first 256 of them in registers (the densest cells of the dense frame have about 300).  One dense frame: the
// kernel 19.0 -> 12.7 us, the call 76.3 -> 70.5; four nuScenes-shaped frames: the kernel 38.0 -> 34.9.
constexpr int kHeld = 8;

template <int C>
__global__ void __launch_bounds__(kThreads, 6)
vox_finalize_kernel(const float* __restrict__ pts, long long total, AccumArgs a, int ovf_blocks) {
    await_predecessor();
    constexpr int kWarps = kThreads / 32;
    const int lane = threadIdx.x & 31;
    if ((int)blockIdx.x < ovf_blocks) {
        const int warp = (blockIdx.x * kThreads + threadIdx.x) >> 5;
        const int nwarps = ovf_blocks * kWarps;
        for (int sc = 0; sc < 2; ++sc) {
            const ScaleDev& g = a.s[sc];
            if (g.cap <= 0) continue;
            const int4 tot = *reinterpret_cast<const int4*>(g.totals);
            if (tot.y != 0 && warp == 0 && lane == 0) a.num_voxels[sc] = 0;   // see refuse_lists
            const int novf = tot.x == 0 || tot.y != 0 ? 0 : min(tot.w, (int)g.max_ovf);
            int32_t* pv = a.point_voxel[sc];
            for (int j = warp; j < novf; j += nwarps) {
                const int m = g.ovf_vox[j];
                const uint32_t start = (uint32_t)g.ovf_off[j];
                const int* list = g.ovf_list + start;
                const int n = start < g.max_list ? min(g.ovf_cursor[(size_t)j * kCursorStride], (int)(g.max_list - start)) : 0;
                // Smallest index value v with #{list <= v} >= cap, by bisection on the value, between the smallest
                // and the largest of the list.
                int held[kHeld];
                int lo = 0x7FFFFFFF, hi = -1;
#pragma unroll
                for (int u = 0; u < kHeld; ++u) {
                    held[u] = 32 * u + lane < n ? list[32 * u + lane] : 0x7FFFFFFF;
                    if (32 * u + lane < n) { lo = min(lo, held[u]); hi = max(hi, held[u]); }
                }
                for (int i = 32 * kHeld + lane; i < n; i += 32) { lo = min(lo, list[i]); hi = max(hi, list[i]); }
                lo = __reduce_min_sync(0xFFFFFFFFu, lo) - 1;
                hi = __reduce_max_sync(0xFFFFFFFFu, hi);
                while (hi - lo > 1) {
                    const int mid = lo + (hi - lo) / 2;
                    int c = 0;
#pragma unroll
                    for (int u = 0; u < kHeld; ++u) c += held[u] <= mid;
                    for (int i = 32 * kHeld + lane; i < n; i += 32) c += list[i] <= mid;
                    c = warp_sum(c);
                    if (c >= g.cap) hi = mid; else lo = mid;
                }
                double acc[C];
#pragma unroll
                for (int k = 0; k < C; ++k) acc[k] = 0.0;
                for (int i = lane; i < n; i += 32) {
                    const int v = list[i];
                    const bool mine = (unsigned)v < (unsigned)total;      // always, with this call's own lists
                    const bool keep = mine && v <= hi;
                    if (pv && mine) pv[v] = keep ? m : -1;
                    if (keep) {
#pragma unroll
                        for (int k = 0; k < C; ++k) acc[k] += (double)pts[(size_t)v * C + k];
                    }
                }
#pragma unroll
                for (int k = 0; k < C; ++k) {
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) acc[k] += __shfl_xor_sync(0xFFFFFFFFu, acc[k], d);
                }
                if (lane < C && (unsigned)m < (unsigned)a.capacity[sc]) {
                    double v = 0.0;
#pragma unroll
                    for (int k = 0; k < C; ++k) v = lane == k ? acc[k] : v;
                    const float mu = (float)(v / (double)g.cap);
                    a.mean[sc][(size_t)m * C + lane] = mu;
                    if (sc == 1 && a.bev) {
                        uint32_t r = g.ovf_cell[j], x, y;
                        g.div[0].divmod(r, r, x);
                        g.div[1].divmod(r, r, y);
                        const size_t plane = (size_t)g.dims[1] * g.dims[0];
                        if (frame_in_call(r, a.frames)) a.bev[((size_t)r * C + lane) * plane + (size_t)y * g.dims[0] + x] = mu;
                    }
                }
            }
        }
        return;
    }
    // Voxel rows: a warp takes 32 consecutive rows of one scale at a time, reads their cell ids
    // from the list the rank scan wrote, writes the rows and puts the cells' store sectors back to
    // zero (whole 32-byte sectors: a partial write would first fetch the sector), once per run of voxels.
    // Every warp has its own batch, so the batches' memory latencies overlap, and a batch's loads are all requested before the
    // store of its sectors, which depends on one of them (32 frames of 262,144 points 140 -> 128 us, four nuScenes-shaped frames 33.7 ->
    // 32.8; with the next batch requested ahead at five or four CTAs per SM 126 and 32.9, the calls no faster).
    __shared__ float4 s_stage[kWarps][64];
    float4* stage = s_stage[threadIdx.x >> 5];
    const int tot0 = a.s[0].totals[0], tot1 = a.s[1].totals[0];
    const int nb0 = (tot0 + 31) >> 5, nb1 = (tot1 + 31) >> 5;
    const int nwarps = ((int)gridDim.x - ovf_blocks) * kWarps, batches = nb0 + nb1;
    int v = ((int)blockIdx.x - ovf_blocks) * kWarps + (threadIdx.x >> 5);
    for (; v < batches; v += nwarps) {
        const VoxelBatch b = load_batch(a, v, nb0, tot0, tot1);
        const int sc = v >= nb0 ? 1 : 0;
        const int mb = (sc ? v - nb0 : v) << 5;
        const ScaleDev& g = a.s[sc];
        const int n = min(32, (sc ? tot1 : tot0) - mb);
        const uint32_t sector = g.mode == MODE_BITMAP ? b.entry / (2u * kUnitCells) : (b.entry & ~kOverCap) >> 3;
        const uint32_t before = __shfl_up_sync(0xFFFFFFFFu, sector, 1);
        if (lane < n && !g.design && (lane == 0 || before != sector)) {
            uint4* sp = reinterpret_cast<uint4*>(g.store + 8 * (size_t)sector);
            sp[0] = make_uint4(0u, 0u, 0u, 0u);
            sp[1] = make_uint4(0u, 0u, 0u, 0u);
        }
        write_batch<C>(a, sc, mb, n, b, stage);
    }
    release_successor();
}

template <int C>
int run_voxelize(emc2_bridge* h, int B, int N, const float* d_points, int32_t* const d_coords[2],
                 int32_t* const d_counts[2], float* const d_mean[2], int32_t* const d_point_voxel[2],
                 const int32_t capacity[2], int32_t* d_num_voxels, float* d_bev, cudaStream_t st, bool marked, bool chained) {
    const long long total = (long long)B * N;
    const int ptiles = (int)((total + kThreads - 1) / kThreads);   // one point per thread (two measured 1 - 3 % slower per step)
    ScanArgs sa;
    AccumArgs aa;
    bool any_cap = false;
    for (int s = 0; s < 2; ++s) {
        sa.s[s] = h->scale[s];
        // A scale deduplicated by the hash or sort design has no store to scan; its voxel list is a plain
        // list of cell ids, which the later passes treat like a bitmap scale's.
        if (sa.s[s].design) sa.s[s].mode = MODE_BITMAP;
        aa.s[s] = sa.s[s];
        const uint64_t cells = sa.s[s].design ? 0 : (uint64_t)B * h->scale[s].cells;
        const uint64_t per_tile = sa.s[s].mode == MODE_BITMAP ? kBitmapTileCells : kTableTileCells;
        sa.tiles[s] = (int)((cells + per_tile - 1) / per_tile + kCountTiles - 1) / kCountTiles * kCountTiles;
        sa.capacity[s] = capacity[s];
        sa.counts[s] = d_counts[s];
        aa.capacity[s] = (int)min((long long)capacity[s], (long long)h->scale[s].max_list);
        aa.coords[s] = d_coords[s];
        aa.counts[s] = d_counts[s];
        aa.mean[s] = d_mean[s];
        aa.point_voxel[s] = d_point_voxel ? d_point_voxel[s] : nullptr;
        any_cap = any_cap || h->scale[s].cap > 0;
    }
    sa.num_voxels = d_num_voxels;
    sa.status = h->d_status;
    sa.st = h->scan;
    for (int s = 0; s < 2; ++s) sa.st.words[s] = keeps_tile_marks(h, B, N) ? (sa.tiles[s] + 31) / 32 : 0;
    aa.bev = d_bev;
    aa.frames = (uint32_t)B;
    aa.num_voxels = d_num_voxels;
    aa.status = h->d_status;

    const size_t bev_n = d_bev ? (size_t)B * C * h->scale[1].dims[1] * h->scale[1].dims[0] : 0;
    const bool bev_vec = bev_by_kernel(bev_n);
    if (!marked && bev_n && !bev_vec) cudaMemsetAsync(d_bev, 0, bev_n * sizeof(float), st);
    if (!marked) {
        // Also zeroes the BEV image; with no points it still runs for that.
        const int zeroing = bev_n && bev_vec ? (h->num_sms + B - 1) / B : 0;
        const FastDiv group = make_fast_div((uint32_t)frames_per_group(store_bytes(h), B));
        const dim3 grid = marking_grid(max((N + kTile - 1) / kTile, zeroing), B, group);
        if (B > 0 && grid.x > 0) {
            LaunchScope ls(h, K_VOX_MARK, st);
            vox_mark_kernel<C><<<grid, kThreads, 0, st>>>(d_points, B, N, group, sa.s[0], sa.s[1],
                                                          bev_vec ? reinterpret_cast<float4*>(d_bev) : nullptr,
                                                          bev_vec ? (uint32_t)(bev_n >> 2) : 0u, scan_reset(h), tile_marks(h, B, N));
        }
    }
    for (int s = 0; s < 2; ++s) {
        if (!h->scale[s].design) continue;
        const int rc = launch_dedup_arm(h, s, h->scale[s].design, B, N, d_points, capacity[s], d_num_voxels, st);
        if (rc != EMC2_OK) return rc;
    }
    if (total == 0) return check_cuda(h, cudaMemsetAsync(d_num_voxels, 0, 2 * sizeof(int32_t), st));   // no points: no voxels
    const int tiles = sa.tiles[0] + sa.tiles[1];
    if (tiles > 0) {
        {
            LaunchScope ls(h, K_VOX_COUNT, st);
            // In the one-call path its predecessor can be on another stream.
            if (keeps_tile_marks(h, B, N))
                launch_kernel(!marked || chained, vox_count_marked_kernel, min(tiles / kCountTiles, 8 * h->num_sms), kThreads, 0, st, sa);
            else
                launch_kernel(!marked || chained, vox_count_kernel, tiles / kCountTiles, kThreads, 0, st, sa);
        }
        LaunchScope ls(h, K_VOX_RANK, st);
        const int groups = (sa.tiles[0] + kTilesPerGroup - 1) / kTilesPerGroup + (sa.tiles[1] + kTilesPerGroup - 1) / kTilesPerGroup;
        launch_chained(vox_rank_kernel, min(tiles, kRankCtas * h->num_sms), kRankThreads, groups * sizeof(uint32_t), st, sa);
    }
    if (total > 0) {
        LaunchScope ls(h, K_VOX_ACCUM, st);
        launch_chained(vox_accum_kernel<C>, ptiles, kThreads, 0, st, d_points, total, N, aa);
    }
    for (int s = 0; s < 2 && total > 0; ++s) {
        if (aa.s[s].mode != MODE_BITMAP || h->scale[s].cap <= 0) continue;
        {
            LaunchScope ls(h, K_VOX_OVER_FIND, st);
            launch_chained(vox_over_find_kernel, 4 * h->num_sms, kThreads, 0, st, aa, s);
        }
        {
            LaunchScope ls(h, K_VOX_OVER_FILL, st);
            launch_chained(vox_over_fill_kernel<C>, (int)min((long long)8 * h->num_sms, (total + kThreads - 1) / kThreads), kThreads, 0, st, 
                d_points, total, N, aa, s);
        }
    }
    if (total > 0) {
        // The number of voxels is only known on the device: a fixed grid strides over them.
        const int ovf_blocks = any_cap ? 2 * h->num_sms : 0;    // CTAs that serve cells over the cap
        const int vox_blocks = (int)min((long long)h->num_sms * 8, (2 * total + 32 * 8 - 1) / (32 * 8) + 1);
        LaunchScope ls(h, K_VOX_FINALIZE, st);
        launch_chained(vox_finalize_kernel<C>, ovf_blocks + vox_blocks, kThreads, 0, st, d_points, total, aa, ovf_blocks);
    }
    return check_cuda(h, cudaGetLastError());
}

}  // namespace

int launch_voxelize(emc2_bridge* h, int B, int N, const float* d_points, int32_t* const d_coords[2],
                    int32_t* const d_counts[2], float* const d_mean[2], int32_t* const d_point_voxel[2],
                    const int32_t capacity[2], int32_t* d_num_voxels, float* d_bev, cudaStream_t st, bool marked, bool chained) {
    if (h->cfg.point_floats == 4)
        return run_voxelize<4>(h, B, N, d_points, d_coords, d_counts, d_mean, d_point_voxel, capacity,
                               d_num_voxels, d_bev, st, marked, chained);
    return run_voxelize<5>(h, B, N, d_points, d_coords, d_counts, d_mean, d_point_voxel, capacity,
                           d_num_voxels, d_bev, st, marked, chained);
}

}  // namespace emc2
