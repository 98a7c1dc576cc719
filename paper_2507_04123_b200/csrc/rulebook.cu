// Rulebook of a 3 x 3 x 3 submanifold sparse convolution over a voxel list: the index structure of
// the 3D sparse convolution that consumes the voxel lists (Sec. 3.5), built with prefix sums in
// place of an index search (Sec. 3.6).  For kernel offset k = (dz+1)*9 + (dy+1)*3 + (dx+1) the rule
// list holds the pairs (in = n, out = m) with coords[n] = coords[m] + (dz, dy, dx) in the same
// frame, in ascending m.
//
// A neighbour is found in O(1): the scale's direct-addressed cell store (all zero between calls)
// is filled from the list, {96 cell bits, row of the unit's first voxel} per 96 cells for large
// grids, the row + 1 per cell for small ones.  Because the list is in cell order, a voxel's row is
// the unit's first row plus the number of set bits below it.
//   rb_mark   every voxel sets its cell; the first voxel of a unit stores its row there
//   rb_count  13 neighbours per voxel -> neighbour bits per voxel, pair counts per (offset, tile)
//   rb_scan   one CTA per offset: exclusive prefix sum of its counts over the tiles, and its total
//   rb_fill   offsets[28] from the totals; every tile ranks its pairs per offset with warp ballots
//             and writes them
// Only the 13 offsets k < 13, whose neighbour comes before the voxel in the list, are looked up.  The
// neighbour at offset 26 - k is the opposite one, and adding a fixed step of cells keeps the order of the
// list, so the pairs of offset 26 - k are those of offset k in the same order with in and out exchanged;
// offset 13 pairs every row with itself (in a list that is not one of the grid also rows outside it; the status
// says so).  The three x-neighbours of a (dz, dy) have consecutive rows: one
// look-up gives the first, and the neighbour at dx = -1 in the voxel's own row is the voxel before it.
// Both passes are bound by instruction issue: with 27 look-ups each they took 28 and 62 us for 894 k voxels
// with 4.8 M pairs (B200).
//   rb_clear  the touched units of the store go back to zero
#include "bridge_internal.cuh"

namespace emc2 {
namespace {

constexpr int kStatusCapacity = 1;
constexpr int kStatusBadList = 4;
constexpr int kOffsets = 27, kHalf = 13;
constexpr int kRbScanThreads = 1024;

struct RbArgs {
    ScaleDev g;
    const int4* coords;          // [capacity] rows (b, z, y, x)
    const int32_t* num_voxels;   // device: voxels in the list
    int capacity, max_batch;
    int tiles;                   // ceil(capacity / kTile)
    uint32_t* nbr_bits;          // [capacity] bit k: the neighbour at offset k exists
    int* tile_counts;            // [13][tiles]
    int* tile_base;              // [13][tiles] exclusive prefix sum of tile_counts along the tiles
    int* offset_pairs;           // [13] pairs per offset
    int32_t* offsets;            // [28]
    int32_t* rule_in;
    int32_t* rule_out;
    long long pair_capacity;
    int* status;
};

__device__ __forceinline__ int voxels_in_list(const RbArgs& a) { return min(*a.num_voxels, a.capacity); }

// Cell id of (b, z, y, x) inside the batch, 0xFFFFFFFF outside the grid.
__device__ __forceinline__ uint32_t cell_at(const RbArgs& a, int b, int z, int y, int x) {
    const ScaleDev& g = a.g;
    if ((unsigned)b >= (unsigned)a.max_batch || (unsigned)z >= (unsigned)g.dims[2] ||
        (unsigned)y >= (unsigned)g.dims[1] || (unsigned)x >= (unsigned)g.dims[0])
        return 0xFFFFFFFFu;
    return (((uint32_t)b * g.dims[2] + z) * g.dims[1] + y) * g.dims[0] + x;
}

__global__ void __launch_bounds__(kThreads) rb_mark_kernel(const __grid_constant__ RbArgs a) {
    const int M = voxels_in_list(a);
    const int m = blockIdx.x * kThreads + threadIdx.x;
    if (m >= M) return;
    const int4 c = a.coords[m];
    const uint32_t cell = cell_at(a, c.x, c.y, c.z, c.w);
    uint32_t before = 0xFFFFFFFFu;
    if (m > 0) {
        const int4 p = a.coords[m - 1];
        before = cell_at(a, p.x, p.y, p.z, p.w);
    }
    // Rows outside the grid, repeated or not in ascending cell order: not a list of this grid.
    if (cell == 0xFFFFFFFFu || (m > 0 && (before == 0xFFFFFFFFu || before >= cell))) {
        atomicOr(a.status, kStatusBadList);
        if (cell == 0xFFFFFFFFu) return;
    }
    if (a.g.mode == MODE_BITMAP) {
        uint32_t pos;
        const uint32_t u = unit_of(cell, pos);
        uint32_t* unit = a.g.store + 4 * (size_t)u;
        atomicOr(unit + (pos >> 5), 1u << (pos & 31u));
        if (m == 0 || before == 0xFFFFFFFFu || before / kUnitCells != u) unit[3] = (uint32_t)m;
    } else {
        a.g.store[cell] = (uint32_t)m + 1u;
    }
    release_successor();
}

__global__ void __launch_bounds__(kThreads) rb_clear_kernel(const __grid_constant__ RbArgs a) {
    await_predecessor();
    const int M = voxels_in_list(a);
    const int m = blockIdx.x * kThreads + threadIdx.x;
    if (m >= M) return;
    const int4 c = a.coords[m];
    const uint32_t cell = cell_at(a, c.x, c.y, c.z, c.w);
    if (cell == 0xFFFFFFFFu) return;
    if (a.g.mode == MODE_BITMAP) reinterpret_cast<uint4*>(a.g.store)[cell / kUnitCells] = make_uint4(0u, 0u, 0u, 0u);
    else a.g.store[cell] = 0u;
    release_successor();
}

// Where a voxel sits: its cell, the cell strides and which of its 3 x 3 x 3 neighbours the grid has.
struct Site {
    uint32_t cell, sy, sz;
    bool okz[3], oky[3], okx[3];
};

__device__ __forceinline__ Site site_of(const RbArgs& a, const int4 c) {
    const ScaleDev& g = a.g;
    Site s;
    s.cell = cell_at(a, c.x, c.y, c.z, c.w);
    s.sy = (uint32_t)g.dims[0];
    s.sz = s.sy * (uint32_t)g.dims[1];
    s.okz[0] = c.y > 0; s.okz[1] = true; s.okz[2] = c.y + 1 < g.dims[2];
    s.oky[0] = c.z > 0; s.oky[1] = true; s.oky[2] = c.z + 1 < g.dims[1];
    s.okx[0] = c.w > 0; s.okx[1] = true; s.okx[2] = c.w + 1 < g.dims[0];
    return s;
}

// Row of the first of the x-neighbours `three` (bit dx + 1, at least one) at (dz, dy) = (j / 3 - 1, j % 3 - 1).
__device__ __forceinline__ int first_row(const ScaleDev& g, const Site& s, int j, uint32_t three) {
    const int dz = j / 3 - 1, dy = j % 3 - 1;
    const uint32_t mid = s.cell + (uint32_t)dz * s.sz + (uint32_t)dy * s.sy;   // wraps like the signed sum
    if (g.mode == MODE_TABLE) return (int)g.store[mid + (uint32_t)__ffs(three) - 2u] - 1;
    const uint4* units = reinterpret_cast<const uint4*>(g.store);
    // Look-up at the first neighbour's own unit: a unit without voxels has no rank.
    uint32_t pos;
    const uint32_t u = unit_of(mid + (uint32_t)__ffs(three) - 2u, pos);
    const uint4 q = units[u];
    return (int)(q.w + bits_below(q, pos));
}

// Which of the three x-neighbours at (dz, dy) exist (bit dx + 1), for a valid site.
__device__ __forceinline__ uint32_t exist3(const ScaleDev& g, const Site& s, int j) {
    const int dz = j / 3 - 1, dy = j % 3 - 1;
    if (!s.okz[dz + 1] || !s.oky[dy + 1]) return 0u;
    const uint32_t mid = s.cell + (uint32_t)dz * s.sz + (uint32_t)dy * s.sy;
    const uint32_t inside = (s.okx[0] ? 1u : 0u) | 2u | (s.okx[2] ? 4u : 0u);
    if (g.mode == MODE_BITMAP) {
        const uint4* units = reinterpret_cast<const uint4*>(g.store);
        uint32_t pos;
        const uint32_t u = unit_of(mid, pos);
        const uint4 q = units[u];
        uint32_t three;                            // bits pos - 1, pos, pos + 1
        if (pos == 0) three = (q.x & 3u) << 1 | (s.okx[0] ? units[u - 1].z >> 31 : 0u);
        else if (pos == kUnitCells - 1) three = (q.z >> 30) | (s.okx[2] ? (units[u + 1].x & 1u) << 2 : 0u);
        else if (pos <= 32u) three = __funnelshift_r(q.x, q.y, pos - 1);
        else if (pos <= 64u) three = __funnelshift_r(q.y, q.z, pos - 33);
        else three = q.z >> (pos - 65);
        return three & inside;
    }
    uint32_t three = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if (s.okx[i] && g.store[mid + i - 1]) three |= 1u << i;
    return three;
}

__global__ void __launch_bounds__(kThreads) rb_count_kernel(const __grid_constant__ RbArgs a) {
    await_predecessor();
    __shared__ int wcount[kThreads / 32][kHalf];
    const int M = voxels_in_list(a);
    if ((int)blockIdx.x * kTile >= M) return;                // nothing reads the counts of tiles past the list
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int m = blockIdx.x * kTile + t;
    uint32_t bits = 0;
    if (m < M) {
        const int4 c = a.coords[m], p = a.coords[max(m - 1, 0)];
        const Site s = site_of(a, c);
        if (s.cell != 0xFFFFFFFFu) {
#pragma unroll
            for (int j = 0; j < 4; ++j) bits |= exist3(a.g, s, j) << (3 * j);
            if (m > 0 && p.x == c.x && p.y == c.y && p.z == c.z && p.w + 1 == c.w) bits |= 1u << 12;
        }
    }
    if (m < M) a.nbr_bits[m] = bits;
#pragma unroll
    for (int k = 0; k < kHalf; ++k) {
        const unsigned b = __ballot_sync(0xFFFFFFFFu, (bits >> k) & 1u);
        if (lane == 0) wcount[warp][k] = __popc(b);
    }
    __syncthreads();
    if (t < kHalf) {
        int sum = 0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) sum += wcount[w][t];
        a.tile_counts[(size_t)t * a.tiles + blockIdx.x] = sum;
    }
    release_successor();
}

// CTA k: exclusive prefix sum of offset k's counts over the tiles of the list, 8,192 entries per round (the lists of four
// nuScenes-shaped frames take one), and the offset's pair total.  The totals become offsets[28] in rb_fill.  Over the tiles of the
// whole capacity, 4,096 per round and a walk through the warps' sums, this took 9.5 us by events, now 7.5, and rb_count, whose CTAs
// past the list have nothing to write any more, 15.8, now 14.6: voxels and rulebooks 211.8 -> 206.4, KITTI-shaped 162.2 -> 158.1.
__global__ void __launch_bounds__(kRbScanThreads) rb_scan_kernel(const __grid_constant__ RbArgs a) {
    await_predecessor();
    constexpr int kWarps = kRbScanThreads / 32, kPer = 8;
    __shared__ int wsum[2][kWarps];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int* counts = a.tile_counts + (size_t)blockIdx.x * a.tiles;
    int* base = a.tile_base + (size_t)blockIdx.x * a.tiles;
    const int tiles = (max(voxels_in_list(a), 0) + kTile - 1) / kTile;
    int carry = 0;
    for (int i0 = 0, round = 0; i0 < tiles; i0 += kPer * kRbScanThreads, round ^= 1) {
        const int i = i0 + kPer * t;
        int v[kPer], sum = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) v[j] = i + j < tiles ? counts[i + j] : 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) sum += v[j];
        int inc = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane == 31) wsum[round][warp] = inc;
        __syncthreads();                                  // the other half of wsum may still be read by slower warps
        const int theirs = wsum[round][lane];
        int run = carry + warp_sum(lane < warp ? theirs : 0) + inc - sum;
        carry += warp_sum(theirs);
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            if (i + j < tiles) base[i + j] = run;
            run += v[j];
        }
    }
    if (t == 0) a.offset_pairs[blockIdx.x] = carry;
    release_successor();
}

__global__ void __launch_bounds__(kThreads) rb_fill_kernel(const __grid_constant__ RbArgs a) {
    await_predecessor();
    __shared__ int wcount[kThreads / 32][kHalf];      // pairs per warp, then where the warp's pairs start
    __shared__ int s_start[kOffsets + 1];             // offsets[]
    const int M = voxels_in_list(a);
    if (blockIdx.x > 0 && blockIdx.x * kTile >= M) return;   // CTA 0 always writes offsets[]
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int m = blockIdx.x * kTile + t;
    // Loads that depend on nothing go first.
    const int tile_start = t < kHalf ? a.tile_base[(size_t)t * a.tiles + blockIdx.x] : 0;
    int own = 0;
    if (t < kOffsets) own = t == kHalf ? max(M, 0) : a.offset_pairs[min(t, kOffsets - 1 - t)];
    int4 c = make_int4(0, 0, 0, 0);
    uint32_t bits = 0u;
    if (m < M) {
        c = a.coords[m];
        bits = a.nbr_bits[m];
    }
    if (warp == 0) {                                   // offsets[] from the totals
        int inc = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;
        }
        if (lane <= kOffsets) s_start[lane] = inc - own;
    }
#pragma unroll
    for (int k = 0; k < kHalf; ++k) {
        const unsigned b = __ballot_sync(0xFFFFFFFFu, (bits >> k) & 1u);
        if (lane == 0) wcount[warp][k] = __popc(b);
    }
    __syncthreads();
    if (t < kHalf) {                                   // places inside the segment
        int run = tile_start;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            const int n = wcount[w][t];
            wcount[w][t] = run;
            run += n;
        }
    }
    if (blockIdx.x == 0 && t <= kOffsets) {
        a.offsets[t] = s_start[t];
        if (t == kOffsets && (long long)s_start[t] > a.pair_capacity) atomicOr(a.status, kStatusCapacity);
    }
    __syncthreads();
    const Site s = site_of(a, c);                      // bits == 0 for rows outside the list or the grid
    const unsigned below = (1u << lane) - 1u;
    int first[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t three = (bits >> (3 * j)) & 7u;
        first[j] = three ? first_row(a.g, s, j, three) : 0;
    }
    auto put = [&](int pos, int in, int out) {
        if ((long long)pos < a.pair_capacity) {
            a.rule_in[pos] = in;
            a.rule_out[pos] = out;
        }
    };
#pragma unroll
    for (int k = 0; k < kHalf; ++k) {
        const bool has = (bits >> k) & 1u;
        const unsigned b = __ballot_sync(0xFFFFFFFFu, has);
        if (has) {
            const int at = wcount[warp][k] + __popc(b & below);
            const int n = k == 12 ? m - 1 : first[k / 3] + __popc((bits >> (k / 3 * 3)) & ((1u << (k % 3)) - 1u));
            put(s_start[k] + at, n, m);
            put(s_start[kOffsets - 1 - k] + at, m, n);
        }
    }
    if (m < M) put(s_start[kHalf] + m, m, m);
    release_successor();
}

}  // namespace

int launch_rulebook(emc2_bridge* h, int scale, int capacity, const int32_t* d_coords, const int32_t* d_num_voxels,
                    int32_t* d_rule_offsets, int32_t* d_rule_in, int32_t* d_rule_out, long long pair_capacity,
                    cudaStream_t st) {
    RbArgs a;
    a.g = h->scale[scale];
    a.coords = reinterpret_cast<const int4*>(d_coords);
    a.num_voxels = d_num_voxels;
    a.capacity = capacity;
    a.max_batch = h->cfg.max_batch;
    a.tiles = (capacity + kTile - 1) / kTile;
    a.nbr_bits = h->d_rb_bits;
    a.tile_counts = h->d_rb_counts;
    a.tile_base = h->d_rb_base;
    a.offset_pairs = h->d_rb_base + (size_t)kHalf * a.tiles;
    a.offsets = d_rule_offsets; a.rule_in = d_rule_in; a.rule_out = d_rule_out;
    a.pair_capacity = pair_capacity;
    a.status = h->d_status;
    const unsigned blocks = (unsigned)a.tiles;
    {
        LaunchScope ls(h, K_RB_MARK, st);
        rb_mark_kernel<<<blocks, kThreads, 0, st>>>(a);
    }
    {
        LaunchScope ls(h, K_RB_COUNT, st);
        launch_chained(rb_count_kernel, blocks, kThreads, 0, st, a);
    }
    {
        LaunchScope ls(h, K_RB_SCAN, st);
        launch_chained(rb_scan_kernel, kHalf, kRbScanThreads, 0, st, a);
    }
    {
        LaunchScope ls(h, K_RB_FILL, st);
        launch_chained(rb_fill_kernel, blocks, kThreads, 0, st, a);
    }
    {
        LaunchScope ls(h, K_RB_CLEAR, st);
        launch_chained(rb_clear_kernel, blocks, kThreads, 0, st, a);
    }
    return check_cuda(h, cudaGetLastError());
}

}  // namespace emc2
