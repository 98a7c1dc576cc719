// Stage 2 of the bridge: LiDAR-to-camera projection with an in-frustum mask, then a bilinear
// gather from the chosen camera's channels-last feature map (Sec. 3.1; zero rows for points
// without a pixel, Fig. 5).
//
// One CTA owns a tile of 256 consecutive points.  Phase 1: one thread per point projects into
// all K cameras (fp32 fma chain and IEEE divide, so the mask is reproducible bit for bit),
// writes uvd / mask / camera, and leaves one 16-byte record per point in shared memory: the
// address of tap (y0, x0), two clamp flags and the two weights.  Phase 2: the CTA is laid out
// as 16 rows x (Cf/4) columns of threads; every thread keeps its float4 column and walks the
// tile's rows 16 at a time, so a warp's 128-bit loads and stores cover whole contiguous rows,
// no index division is needed, and each thread has 16 independent tap loads in flight.
#include "bridge_internal.cuh"

namespace emc2 {
namespace {

struct PgArgs {
    const float* pts;
    const float* proj;
    const float4* feat;
    float* uvd;
    uint8_t* vis;
    int8_t* cam;
    float4* out;
    long long total;
    int N, K, H, W, Hf, Wf, cf4;
    float min_depth, inv_stride, offset;
    bool stream;          // rows too many for L2: streaming stores
};

// Projection of one point into the K cameras of its frame (P: [K][3][4] row-major).
struct Projected {
    unsigned mask;      // bit k: visible in camera k
    int best;           // lowest visible camera, -1 if none
    float u, v, d;      // pixel and depth in `best`; (-1, -1, depth in camera 0 or 0) if none
};

// Two fp32 operations per instruction (fma.rn.f32x2 and mul.rn.f32x2 of sm_100): the same roundings as the
// scalar forms.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// A camera's matrix as the projection reads it: rows 0 and 1 side by side, for paired arithmetic.
struct __align__(16) Camera {
    uint64_t x, y, z, w;    // columns of rows 0 and 1
    float4 r2;              // row 2
};

// (t0, t1) and t2: the numerators and the depth of one point, fp32 fma chains.
__device__ __forceinline__ void chains(const Camera& c, float x, float y, float z, uint64_t& t01, float& t2) {
    t01 = fma2(c.x, pack2(x, x), fma2(c.y, pack2(y, y), fma2(c.z, pack2(z, z), c.w)));
    t2 = __fmaf_rn(c.r2.x, x, __fmaf_rn(c.r2.y, y, __fmaf_rn(c.r2.z, z, c.r2.w)));
}

// The visibility decision is the one of the plain definition (fp32 fma chains, IEEE divide, compare), but
// the divide is only executed where it can matter: the distance of the numerator from the image centre,
// compared with half the image size scaled by the depth, settles every pixel that is not within `eps` of an
// image edge (eps is far above the roundings of these products), and only the chosen camera's (u, v) is
// divided out.  The loop over the cameras has no branches; cameras that are left undecided are taken up
// after it.  `cam`: the frame's K cameras in shared memory.
// A warp of the six-camera workload took 860 instructions with a test per camera in scalar arithmetic and divides for
// the six cell indices, now 680.  That shows in project_route_kernel where instruction issue bounds it: 32 frames of
// 262,144 points 222 -> 179 us, eight KITTI-shaped frames 33.9 -> 31.2.  On four nuScenes-shaped frames it did not
// (43.9 and 44.3 us) as long as their marks were queueing at the hottest sectors of the stores (see frames_side_by_side).
__device__ __forceinline__ Projected project_point(const Camera* cam, int K, float x, float y, float z,
                                                    int W, int H, float min_depth) {
    Projected r;
    const float fw = (float)W, fh = (float)H;
    const float cu = 0.5f * fw, cv = 0.5f * fh;
    const float eu = 1e-2f + 1e-6f * fw, ev = 1e-2f + 1e-6f * fh;
    const uint64_t centre = pack2(-cu, -cv), inside = pack2(cu - eu, cv - ev), outside = pack2(cu + eu, cv + ev);
    unsigned mask = 0u, open = 0u, bit = 1u;
#pragma unroll 2
    for (int k = 0; k < K; ++k, bit += bit) {
        uint64_t t01;
        float t2, au, av, iu, iv, ou, ov;
        chains(cam[k], x, y, z, t01, t2);
        const uint64_t dd = pack2(t2, t2);
        unpack2(fma2(centre, dd, t01), au, av);
        unpack2(mul2(inside, dd), iu, iv);
        unpack2(mul2(outside, dd), ou, ov);
        if (t2 > min_depth) {                     // false for NaN
            const bool in_sure = (fabsf(au) < iu) & (fabsf(av) < iv);
            const bool out_sure = (fabsf(au) > ou) | (fabsf(av) > ov);
            if (in_sure) mask |= bit;
            else if (!out_sure) open |= bit;
        }
    }
    for (; open; open &= open - 1u) {             // within a hair of an edge, or not finite: decide exactly
        const int k = __ffs(open) - 1;
        uint64_t t01;
        float t0, t1, t2;
        chains(cam[k], x, y, z, t01, t2);
        unpack2(t01, t0, t1);
        const float u = __fdiv_rn(t0, t2), v = __fdiv_rn(t1, t2);
        if ((u >= 0.0f) && (u < fw) && (v >= 0.0f) && (v < fh)) mask |= 1u << k;
    }
    r.mask = mask;
    r.best = __ffs(mask) - 1;
    uint64_t t01;
    chains(cam[max(r.best, 0)], x, y, z, t01, r.d);
    if (mask) {
        float t0, t1;
        unpack2(t01, t0, t1);
        r.u = __fdiv_rn(t0, r.d);
        r.v = __fdiv_rn(t1, r.d);
    } else {
        r.u = -1.0f; r.v = -1.0f;
        if (!isfinite(r.d)) r.d = 0.0f;           // depth in camera 0
    }
    return r;
}

// Copies the 3x4 matrices of `frames` frames of K cameras, from frame b on, into shared memory.
__device__ __forceinline__ void load_cameras(const float* __restrict__ proj, int b, int frames, int K, Camera* cam) {
    const float* src = proj + (size_t)b * K * 12;
    for (int i = threadIdx.x; i < frames * K * 12; i += blockDim.x) {
        const int k = i / 12, r = (i % 12) / 4, c = i % 4;
        reinterpret_cast<float*>(cam + k)[r < 2 ? 2 * c + r : 8 + c] = __ldg(src + i);
    }
}

// CF4 > 0: Cf/4 known at compile time, blockDim.x == 16 * CF4; else blockDim.x == row_threads(cf4), with 40 registers
// (three CTAs per SM; left to itself the compiler takes 32 and the rows lose their loads in flight: 256 channels,
// 1,800 tiles of mostly visible points: 127 -> 136 us).  Rows of more than 1 KB and an odd number of columns are the
// one case where whole rows can lose against one divide per float4, which kept all stores on sectors: 260 channels,
// 1,800 tiles: 99 against 87 us where few points are visible, 156 against 169 where most are.
// kFrames: most frames that the points of a tile belong to, see frames_of_tile: two but for frames of fewer than 255
// points, whose cameras are all staged at once (32 frames of 8 points through 6 cameras: 31 us with the cameras of two
// frames at a time in turn, 10.3 with every point reading its own from global memory, 9.8 this way).
template <int C, int CF4, int kFrames = 2>
__global__ void __launch_bounds__(CF4 > 0 ? 16 * CF4 : kMaxRowThreads, CF4 > 0 ? 0 : 3) project_gather_kernel(PgArgs a) {
    __shared__ __align__(16) float sp[kTile * C];
    __shared__ float suvd[kTile * 3];
    __shared__ uint4 srow[kTile];          // {tap (y0,x0) as a float4 index, clamp flags, wx, wy}
    __shared__ Camera sP[kFrames * EMC2_MAX_CAMERAS];      // cameras of the tile's frames

    const long long g0 = (long long)blockIdx.x * kTile;
    const int npts = (int)min((long long)kTile, a.total - g0);
    load_tile_f32(a.pts + g0 * C, npts * C, sp);
    const int bfirst = (int)(g0 / a.N);
    const int nframes = (int)((g0 + npts - 1) / a.N) - bfirst + 1;
    const int t = threadIdx.x;
    const int cf4 = CF4 > 0 ? CF4 : a.cf4;
    load_cameras(a.proj, bfirst, nframes, a.K, sP);
    __syncthreads();
    if (t < npts) {
        const float x = sp[t * C], y = sp[t * C + 1], z = sp[t * C + 2];
        const long long gi = g0 + t;
        const int b = (int)(gi / a.N);
        const Projected pr = project_point(sP + (b - bfirst) * a.K, a.K, x, y, z, a.W, a.H, a.min_depth);
        suvd[t * 3] = pr.u; suvd[t * 3 + 1] = pr.v; suvd[t * 3 + 2] = pr.d;
        a.vis[gi] = (uint8_t)pr.mask;
        a.cam[gi] = (int8_t)pr.best;
        const uint4 rec = tap_record(b, pr.best, pr.u, pr.v, a.K, a.Hf, a.Wf, cf4, a.inv_stride, a.offset);
        srow[t] = rec;
    }
    __syncthreads();

    // uvd: the tile's 3*npts floats are contiguous in global memory.
    for (int i = t; i < npts * 3; i += blockDim.x) a.uvd[g0 * 3 + i] = suvd[i];

    // Rows that fit in L2 are stored plainly, because the dispatch reads them next: us for this kernel and the stage call of
    // the dispatch, streaming / plain stores: one frame of 120,000 points 64 channels (31 MB) 30.7 / 29.4, 256 channels
    // (123 MB) 89.0 / 84.0, two frames of 120,001 80 channels (77 MB) 72.8 / 69.6.  By itself this kernel loses up to 2 us,
    // because the next stores have to write them back first (12.3 / 14.0, 38.6 / 39.4, 36.3 / 36.2).  Past L2 the plain
    // stores only lose: 154 MB 160.1 / 161.8, 246 MB 180.7 / 182.1, 384 MB 275.3 / 276.5.
    float4* out = a.out + (size_t)g0 * cf4;
    const uint32_t dyv = (uint32_t)a.Wf * cf4;
    auto store = [&](float4* p, const float4& v) { if (a.stream) __stcs(p, v); else *p = v; };
    if (CF4 > 0 || cf4 <= (int)blockDim.x) {
        const int c = t % cf4, rows = CF4 > 0 ? 16 : (int)blockDim.x / cf4;
#pragma unroll 4
        for (int r = t / cf4; r < npts; r += rows)
            store(out + r * cf4 + c, gather_column(a.feat, srow[r], c, (uint32_t)cf4, dyv));
    } else {
        const int items = npts * cf4;
        for (int i = t; i < items; i += blockDim.x) {
            const int r = i / cf4, c = i - r * cf4;
            store(out + i, gather_column(a.feat, srow[r], c, (uint32_t)cf4, dyv));
        }
    }
}

// ------------------------------------------------------------------ stages 2 - 4 in one pass
// The one-call path (emc2_bridge_run) does not send the gathered rows through memory twice.
//   project_route   per 256-point tile of a frame: projection, mask, camera, uvd, and - since the
//                   mask is now known - the expert id and the tile's expert histogram.
//   route_scan      tile histograms -> frame offsets and tile bases (shared with the staged path).
//   gather_scatter  per tile: stable rank of every point inside its expert's segment, then each
//                   feature row is blended once and stored twice, at its own row of `gathered`
//                   and at its slot of `feat_out`; point rows and the permutation go along.
// Outputs are those of the staged calls, bit for bit.
struct PrArgs {
    const float* pts;
    const float* proj;
    float* uvd;
    uint8_t* vis;
    int8_t* cam;
    uint8_t* expert;
    int* tile_counts;     // [B, tiles, E]
    int N, tiles, K, H, W;
    float min_depth;
    RouteParams rp;
    int B;
    FastDiv group;        // frames of a group, see marking_grid
    int frame0;           // kMark: frame index (in the whole batch) of this launch's first frame
    ScaleDev s0, s1;      // kMark: the voxel grids whose cells the points mark
    float4* bev;          // kMark: BEV image to zero (bev_n4 float4), or null
    uint32_t bev_n4;
    ScanReset reset;      // kMark: state of the rank scan to zero
    TileMarks marks;      // kNote
};

// See marking_grid; tiles never straddle frames.  kMark: the kernel also does the
// voxelizer's marking pass (every point marks its cell in both scales' stores, and the BEV image
// is zeroed, spread over the grid), so that stage 1 starts from marked stores and reads the
// points once less; the reductions are fire-and-forget and land while the projection computes.
// kNote: and notes the tiles that they touch (see keeps_frame_notes).  A variant of its own, so that calls without notes have
// neither their shared memory nor their code: one frame of 30,000 points and 256 channels 47.2 -> 46.0 us, of 20,000 and 192
// 39.2 -> 38.0.
// Bound by instruction issue (0.82 per cycle and scheduler) where the marks' sectors are in L2: the experts are counted by one
// reduction of packed fields per warp, the words of a frame's notes come from a table, one CTA resets the scan and a warp
// stores its own pixels.  With ballots per expert, divides for the words and the pixels stored by the CTA (with notes, us)
// four nuScenes-shaped frames took 39.4, now 38.0, 32 KITTI-shaped ones of 262,144 points 168.5, now 161, with six cameras 220, now
// 210; eight of 120,000 points 33.3, now 33.1.
template <int C, bool kMark, bool kNote = false>
__global__ void __launch_bounds__(kThreads, 8) project_route_kernel(const __grid_constant__ PrArgs a) {
    __shared__ __align__(16) float suvd[kTile * 3];
    __shared__ int hist[EMC2_MAX_EXPERTS];
    __shared__ Camera sP[EMC2_MAX_CAMERAS];
    const int t = threadIdx.x, lane = t & 31;
    uint32_t tile_u, in_group;
    a.group.divmod(blockIdx.x, tile_u, in_group);
    const int tile = (int)tile_u, b = (int)(blockIdx.y * a.group.d + in_group);
    if (b < a.B) load_cameras(a.proj, b, 1, a.K, sP);
    const int i0 = tile * kTile;
    const int npts = b < a.B ? min(kTile, a.N - i0) : 0;       // the last group can have fewer frames
    const size_t g0 = (size_t)b * a.N + i0;
    if (t < EMC2_MAX_EXPERTS) hist[t] = 0;
    FrameTiles* const tiles = frame_tiles<kNote>();
    if (kNote) begin_tiles(*tiles);
    __syncthreads();
    int e = -1;
    if (t < npts) {
        const float* p = a.pts + (g0 + t) * C;
        float x, y, z;
        if (C == 4) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(p));
            x = q.x; y = q.y; z = q.z;
        } else {
            x = __ldg(p); y = __ldg(p + 1); z = __ldg(p + 2);
        }
        if (kMark) {
            int at[2];
            mark_point(a.s0, a.s1, x, y, z, a.frame0 + b, at);
            if (kNote) note_tiles(*tiles, a.marks, a.frame0 + b, at);
        }
        const Projected pr = project_point(sP, a.K, x, y, z, a.W, a.H, a.min_depth);
        suvd[t * 3] = pr.u; suvd[t * 3 + 1] = pr.v; suvd[t * 3 + 2] = pr.d;
        a.vis[g0 + t] = (uint8_t)pr.mask;
        a.cam[g0 + t] = (int8_t)pr.best;
        const float r2 = __fmaf_rn(x, x, __fmul_rn(y, y));
        int bucket = 0;
        for (int k = 0; k < a.rp.T; ++k) bucket += (r2 >= a.rp.thr2[k]) ? 1 : 0;
        e = a.rp.lut[(pr.mask != 0u ? 8 : 0) + bucket];
        a.expert[g0 + t] = (uint8_t)e;
    }
    // The tile's experts, five at a time in fields of six bits.
    for (int k0 = 0; k0 < a.rp.E; k0 += 5) {
        const unsigned field = 6u * (unsigned)(e - k0);
        const unsigned sum = __reduce_add_sync(0xFFFFFFFFu, (unsigned)(e - k0) < 5u ? 1u << field : 0u);
        if (lane < 5 && k0 + lane < a.rp.E) atomicAdd(&hist[k0 + lane], (int)(sum >> (6 * lane) & 63u));
    }
    __syncwarp();
    // A warp's pixels are contiguous in global memory: whole 16-byte groups, if they are aligned.
    const int w0 = t - lane;
    float* uvd = a.uvd + (g0 + w0) * 3;
    if (npts - w0 >= 32 && (reinterpret_cast<uintptr_t>(uvd) & 15) == 0) {
        if (lane < 24) reinterpret_cast<float4*>(uvd)[lane] = reinterpret_cast<const float4*>(suvd + w0 * 3)[lane];
    } else {
        for (int i = lane; i < min(npts - w0, 32) * 3; i += 32) uvd[i] = suvd[w0 * 3 + i];
    }
    __syncthreads();
    if (t < a.rp.E && b < a.B) a.tile_counts[((size_t)b * a.tiles + tile) * a.rp.E + t] = hist[t];
    if (kNote && b < a.B) publish_tiles(*tiles, a.marks, a.frame0 + b, (uint32_t)tile);
    if (kMark) {
        if (blockIdx.x + blockIdx.y == 0) reset_scan(a.reset);
        if (a.bev) zero_bev(a.bev, a.bev_n4);
    }
    release_successor();
}

struct GsArgs {
    const float* pts;
    const float* uvd;
    const int8_t* cam;
    const uint8_t* expert;
    const int* tile_base;     // [B, tiles, E]
    const float4* feat;
    int32_t* perm;
    float* pts_out;
    float4* gathered;
    float4* feat_out;
    int N, tiles, E, K, Hf, Wf, cf4;
    float inv_stride, offset;
};

// CF4 > 0: Cf/4 known at compile time, blockDim.x == kGsRows<CF4> * CF4; else blockDim.x == row_threads(cf4).
// Two rows of 4 Cf bytes per point are written, 384 MB each on four nuScenes-shaped frames.  A plain kernel writes
// those bytes in 113 us, this one takes 176 with its taps (188 before the point rows left in expert order; 158 of those
// without the taps).  No unit of the chip is busy all the time; what the tap reads and the two streams of writes cost
// beyond the writes alone is how they interleave.  More resident warps do not move it, nor do more rows in flight per
// thread or other cache policies of the stores; a persistent grid writes 10 % slower than tiles in launch order.
// Rows at a time, with the registers the compiler takes or is held to, and the time alone (us):
//   80 channels, 4 x 300,000 points, C = 5        64 channels, 8 x 120,000 points, C = 4
//     16 rows, 42 registers, 40 warps   176         32 rows, 40 registers, 48 warps   108
//     16 rows, 32 registers, 50 warps   179         32 rows, 32 registers, 64 warps   109
//     16 rows, 32 registers, 60 warps   182         32 rows, 56 registers, 32 warps   115
//     24 rows, 40 registers, 45 warps   174         16 rows, 40 registers, 48 warps   111
//     24 rows, 32 registers, 60 warps   178         16 rows, 32 registers, 64 warps   113
//     32 rows, 40 registers, 40 warps   187         16 rows, 56 registers, 32 warps   109
// (32 registers spill a word; as a step the rows of 80 channels differ by 1 %.)  One small frame of 64 channels: 32 rows
// 10.7 us, 16 rows 12.7: a tile is through sooner.  Other widths take as many rows as 512 threads hold (128 channels: 90
// -> 83 us).
template <int CF4> constexpr int kGsRows = CF4 == 16 ? 32 : 16;

template <int C, int CF4>
__global__ void __launch_bounds__(CF4 > 0 ? kGsRows<CF4> * CF4 : kMaxRowThreads) gather_scatter_kernel(const __grid_constant__ GsArgs a) {
    await_predecessor();
    constexpr int kRows = kGsRows<CF4>;
    __shared__ uint4 srow[kTile];
    __shared__ TileOrder<C> order;
    const int b = blockIdx.y, tile = blockIdx.x, t = threadIdx.x;
    const int i0 = tile * kTile;
    const int npts = min(kTile, a.N - i0);
    const size_t f0 = (size_t)b * a.N;        // first row of the frame
    const size_t g0 = f0 + i0;
    const int cf4 = CF4 > 0 ? CF4 : a.cf4;
    // Everything the tile needs is requested first: nothing below waits for a second round trip to memory
    // before the rows start to move.
    float u = 0.f, v = 0.f;
    int cam = -1;
    if (t < npts) {
        u = a.uvd[(g0 + t) * 3];
        v = a.uvd[(g0 + t) * 3 + 1];
        cam = (int)a.cam[g0 + t];
    }
    const TilePoint<C> p = load_tile_point<C>(order, a.pts, a.expert, a.tile_base + ((size_t)b * a.tiles + tile) * a.E, g0, npts, a.E);
    if (t < npts) srow[t] = tap_record(b, cam, u, v, a.K, a.Hf, a.Wf, cf4, a.inv_stride, a.offset);
    order_tile<C>(order, p, a.perm, a.pts_out, f0, i0, npts, a.E);
    // Feature rows: blockDim.x / (Cf/4) rows x Cf/4 columns of threads; blended once, stored at both places
    // (the rows in point order only if the caller wants them).
    const bool keep = a.gathered != nullptr;
    float4* out = a.gathered + g0 * cf4;
    float4* fdst = a.feat_out + f0 * cf4;
    const uint32_t dyv = (uint32_t)a.Wf * cf4;
    if (CF4 > 0 || cf4 <= (int)blockDim.x) {
        const int c = t % cf4, rows = CF4 > 0 ? kRows : (int)blockDim.x / cf4;
#pragma unroll 4
        for (int r = t / cf4; r < npts; r += rows) {
            const float4 o = gather_column(a.feat, srow[r], c, (uint32_t)cf4, dyv);
            if (keep) __stcs(out + r * cf4 + c, o);
            __stcs(fdst + (size_t)order.dest[r] * cf4 + c, o);
        }
    } else {
        const int items = npts * cf4;
        for (int i = t; i < items; i += blockDim.x) {
            const int r = i / cf4, c = i - r * cf4;
            const float4 o = gather_column(a.feat, srow[r], c, (uint32_t)cf4, dyv);
            if (keep) __stcs(out + i, o);
            __stcs(fdst + (size_t)order.dest[r] * cf4 + c, o);
        }
    }
    release_successor();
}

// ---- the same pass with the rows staged in shared memory and written by bulk asynchronous copies
// A thread of gather_scatter_kernel issues, per 16 bytes of output, four 128-bit tap loads and two
// 128-bit global stores; the load/store path of the SM is its busiest unit.  Here the blended
// values go to shared memory instead, a sub-tile of 32 rows at a time (the rows of one warp of the
// ranking phase), once in point order and once ordered by expert.  The first copy is one contiguous
// block of `gathered`; in the second, the rows of one expert are one contiguous run of `feat_out`
// (ranks inside a tile are stable and tile bases are prefix sums), so a sub-tile leaves as at most
// 1 + E bulk copies (cp.async.bulk shared -> global) issued by one warp, and the global stores no
// longer pass through the threads' load/store instructions.  Two stage buffers: the copies of one
// sub-tile run while the next is blended.
__device__ __forceinline__ void bulk_store(void* gdst, const void* ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 :: "l"(gdst), "r"((uint32_t)__cvta_generic_to_shared(ssrc)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Waits until at most `kPending` of this thread's bulk groups still read their shared-memory source.
template <int kPending>
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" :: "n"(kPending) : "memory");
}
// Makes this thread's earlier shared-memory writes visible to the asynchronous copy engine.
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// kBoth: also stage and bulk-copy the rows in point order; otherwise those are stored from registers.
template <int C, int CF4, bool kBoth>
__global__ void __launch_bounds__(16 * CF4) gather_scatter_bulk_kernel(const __grid_constant__ GsArgs a) {
    await_predecessor();
    constexpr int kSub = 32, kBufs = 2, kWarpsTile = kTile / 32;
    __shared__ __align__(128) float4 stage[kBufs][kBoth ? 2 : 1][kSub * CF4];   // [buffer][expert order, point order]
    __shared__ uint4 srow[kTile];
    __shared__ int sdest[kTile];
    __shared__ uint8_t spos[kTile];                       // row's place in its sub-tile when ordered by expert
    __shared__ int wcnt[kWarpsTile][EMC2_MAX_EXPERTS];    // rows of expert k in sub-tile w
    __shared__ int wrow[kWarpsTile][EMC2_MAX_EXPERTS];    // first feat_out row (in the frame) of that run
    const int b = blockIdx.y, tile = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int i0 = tile * kTile;
    const int npts = min(kTile, a.N - i0);
    const size_t f0 = (size_t)b * a.N;
    const size_t g0 = f0 + i0;
    __shared__ int tbase[EMC2_MAX_EXPERTS];
    if (t >= (int)blockDim.x - EMC2_MAX_EXPERTS) {
        const int k = t - ((int)blockDim.x - EMC2_MAX_EXPERTS);
        if (k < a.E) tbase[k] = a.tile_base[((size_t)b * a.tiles + tile) * a.E + k];
    }

    int e = -1, rank = 0;
    if (t < kTile) {
        if (t < npts) {
            e = (int)a.expert[g0 + t];
            const float u = a.uvd[(g0 + t) * 3], v = a.uvd[(g0 + t) * 3 + 1];
            srow[t] = tap_record(b, (int)a.cam[g0 + t], u, v, a.K, a.Hf, a.Wf, CF4, a.inv_stride, a.offset);
        }
        for (int k = 0; k < a.E; ++k) {
            const unsigned m = __ballot_sync(0xFFFFFFFFu, e == k);
            if (e == k) rank = __popc(m & ((1u << lane) - 1u));
            if (lane == 0) wcnt[warp][k] = __popc(m);
        }
    }
    __syncthreads();
    if (t < npts) {
        int before = 0, below = 0;
        for (int w = 0; w < warp; ++w) before += wcnt[w][e];
        for (int k = 0; k < e; ++k) below += wcnt[warp][k];
        const int d = tbase[e] + before + rank;
        sdest[t] = d;
        spos[t] = (uint8_t)(below + rank);
        a.perm[f0 + d] = i0 + t;
    }
    if (t < kWarpsTile * a.E) {
        const int w = t / a.E, k = t - w * a.E;
        int before = 0;
        for (int w2 = 0; w2 < w; ++w2) before += wcnt[w2][k];
        wrow[w][k] = tbase[k] + before;
    }
    __syncthreads();

    const float* psrc = a.pts + g0 * C;
    float* pdst = a.pts_out + f0 * C;
    for (int i = t; i < npts * C; i += blockDim.x) {
        const int r = i / C, c = i - r * C;
        pdst[(size_t)sdest[r] * C + c] = __ldg(psrc + i);
    }

    const bool keep = a.gathered != nullptr;
    float4* out = a.gathered + g0 * CF4;
    float4* fdst = a.feat_out + f0 * CF4;
    const uint32_t dyv = (uint32_t)a.Wf * CF4;
    const int c = t % CF4, r0 = t / CF4;
    const int nsub = (npts + kSub - 1) / kSub;
    for (int s = 0; s < nsub; ++s) {
        const int buf = s & 1;
        if (s >= kBufs) {                                 // the copies that read this buffer must have read it
            if (warp == 0) bulk_wait_read<kBufs - 1>();
            __syncthreads();
        }
        const int nr = min(kSub, npts - s * kSub);
#pragma unroll
        for (int jj = 0; jj < kSub / 16; ++jj) {
            const int rl = r0 + 16 * jj;
            if (rl < nr) {
                const int r = s * kSub + rl;
                const float4 o = gather_column(a.feat, srow[r], c, (uint32_t)CF4, dyv);
                stage[buf][0][(int)spos[r] * CF4 + c] = o;
                if (kBoth) { if (keep) stage[buf][kBoth ? 1 : 0][rl * CF4 + c] = o; }
                else if (keep) __stcs(out + r * CF4 + c, o);
            }
        }
        fence_async_shared();
        __syncthreads();
        if (warp == 0) {
            if (lane < a.E) {
                const int cnt = wcnt[s][lane];
                int start = 0;
                for (int k = 0; k < lane; ++k) start += wcnt[s][k];
                if (cnt > 0)
                    bulk_store(fdst + (size_t)wrow[s][lane] * CF4, &stage[buf][0][start * CF4], (uint32_t)cnt * CF4 * 16u);
            } else if (kBoth && lane == 31 && keep) {
                bulk_store(out + (size_t)s * kSub * CF4, &stage[buf][kBoth ? 1 : 0][0], (uint32_t)nr * CF4 * 16u);
            }
            bulk_commit();
        }
    }
    if (warp == 0) bulk_wait_read<0>();                   // shared memory must outlive the copies that read it
}

// ---- the same pass with 256-bit accesses (sm_100: ld/st.global.v8.f32)
// A thread owns eight channels of a row instead of four: half as many load and store instructions
// (and requests into the SM's memory pipeline) per byte moved, 32 rows x Cf/8 columns per round.
// Needs Cf a multiple of 8 and 32-byte aligned maps and row buffers (checked at launch).
struct F8 { float v[8]; };

__device__ __forceinline__ F8 ldg8(const float* p) {
    F8 r;
    asm volatile("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3]), "=f"(r.v[4]), "=f"(r.v[5]), "=f"(r.v[6]), "=f"(r.v[7])
                 : "l"(p));
    return r;
}
__device__ __forceinline__ void stcs8(float* p, const F8& r) {
    asm volatile("st.global.cs.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 :: "l"(p), "f"(r.v[0]), "f"(r.v[1]), "f"(r.v[2]), "f"(r.v[3]), "f"(r.v[4]), "f"(r.v[5]), "f"(r.v[6]), "f"(r.v[7])
                 : "memory");
}

// Blended channels [8c, 8c + 8) of the row described by `rec` (zeros for kZeroRow); same arithmetic as blend().
__device__ __forceinline__ F8 gather_column8(const float* __restrict__ feat, const uint4& rec, int c, uint32_t cf4,
                                             uint32_t row_stride) {
    F8 o;
#pragma unroll
    for (int k = 0; k < 8; ++k) o.v[k] = 0.f;
    if (rec.x != kZeroRow) {
        const float* p = feat + ((size_t)rec.x << 2) + 8 * c;
        const size_t dx = (rec.y & 1u) ? (size_t)cf4 * 4 : 0, dy = (rec.y & 2u) ? (size_t)row_stride * 4 : 0;
        const F8 f00 = ldg8(p), f01 = ldg8(p + dx), f10 = ldg8(p + dy), f11 = ldg8(p + dy + dx);
        const float wx = __uint_as_float(rec.z), wy = __uint_as_float(rec.w);
        const float ax = 1.0f - wx, ay = 1.0f - wy;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            o.v[k] = ay * (ax * f00.v[k] + wx * f01.v[k]) + wy * (ax * f10.v[k] + wx * f11.v[k]);
    }
    return o;
}

template <int C, int CF8>
__global__ void __launch_bounds__(32 * CF8) gather_scatter_wide_kernel(const __grid_constant__ GsArgs a) {
    await_predecessor();
    __shared__ uint4 srow[kTile];
    __shared__ int sdest[kTile];
    __shared__ int wcnt[kTile / 32][EMC2_MAX_EXPERTS];
    __shared__ int tbase[EMC2_MAX_EXPERTS];
    const int b = blockIdx.y, tile = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int i0 = tile * kTile;
    const int npts = min(kTile, a.N - i0);
    const size_t f0 = (size_t)b * a.N;
    const size_t g0 = f0 + i0;
    constexpr int CF4 = 2 * CF8;
    if (t >= (int)blockDim.x - EMC2_MAX_EXPERTS) {
        const int k = t - ((int)blockDim.x - EMC2_MAX_EXPERTS);
        if (k < a.E) tbase[k] = a.tile_base[((size_t)b * a.tiles + tile) * a.E + k];
    }
    int e = -1, rank = 0;
    if (t < kTile) {
        if (t < npts) {
            e = (int)a.expert[g0 + t];
            const float u = a.uvd[(g0 + t) * 3], v = a.uvd[(g0 + t) * 3 + 1];
            srow[t] = tap_record(b, (int)a.cam[g0 + t], u, v, a.K, a.Hf, a.Wf, CF4, a.inv_stride, a.offset);
        }
        for (int k = 0; k < a.E; ++k) {
            const unsigned m = __ballot_sync(0xFFFFFFFFu, e == k);
            if (e == k) rank = __popc(m & ((1u << lane) - 1u));
            if (lane == 0) wcnt[warp][k] = __popc(m);
        }
    }
    __syncthreads();
    if (t < npts) {
        int before = 0;
        for (int w = 0; w < warp; ++w) before += wcnt[w][e];
        const int d = tbase[e] + before + rank;
        sdest[t] = d;
        a.perm[f0 + d] = i0 + t;
    }
    __syncthreads();
    const float* psrc = a.pts + g0 * C;
    float* pdst = a.pts_out + f0 * C;
    for (int i = t; i < npts * C; i += blockDim.x) {
        const int r = i / C, c = i - r * C;
        pdst[(size_t)sdest[r] * C + c] = __ldg(psrc + i);
    }
    const bool keep = a.gathered != nullptr;
    float* out = reinterpret_cast<float*>(a.gathered) + g0 * (size_t)(8 * CF8);
    float* fdst = reinterpret_cast<float*>(a.feat_out) + f0 * (size_t)(8 * CF8);
    const float* feat = reinterpret_cast<const float*>(a.feat);
    const uint32_t dyv = (uint32_t)a.Wf * CF4;
    const int c = t % CF8, r0 = t / CF8;
#pragma unroll 2
    for (int j = 0; j < kTile / 32; ++j) {
        const int r = r0 + 32 * j;
        if (r >= npts) break;
        const F8 o = gather_column8(feat, srow[r], c, (uint32_t)CF4, dyv);
        if (keep) stcs8(out + (size_t)r * (8 * CF8) + 8 * c, o);
        stcs8(fdst + (size_t)sdest[r] * (8 * CF8) + 8 * c, o);
    }
    release_successor();
}


template <int C>
void launch_gs(emc2_bridge* h, const GsArgs& a, dim3 grid, bool chained, cudaStream_t st) {
    LaunchScope ls(h, K_GATHER_SCATTER, st);
    const int mode = h->tune[EMC2_TUNE_ROW_STORE];
    if (mode == 1 && a.E < 31) {
        if (a.cf4 == 16) { launch_kernel(chained, gather_scatter_bulk_kernel<C, 16, true>, grid, 16 * 16, 0, st, a); return; }
        if (a.cf4 == 20) { launch_kernel(chained, gather_scatter_bulk_kernel<C, 20, true>, grid, 16 * 20, 0, st, a); return; }
    } else if (mode == 3 && ((reinterpret_cast<uintptr_t>(a.feat) | reinterpret_cast<uintptr_t>(a.gathered) |
                              reinterpret_cast<uintptr_t>(a.feat_out)) & 31) == 0) {
        if (a.cf4 == 16) { launch_kernel(chained, gather_scatter_wide_kernel<C, 8>, grid, 32 * 8, 0, st, a); return; }
        if (a.cf4 == 20) { launch_kernel(chained, gather_scatter_wide_kernel<C, 10>, grid, 32 * 10, 0, st, a); return; }
    } else if (mode == 2) {
        if (a.cf4 == 16) { launch_kernel(chained, gather_scatter_bulk_kernel<C, 16, false>, grid, 16 * 16, 0, st, a); return; }
        if (a.cf4 == 20) { launch_kernel(chained, gather_scatter_bulk_kernel<C, 20, false>, grid, 16 * 20, 0, st, a); return; }
    }
    switch (a.cf4) {
        case 16: launch_kernel(chained, gather_scatter_kernel<C, 16>, grid, kGsRows<16> * 16, 0, st, a); break;
        case 20: launch_kernel(chained, gather_scatter_kernel<C, 20>, grid, kGsRows<20> * 20, 0, st, a); break;
        default: launch_kernel(chained, gather_scatter_kernel<C, 0>, grid, row_threads(a.cf4), 0, st, a); break;
    }
}

// ------------------------------------------------------------------ planar -> channels-last
// Per map the planar data is a Cf x P matrix (P = Hf * Wf pixels) and the channels-last data its
// transpose.  A CTA moves `chan` channels x kPix pixels through shared memory.
//   in   one warp per channel row, 32 consecutive pixels (128 B) per instruction; a thread requests ten or twelve of
//        its words before it waits for any;
//   out  a warp instruction covers 8 pixels x 16 channels, 64 contiguous bytes of a pixel's row per four lanes.
//        With a row stride of kPix + 2 words the column reads from the tile (bank = 2 * channel + pixel mod 32) are
//        conflict-free.
// Bound by the memory system (each byte is read and written once).  The tile, measured on 12 maps of 113 x 200
// texels (us per call; 64 x 128 pixels, ragged at the last channels, is what every width took once):
//   channels                          8      32     48     64     80     96    128    192    256    512
//   64 x 128 pixels, ragged         10.3   14.5   19.1   27.4   41.5   49.7   57.9   88.4    111    220
//   all (at most 128) x 64 pixels   12.8   15.4   21.7   27.1   33.3   46.5   62.0   90.7    119    234
//   64 x 64 pixels                  12.8   14.8   21.2   27.2   37.4   49.8   51.7   76.3   98.8    194
//   all (at most 64) x 128 pixels    9.0   14.8   18.9   29.6   35.9   53.6   57.9   90.6    119    236
// So: 128 pixels up to 48 channels, where a tile of 64 is too little work for a CTA; chunks of 64 channels where they
// divide the width, whole sectors of the rows in small tiles; else as few CTAs per row as 128 channels allow, so that
// no CTA is left with a few channels.
constexpr int kClMaxChan = 128;
template <int kPix> constexpr int kClStride = kPix + 2;

struct ClTile {
    int pix, chan;
};

inline ClTile channels_last_tile(int Cf) {
    if (Cf <= 48) return {128, Cf};
    if (Cf % 64 == 0) return {64, 64};
    const int ctas = (Cf + kClMaxChan - 1) / kClMaxChan;
    return {64, ((Cf + ctas - 1) / ctas + 3) / 4 * 4};
}

template <int kPix>
__global__ void __launch_bounds__(256)
channels_last_kernel(const float* __restrict__ planar, float* __restrict__ last, int Cf, int P, int ptiles, int chan) {
    constexpr int kStride = kClStride<kPix>, kParts = kPix / 32, kBatch = kParts == 2 ? 10 : 12;
    extern __shared__ float tile[];                         // [chan][kStride]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t m = blockIdx.x / ptiles;
    const int p0 = (int)(blockIdx.x - m * ptiles) * kPix;
    const int c0 = blockIdx.y * chan;
    const int nc = min(chan, Cf - c0);
    const float* src = planar + (m * Cf + c0) * (size_t)P + p0;
    // Item i of a warp: part i % kParts of channel row warp + 8 * (i / kParts).
    bool in[kParts];
#pragma unroll
    for (int i = 0; i < kParts; ++i) in[i] = p0 + 32 * i + lane < P;
    const int items = kParts * ((nc - warp + 7) / 8);
    for (int i0 = 0; i0 < items; i0 += kBatch) {
        float v[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int c = warp + 8 * ((i0 + u) / kParts), part = u % kParts;
            v[u] = c < nc && in[part] ? __ldcs(src + (size_t)c * P + 32 * part + lane) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int c = warp + 8 * ((i0 + u) / kParts);
            if (c < nc) tile[c * kStride + 32 * (u % kParts) + lane] = v[u];
        }
    }
    __syncthreads();
    float* dst = last + (m * P + p0) * (size_t)Cf + c0;
    const int q8 = lane >> 2, cq = 4 * (lane & 3);          // pixel of a group of 8, channel of a group of 16
    const int quads = (nc + 15) / 16;
    for (int job = warp; job < quads * (kPix / 8); job += 8) {
        const int g = job / quads;                          // consecutive jobs share their pixels
        const int c = cq + 16 * (job - g * quads), q = 8 * g + q8;
        if (c >= nc || p0 + q >= P) continue;               // Cf % 4 == 0: a whole float4 or none
        const float* col = tile + c * kStride + q;
        // Not a streaming store: whoever takes the maps next finds the last ones in L2 (see pool_features_kernel).
        *reinterpret_cast<float4*>(dst + (size_t)q * Cf + c) =
            make_float4(col[0], col[kStride], col[2 * kStride], col[3 * kStride]);
    }
}

// ------------------------------------------------------------------ Multiscale Pooling (Sec. 3.5)
// One thread per (pooled texel, float4 column); grid = (columns of a pooled row, pooled rows,
// maps).  Consecutive threads read consecutive columns of the same input rows, so every load
// covers whole 256/320-byte rows.  Streams the maps once.  PW: window size known at compile time
// (2 and 4: all texels of a whole window are requested at once; 60 -> 40 us for 24 maps of 113 x 200 x 80 at
// p = 2), 0 = any.  The sum is rows outer, columns inner for every size.
// The maps are taken from the last one back: what was written last before this call, by the layout change for one, is
// what L2 still holds.  24 maps of 113 x 200 x 80 (174 MB, L2 126 MB) right after their layout change, the two calls
// together: 94.4 us in ascending order, 91.3 in descending order, 86.8 with the layout change's plain stores as well
// (this kernel, by events, 39.4 -> 35.9 -> 31.4 us).
template <int PW>
__global__ void __launch_bounds__(kThreads)
pool_features_kernel(const float4* __restrict__ feat, float4* __restrict__ pooled, int Hf, int Wf, int Hp, int Wp,
                     int cf4, int pw) {
    const int p = PW > 0 ? PW : pw;
    const int ic = blockIdx.x * kThreads + threadIdx.x;     // I * cf4 + c
    if (ic >= Wp * cf4) return;
    const int I = ic / cf4, c = ic - I * cf4;
    const int J = Hp - 1 - (int)blockIdx.y;
    const size_t m = gridDim.z - 1 - blockIdx.z;            // map index b * K + k
    const int j0 = J * p, j1 = min(Hf, j0 + p), i0 = I * p, i1 = min(Wf, i0 + p);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    auto add = [&](const float4& v) { s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w; };
    const float4* corner = feat + ((m * Hf + j0) * Wf + i0) * cf4 + c;
    if (PW > 0 && j1 - j0 == p && i1 - i0 == p) {
        constexpr int kW = PW > 0 ? PW : 1;
        float4 v[kW][kW];
#pragma unroll
        for (int j = 0; j < kW; ++j)
#pragma unroll
            for (int x = 0; x < kW; ++x) v[j][x] = __ldcs(corner + ((size_t)j * Wf + x) * cf4);
#pragma unroll
        for (int j = 0; j < kW; ++j)
#pragma unroll
            for (int x = 0; x < kW; ++x) add(v[j][x]);
    } else {
        // Four loads in flight at 40 registers.  The offset is 32 bits wide (a map has fewer float4 than that, see create)
        // and added to a pointer that steps from row to row: with a 64-bit product of both indices per load the kernel
        // spilled in this loop (24 maps of 113 x 200 x 80: p = 8 37.6 us, now 31.8; p = 5 42.5, now 36.3; one map of
        // 47 x 156 x 64, p = 8: 22.6, now 15.8).
        const uint32_t step = (uint32_t)Wf * (uint32_t)cf4;
        for (int j = j0; j < j1; ++j, corner += step) {
#pragma unroll 4
            for (int x = 0; x < i1 - i0; ++x) add(__ldcs(corner + (uint32_t)x * (uint32_t)cf4));
        }
    }
    const float inv = 1.0f / (float)((j1 - j0) * (i1 - i0));
    pooled[((m * Hp + J) * Wp) * cf4 + ic] = make_float4(s.x * inv, s.y * inv, s.z * inv, s.w * inv);
}

template <int C>
void launch_c(emc2_bridge* h, const PgArgs& a, int tiles, cudaStream_t st) {
    LaunchScope ls(h, K_PROJECT_GATHER, st);
    if (frames_of_tile(a.total / a.N, a.N) > 2) {
        project_gather_kernel<C, 0, EMC2_MAX_BATCH><<<tiles, row_threads(a.cf4), 0, st>>>(a);
        return;
    }
    switch (a.cf4) {
        case 16: project_gather_kernel<C, 16><<<tiles, 16 * 16, 0, st>>>(a); break;
        case 20: project_gather_kernel<C, 20><<<tiles, 16 * 20, 0, st>>>(a); break;
        default: project_gather_kernel<C, 0><<<tiles, row_threads(a.cf4), 0, st>>>(a); break;
    }
}

}  // namespace

int launch_project_gather(emc2_bridge* h, int B, int N, const float* d_points, const float* d_proj,
                          const float* d_feat, float* d_uvd, uint8_t* d_vis_mask, int8_t* d_cam,
                          float* d_gathered, cudaStream_t st) {
    const emc2_config_t& c = h->cfg;
    PgArgs a;
    a.pts = d_points; a.proj = d_proj; a.feat = reinterpret_cast<const float4*>(d_feat);
    a.uvd = d_uvd; a.vis = d_vis_mask; a.cam = d_cam; a.out = reinterpret_cast<float4*>(d_gathered);
    a.total = (long long)B * N;
    a.N = N; a.K = c.num_cameras; a.H = c.img_h; a.W = c.img_w; a.Hf = c.feat_h; a.Wf = c.feat_w;
    a.cf4 = c.feat_c / 4;
    a.min_depth = c.min_depth;
    a.inv_stride = 1.0f / (float)c.feat_stride;
    a.offset = c.feat_offset;
    a.stream = !rows_stay_in_l2((uint64_t)a.total, c.feat_c);
    const int tiles = (int)((a.total + kTile - 1) / kTile);
    if (tiles == 0) return EMC2_OK;
    if (c.point_floats == 4) launch_c<4>(h, a, tiles, st); else launch_c<5>(h, a, tiles, st);
    return check_cuda(h, cudaGetLastError());
}

// Frames [b0, b0 + B) of a batch whose buffers are given whole; `bev_frames` > 0: this launch also
// zeroes the BEV image of that many frames.
int launch_project_route(emc2_bridge* h, int b0, int B, int N, const float* d_points, const float* d_proj,
                         float* d_uvd, uint8_t* d_vis_mask, int8_t* d_cam, uint8_t* d_expert, bool mark,
                         float* d_bev_to_zero, int bev_frames, const TileMarks& marks, cudaStream_t st) {
    const emc2_config_t& c = h->cfg;
    const int tiles = (N + kTile - 1) / kTile;
    if (B == 0 || tiles == 0) return EMC2_OK;
    const FastDiv group = make_fast_div((uint32_t)frames_per_group(store_bytes(h), B));
    const dim3 grid = marking_grid(tiles, B, group);
    const size_t p0 = (size_t)b0 * N;                      // first point of the range
    PrArgs pa;
    pa.pts = d_points + p0 * c.point_floats; pa.proj = d_proj + (size_t)b0 * c.num_cameras * 12;
    pa.uvd = d_uvd + p0 * 3; pa.vis = d_vis_mask + p0; pa.cam = d_cam + p0;
    pa.expert = d_expert + p0; pa.tile_counts = h->d_tile_counts + (size_t)b0 * tiles * c.num_experts;
    pa.N = N; pa.tiles = tiles; pa.K = c.num_cameras; pa.H = c.img_h; pa.W = c.img_w;
    pa.min_depth = c.min_depth;
    pa.rp = route_params(h);
    pa.B = B; pa.group = group;
    pa.frame0 = b0;
    pa.s0 = h->scale[0]; pa.s1 = h->scale[1];
    pa.bev = nullptr; pa.bev_n4 = 0;
    pa.reset = scan_reset(h);
    pa.marks = marks;
    if (!mark || b0 > 0) { pa.reset.n = 0; pa.reset.totals[0] = pa.reset.totals[1] = nullptr; }
    if (mark && d_bev_to_zero && bev_frames > 0) {
        const size_t bev_n = (size_t)bev_frames * c.point_floats * h->scale[1].dims[1] * h->scale[1].dims[0];
        if (!bev_by_kernel(bev_n)) {
            cudaMemsetAsync(d_bev_to_zero, 0, bev_n * sizeof(float), st);
        } else {
            pa.bev = reinterpret_cast<float4*>(d_bev_to_zero);
            pa.bev_n4 = (uint32_t)(bev_n >> 2);
        }
    }
    {
        LaunchScope ls(h, K_PROJECT_ROUTE, st);
        if (c.point_floats == 4) {
            if (mark && pa.marks.marked[0]) project_route_kernel<4, true, true><<<grid, kThreads, 0, st>>>(pa);
            else if (mark) project_route_kernel<4, true><<<grid, kThreads, 0, st>>>(pa);
            else project_route_kernel<4, false><<<grid, kThreads, 0, st>>>(pa);
        } else {
            if (mark && pa.marks.marked[0]) project_route_kernel<5, true, true><<<grid, kThreads, 0, st>>>(pa);
            else if (mark) project_route_kernel<5, true><<<grid, kThreads, 0, st>>>(pa);
            else project_route_kernel<5, false><<<grid, kThreads, 0, st>>>(pa);
        }
    }
    return check_cuda(h, cudaGetLastError());
}

int launch_gather_scatter(emc2_bridge* h, int b0, int B, int N, const float* d_points, const float* d_feat,
                          const float* d_uvd, const int8_t* d_cam, float* d_gathered, const uint8_t* d_expert,
                          int32_t* d_perm, float* d_points_out, float* d_feat_out, bool chained, cudaStream_t st) {
    const emc2_config_t& c = h->cfg;
    if (B == 0) return EMC2_OK;
    const int tiles = (N + kTile - 1) / kTile;
    const dim3 grid(tiles > 0 ? tiles : 1, B);
    const int E = c.num_experts;
    const size_t p0 = (size_t)b0 * N, t0 = (size_t)b0 * tiles * E;
    if (tiles > 0) {
        GsArgs ga;
        ga.pts = d_points + p0 * c.point_floats; ga.uvd = d_uvd + p0 * 3; ga.cam = d_cam + p0; ga.expert = d_expert + p0;
        ga.tile_base = h->d_tile_base + t0;
        ga.feat = reinterpret_cast<const float4*>(d_feat + (size_t)b0 * c.num_cameras * c.feat_h * c.feat_w * c.feat_c);
        ga.perm = d_perm + p0; ga.pts_out = d_points_out + p0 * c.point_floats;
        ga.gathered = d_gathered ? reinterpret_cast<float4*>(d_gathered + p0 * c.feat_c) : nullptr;
        ga.feat_out = reinterpret_cast<float4*>(d_feat_out + p0 * c.feat_c);
        ga.N = N; ga.tiles = tiles; ga.E = E; ga.K = c.num_cameras; ga.Hf = c.feat_h; ga.Wf = c.feat_w;
        ga.cf4 = c.feat_c / 4;
        ga.inv_stride = 1.0f / (float)c.feat_stride;
        ga.offset = c.feat_offset;
        if (c.point_floats == 4) launch_gs<4>(h, ga, grid, chained, st); else launch_gs<5>(h, ga, grid, chained, st);
    }
    return check_cuda(h, cudaGetLastError());
}

int launch_channels_last(emc2_bridge* h, int B, const float* d_planar, float* d_feat, cudaStream_t st) {
    const emc2_config_t& c = h->cfg;
    const long long P = (long long)c.feat_h * c.feat_w;
    const ClTile tile = channels_last_tile(c.feat_c);
    const long long ptiles = (P + tile.pix - 1) / tile.pix;
    const long long ctas = (long long)B * c.num_cameras * ptiles;
    const int ct = (c.feat_c + tile.chan - 1) / tile.chan;
    if (P > 0x7FFFFFFFLL || ctas > 0x7FFFFFFFLL || ct > 65535) return EMC2_ERR_INVALID_ARG;
    LaunchScope ls(h, K_CHANNELS_LAST, st);
    const dim3 grid((unsigned)ctas, ct);
    if (tile.pix == 128)
        channels_last_kernel<128><<<grid, 256, (size_t)tile.chan * kClStride<128> * sizeof(float), st>>>(
            d_planar, d_feat, c.feat_c, (int)P, (int)ptiles, tile.chan);
    else
        channels_last_kernel<64><<<grid, 256, (size_t)tile.chan * kClStride<64> * sizeof(float), st>>>(
            d_planar, d_feat, c.feat_c, (int)P, (int)ptiles, tile.chan);
    return check_cuda(h, cudaGetLastError());
}

int launch_pool_features(emc2_bridge* h, int B, int p, const float* d_feat, float* d_pooled, cudaStream_t st) {
    const emc2_config_t& c = h->cfg;
    const int Hp = (c.feat_h + p - 1) / p, Wp = (c.feat_w + p - 1) / p, cf4 = c.feat_c / 4;
    if (Hp > 65535) return EMC2_ERR_INVALID_ARG;           // grid limit: one pooled row per blockIdx.y
    const dim3 grid((Wp * cf4 + kThreads - 1) / kThreads, Hp, B * c.num_cameras);
    {
        LaunchScope ls(h, K_POOL_FEATURES, st);
        auto kernel = p == 2 ? pool_features_kernel<2> : p == 4 ? pool_features_kernel<4> : pool_features_kernel<0>;
        kernel<<<grid, kThreads, 0, st>>>(reinterpret_cast<const float4*>(d_feat), reinterpret_cast<float4*>(d_pooled),
                                          c.feat_h, c.feat_w, Hp, Wp, cf4, p);
    }
    return check_cuda(h, cudaGetLastError());
}

}  // namespace emc2
