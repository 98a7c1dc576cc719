// Fusion by voxel (Fig. 5): the image features of the pixels that share a voxel's 3-D coordinate
// go with that voxel, voxels without such pixels get zero rows.  The pixels with a 3-D coordinate
// are the projected LiDAR points, so voxel m receives the mean of the gathered rows of its kept
// points that some camera sees.
//
// Rows are 256/320 bytes: adding them up with reductions would cost twenty 16-byte requests per
// point.  Instead the visible points are listed per voxel and each voxel reads its points' rows whole:
//   vif_scan   exclusive prefix sums of the voxels' kept-point counts (the prefix-sum indexing of Sec. 3.6) -> start
//              of every voxel's list.  The sums go over 1024 voxels; a CTA takes their part of the list array with one
//              ticket, so that no pass over all the counts has to come first.
//   vif_fill   every kept point that a camera sees takes a ticket in its voxel's list (one atomic with return).
//   vif_mean   16 voxels x Cf/4 columns of threads per CTA: a voxel's threads walk its list and
//              read each listed point's row with one contiguous 128-bit load per thread.
//   vif_sample the same, but the rows are blended from the feature maps on the spot
//              (emc2_voxel_image_sampled: no [points, Cf] buffer at all); for it vif_fill stores
//              each listed point's tap record (16 bytes) in place of its index.
#include "bridge_internal.cuh"

namespace emc2 {
namespace {

struct VifArgs {
    const int32_t* pv;          // [total] row of the point's voxel, -1 if none
    const int32_t* counts;      // [M] kept points per voxel
    const int32_t* num_voxels;  // device: voxels found by emc2_voxelize for this scale
    const uint8_t* vis;         // [total], or null: a point is visible iff cam[i] >= 0
    const float4* gathered;     // [total, cf4] (vif_mean)
    const int8_t* cam;          // [total] camera of every point (vif_sample)
    const float* uvd;           // [total, 3] pixel and depth in that camera (vif_sample)
    const float4* feat;         // feature maps (vif_sample)
    int N, K, Hf, Wf;
    float inv_stride, offset;
    int pool, Hp, Wp;           // pool > 1: taps are p x p window means of the maps (Multiscale Pooling folded
                                // into the sampling); Hp x Wp is the pooled map, inv_stride / offset describe it
    float4* vox_img;            // [capacity, cf4]
    int32_t* vox_cnt;           // [capacity]
    int* start;                 // [capacity] first list slot of each voxel
    int* cursor;                // [capacity] next free list slot of each voxel
    int* list;                  // [total] point indices
    uint4* recs;                // [total] vif_sample: tap record of every listed point, in list order
    unsigned long long* taken;  // list slots given out by vif_scan; zero between calls
    int* bad;                   // counts[] add up to more than there are points
    int* status;
    long long total;
    int capacity, cf4;
};

__device__ __forceinline__ int voxels_in_use(const VifArgs& a) { return min(*a.num_voxels, a.capacity); }

// A warp has kScanRows * 32 consecutive voxels, a CTA eight times as many and one ticket: tickets on one address are
// served one after another (about 10 ns each).  As a cooperative launch that summed all counts before any start was known
// this took 14.3 us for the lists of four nuScenes-shaped frames (mean of both scales, by events), now 10.7; the fill, which
// looked the start up and listed invisible points as well, 26.9, now 22.7; both scales together 300.7 -> 282.1 us.  A CTA of 4,096,
// 2,048, 1,024 or 512 voxels: both scales of four nuScenes-shaped frames 274.8, 269.7, 268.7, 270.2 us (more CTAs in flight, more
// tickets), of two KITTI-shaped frames 50.2, 45.7, 44.6, 44.7.
constexpr int kScanRows = 4, kScanVoxels = kThreads * kScanRows;

__global__ void __launch_bounds__(kThreads) vif_scan_kernel(const __grid_constant__ VifArgs a) {
    __shared__ int wsum[kThreads / 32];
    __shared__ long long s_base;
    const int M = voxels_in_use(a);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if ((long long)blockIdx.x * kScanVoxels >= M) return;
    const int m0 = blockIdx.x * kScanVoxels + warp * (32 * kScanRows) + lane;
    // Sums saturate at one more than the points of the call (at most 2^24 + 1): they cannot wrap, and
    // counts[] that add up to more than the points are still seen as such.
    const int limit = (int)min(a.total, (long long)1 << 24) + 1;
    int n[kScanRows];
#pragma unroll
    for (int j = 0; j < kScanRows; ++j) n[j] = m0 + 32 * j < M ? min(max(a.counts[m0 + 32 * j], 0), limit) : 0;
    int carry = 0;
#pragma unroll
    for (int j = 0; j < kScanRows; ++j) {                 // n[j]: slots of the warp's voxels before this one
        int inc = n[j];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
            if (lane >= d) inc += y;                      // 32 terms of at most 2^24 + 1
        }
        n[j] = carry + inc - n[j];
        carry = min(carry + __shfl_sync(0xFFFFFFFFu, inc, 31), limit);
    }
    if (lane == 0) wsum[warp] = carry;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        if (w < warp) before += wsum[w];
        all += wsum[w];
    }
    if (t == 0) s_base = (long long)atomicAdd(a.taken, (unsigned long long)all);
    __syncthreads();
    const long long base = s_base + before;               // exact whenever the counts are consistent
#pragma unroll
    for (int j = 0; j < kScanRows; ++j) {
        if (m0 + 32 * j >= M) break;
        const int at = (int)min(base + n[j], (long long)limit);
        a.start[m0 + 32 * j] = at;
        a.cursor[m0 + 32 * j] = at;
    }
    release_successor();
}

__global__ void __launch_bounds__(kThreads) vif_fill_kernel(const __grid_constant__ VifArgs a) {
    await_predecessor();
    // counts[] that add up to more than the points of the call are not the voxelizer's counts for this
    // batch: the lists would not fit the list array, so nothing is listed and the next kernel does nothing.
    const bool bad = *a.taken > (unsigned long long)a.total;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *a.bad = bad ? 1 : 0;
        if (bad) atomicOr(a.status, 4);
    }
    if (bad) return;
    const int M = voxels_in_use(a);
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < a.total; i += (long long)gridDim.x * kThreads) {
        const int m = a.pv[i];
        if (m < 0 || m >= M) continue;
        // What goes into the list first (its loads do not wait for the ticket), then the ticket.
        uint4 rec = make_uint4(kZeroRow, 0u, 0u, 0u);
        if (a.vis) {
            if (!a.vis[i]) continue;
        } else {                                        // rows will be blended from the maps: keep the taps
            // pooled: the record addresses a TEXEL of the pooled map (not a float4 of a row), see pooled_column
            rec = a.pool > 1 ? tap_record((int)(i / a.N), (int)a.cam[i], a.uvd[3 * i], a.uvd[3 * i + 1], a.K, a.Hp, a.Wp, 1,
                                          a.inv_stride, a.offset)
                             : tap_record((int)(i / a.N), (int)a.cam[i], a.uvd[3 * i], a.uvd[3 * i + 1], a.K, a.Hf, a.Wf,
                                          a.cf4, a.inv_stride, a.offset);
            if (rec.x == kZeroRow) continue;
        }
        const int pos = atomicAdd(&a.cursor[m], 1);
        // Inside the list whenever counts[] are the kept-point counts of pv[] (the voxelizer's outputs
        // for this batch); anything else must not index out of range.
        if ((unsigned)pos >= (unsigned)a.total) continue;
        if (a.vis) a.list[pos] = (int)i;
        else a.recs[pos] = rec;
    }
    release_successor();
}

// CF4 > 0: Cf/4 known at compile time, blockDim.x == 16 * CF4.  CF4 == 0: any Cf, 256 threads.
template <int CF4>
__global__ void __launch_bounds__(CF4 > 0 ? 16 * CF4 : kThreads) vif_mean_kernel(VifArgs a) {
    await_predecessor();
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.taken = 0ull;     // for the next call; nothing reads it any more
    if (*a.bad) return;
    const int M = voxels_in_use(a);
    const int cf4 = CF4 > 0 ? CF4 : a.cf4;
    const int rows = (int)blockDim.x / cf4;                  // voxels a CTA handles at a time
    const int r = (int)threadIdx.x / cf4, c = (int)threadIdx.x - r * cf4;
    if (r >= rows) return;
    // Two voxels per thread and round: their loads (list start and length, first list entry, first
    // row) do not depend on one another and are in flight together.
    const int stride = gridDim.x * rows;
    for (int m0 = blockIdx.x * rows + r; m0 < M; m0 += 2 * stride) {
        int mm[2] = {m0, m0 + stride}, s0[2], n[2], first[2], seen[2] = {0, 0};
        float4 acc[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const bool ok = mm[u] < M;
            s0[u] = ok ? a.start[mm[u]] : 0;
            n[u] = ok ? min(a.counts[mm[u]], a.cursor[mm[u]] - s0[u]) : 0;   // never past what this call appended
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) first[u] = n[u] > 0 ? a.list[s0[u]] : -1;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (first[u] >= 0) {
                acc[u] = __ldcs(a.gathered + (size_t)first[u] * cf4 + c);
                seen[u] = 1;
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            for (int k = 1; k < n[u]; k += 4) {            // four entries in flight; summed in list order
                int idx[4];
                float4 v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) idx[j] = k + j < n[u] ? a.list[s0[u] + k + j] : -1;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (idx[j] >= 0) v[j] = __ldcs(a.gathered + (size_t)idx[j] * cf4 + c);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (idx[j] < 0) continue;
                    acc[u].x += v[j].x; acc[u].y += v[j].y; acc[u].z += v[j].z; acc[u].w += v[j].w;
                    seen[u] += 1;
                }
            }
            if (mm[u] >= M) continue;
            if (seen[u] > 1) {
                const float inv = 1.0f / (float)seen[u];
                acc[u].x *= inv; acc[u].y *= inv; acc[u].z *= inv; acc[u].w *= inv;
            }
            __stcs(a.vox_img + (size_t)mm[u] * cf4 + c, acc[u]);
            if (c == 0) a.vox_cnt[mm[u]] = seen[u];
        }
    }
    release_successor();
}

// Mean of the p x p window of map texels that pooled texel (ty, tx) of map `map` stands for, column c:
// the same sum, in the same order, as pool_features_kernel (rows outer, columns inner, one multiply by
// the reciprocal of the texel count), so the value is the pooled map's, bit for bit.
template <int PW>
__device__ __forceinline__ float4 window_mean(const VifArgs& a, uint32_t map, int ty, int tx, int c, int cf4) {
    const int p = PW > 0 ? PW : a.pool;
    const int j0 = ty * p, j1 = min(a.Hf, j0 + p), i0 = tx * p, i1 = min(a.Wf, i0 + p);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    auto add = [&](const float4& v) { s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w; };
    const float4* row = a.feat + (((size_t)map * a.Hf + j0) * a.Wf + i0) * cf4 + c;
    const uint32_t step = (uint32_t)a.Wf * (uint32_t)cf4;
    if (PW > 0) {
#pragma unroll
        for (int j = 0; j < PW; ++j)
#pragma unroll
            for (int x = 0; x < PW; ++x)
                if (j < j1 - j0 && x < i1 - i0) add(__ldg(row + (uint32_t)j * step + (uint32_t)x * (uint32_t)cf4));
    } else {
        for (int j = j0; j < j1; ++j, row += step) {
            const float4* at = row;
#pragma unroll 4
            for (int x = i0; x < i1; ++x, at += cf4) add(__ldg(at));
        }
    }
    const float inv = 1.0f / (float)((j1 - j0) * (i1 - i0));
    return make_float4(s.x * inv, s.y * inv, s.z * inv, s.w * inv);
}

// gather_column on the pooled map that is never materialised: the four taps are window means.
template <int PW>
__device__ __forceinline__ float4 pooled_column(const VifArgs& a, const uint4& rec, int c, int cf4) {
    if (rec.x == kZeroRow) return make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t t = rec.x;
    const int x0 = (int)(t % (uint32_t)a.Wp);
    t /= (uint32_t)a.Wp;
    const int y0 = (int)(t % (uint32_t)a.Hp);
    const uint32_t map = t / (uint32_t)a.Hp;
    const int x1 = x0 + (int)(rec.y & 1u), y1 = y0 + (int)((rec.y >> 1) & 1u);
    const float4 f00 = window_mean<PW>(a, map, y0, x0, c, cf4);
    const float4 f01 = x1 != x0 ? window_mean<PW>(a, map, y0, x1, c, cf4) : f00;
    const float4 f10 = y1 != y0 ? window_mean<PW>(a, map, y1, x0, c, cf4) : f00;
    const float4 f11 = y1 != y0 ? (x1 != x0 ? window_mean<PW>(a, map, y1, x1, c, cf4) : f10) : f01;
    return blend(f00, f01, f10, f11, __uint_as_float(rec.z), __uint_as_float(rec.w));
}

// vif_mean without the per-point rows: every listed point's row is blended from its four taps of
// the feature maps here (the blend of the gather stage, from the point's pixel and camera), so the
// [points, Cf] buffer is neither written nor read.  Same thread layout as vif_mean.
// A voxel's start and length, its first record and its taps are three loads that wait for one another.  They are taken in
// three rounds: while the taps of one voxel are in flight, the first record of the thread's next voxel and the start and
// length of the one after it are.  Two voxels at once without that took 283.3 us for both scales of four nuScenes-shaped
// frames, this 273.5; 12 rows and 40 registers (48 warps instead of 40) 275.0 without, 307.8 with it (it spills); a CTA per
// 16 voxels instead of a fixed grid 382.  Bound by the wait for the taps (12 of 16 cycles between a warp's instructions, at 56 %
// occupancy); no unit is full: L1 52 %, L2 31 %, DRAM 14 %, issue 0.51 (one nuScenes-shaped frame, cold L2).
// kPool != 0: the taps are window means of the unpooled maps (emc2_voxel_image_pooled), 2: of 2 x 2 texels, known at compile
// time, 1: of any window.  Bound by the windows' loads from L1 and L2, which want registers, so one record is taken at a
// time: with two, as above, the compiler held to 64 registers and spilled.  us for both scales with two records and p at
// run time / so: four nuScenes-shaped frames of 120,001 points p = 2 959 / 443, p = 4 1,578 / 1,240, p = 8 4,759 / 3,709;
// one KITTI-shaped frame of 20,000 p = 8 209 / 152.
template <int CF4, int kPool>
__global__ void __launch_bounds__(CF4 > 0 ? 16 * CF4 : kThreads, kPool == 1 ? 3 : 0) vif_sample_kernel(const __grid_constant__ VifArgs a) {
    await_predecessor();
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.taken = 0ull;     // for the next call; nothing reads it any more
    if (*a.bad) return;
    const int M = voxels_in_use(a);
    const int cf4 = CF4 > 0 ? CF4 : a.cf4;
    const int rows = (int)blockDim.x / cf4;
    const int r = (int)threadIdx.x / cf4, c = (int)threadIdx.x - r * cf4;
    if (r >= rows) return;
    const uint32_t row_stride = (uint32_t)a.Wf * cf4;
    const int stride = gridDim.x * rows;
    auto list_of = [&](int m, int& s0, int& n) {
        s0 = n = 0;
        if (m < M) {
            s0 = a.start[m];
            n = max(min(a.counts[m], a.cursor[m] - s0), 0);      // never past what this call appended, none where counts[] is negative
        }
    };
    const uint4 none = make_uint4(kZeroRow, 0u, 0u, 0u);
    int m = blockIdx.x * rows + r, s0, n, s1, n1;
    list_of(m, s0, n);
    list_of(m + stride, s1, n1);
    uint4 rec = n > 0 ? a.recs[s0] : none;
    for (; m < M; m += stride) {
        int s2 = 0, n2 = 0;
        const uint4 rec1 = n1 > 0 ? a.recs[s1] : none;
        list_of(m + 2 * stride, s2, n2);
        float4 acc = kPool != 0 ? pooled_column<kPool == 1 ? 0 : kPool>(a, rec, c, cf4) : gather_column(a.feat, rec, c, (uint32_t)cf4, row_stride);
        if (kPool != 0) {
            for (int k = 1; k < n; ++k) {
                const float4 v = pooled_column<kPool == 1 ? 0 : kPool>(a, a.recs[s0 + k], c, cf4);
                acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
            }
        } else {
            for (int k = 1; k < n; k += 2) {
                const bool two = k + 1 < n;
                const uint4 ra = a.recs[s0 + k], rb = two ? a.recs[s0 + k + 1] : none;
                const float4 v0 = gather_column(a.feat, ra, c, (uint32_t)cf4, row_stride);
                const float4 v1 = gather_column(a.feat, rb, c, (uint32_t)cf4, row_stride);
                acc.x += v0.x; acc.y += v0.y; acc.z += v0.z; acc.w += v0.w;
                if (two) { acc.x += v1.x; acc.y += v1.y; acc.z += v1.z; acc.w += v1.w; }
            }
        }
        if (n > 1) {
            const float inv = 1.0f / (float)n;
            acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
        }
        __stcs(a.vox_img + (size_t)m * cf4 + c, acc);
        if (c == 0) a.vox_cnt[m] = n;
        rec = rec1; s0 = s1; n = n1; s1 = s2; n1 = n2;
    }
    release_successor();
}

}  // namespace

// d_gathered != null: rows are read from it and d_vis_mask says which points count; else rows are
// sampled from d_feat at d_uvd in camera d_cam, and a point counts iff its camera is >= 0.
int launch_voxel_image(emc2_bridge* h, int B, int N, int capacity, const int32_t* d_point_voxel,
                       const int32_t* d_counts, const int32_t* d_num_voxels, const uint8_t* d_vis_mask,
                       const float* d_gathered, const float* d_uvd, const int8_t* d_cam, const float* d_feat,
                       float* d_vox_img, int32_t* d_vox_img_count, cudaStream_t st, int pool) {
    const emc2_config_t& cfg = h->cfg;
    VifArgs a;
    a.pv = d_point_voxel; a.counts = d_counts; a.num_voxels = d_num_voxels; a.vis = d_vis_mask;
    a.gathered = reinterpret_cast<const float4*>(d_gathered);
    a.cam = d_cam; a.uvd = d_uvd; a.feat = reinterpret_cast<const float4*>(d_feat);
    a.N = N; a.K = cfg.num_cameras; a.Hf = cfg.feat_h; a.Wf = cfg.feat_w;
    a.inv_stride = 1.0f / (float)cfg.feat_stride; a.offset = cfg.feat_offset;
    a.pool = pool; a.Hp = cfg.feat_h; a.Wp = cfg.feat_w;
    if (pool > 1) {
        // The pooled map: texel J sits at the centre of its window, (J p + (p - 1) / 2) texels of stride s in.
        a.Hp = (cfg.feat_h + pool - 1) / pool; a.Wp = (cfg.feat_w + pool - 1) / pool;
        a.inv_stride = 1.0f / ((float)cfg.feat_stride * (float)pool);
        a.offset = cfg.feat_offset + 0.5f * (float)(pool - 1) * (float)cfg.feat_stride;
    }
    a.vox_img = reinterpret_cast<float4*>(d_vox_img); a.vox_cnt = d_vox_img_count;
    a.start = h->d_vif_start; a.cursor = h->d_vif_cursor; a.list = h->d_vif_list;
    a.recs = h->d_vif_recs;
    a.taken = reinterpret_cast<unsigned long long*>(h->d_vif_part);
    a.bad = h->d_vif_part + 2;
    a.status = h->d_status;
    a.total = (long long)B * N;
    a.capacity = (int)min((long long)capacity, a.total);   // a voxel holds at least one point
    a.cf4 = cfg.feat_c / 4;
    if (a.total == 0 || a.capacity == 0) return EMC2_OK;
    if (a.cf4 > kThreads) return EMC2_ERR_INVALID_ARG;      // a feature row must fit one CTA
    {
        LaunchScope ls(h, K_VIF_SCAN, st);
        vif_scan_kernel<<<(a.capacity + kScanVoxels - 1) / kScanVoxels, kThreads, 0, st>>>(a);
    }
    {
        LaunchScope ls(h, K_VIF_FILL, st);
        const int blocks = (int)min((long long)h->num_sms * 16, (a.total + kThreads - 1) / kThreads);
        launch_chained(vif_fill_kernel, blocks, kThreads, 0, st, a);
    }
    const int blocks = (int)min((long long)h->num_sms * 16, ((long long)a.capacity + 15) / 16);
    if (d_gathered) {
        LaunchScope ls(h, K_VIF_MEAN, st);
        switch (a.cf4) {
            case 16: launch_chained(vif_mean_kernel<16>, blocks, 16 * 16, 0, st, a); break;
            case 20: launch_chained(vif_mean_kernel<20>, blocks, 16 * 20, 0, st, a); break;
            default: launch_chained(vif_mean_kernel<0>, blocks, kThreads, 0, st, a); break;
        }
    } else {
        LaunchScope ls(h, K_VIF_SAMPLE, st);
        if (pool > 1) {
            launch_chained(pool == 2 ? vif_sample_kernel<0, 2> : vif_sample_kernel<0, 1>, blocks, kThreads, 0, st, a);
        } else {
            switch (a.cf4) {
                case 16: launch_chained(vif_sample_kernel<16, 0>, blocks, 16 * 16, 0, st, a); break;
                case 20: launch_chained(vif_sample_kernel<20, 0>, blocks, 16 * 20, 0, st, a); break;
                default: launch_chained(vif_sample_kernel<0, 0>, blocks, kThreads, 0, st, a); break;
            }
        }
    }
    return check_cuda(h, cudaGetLastError());
}

}  // namespace emc2
