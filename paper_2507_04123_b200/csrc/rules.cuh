// Arithmetic that decides indices.  It runs in the kernels and compiles for the host as well, so that the CPU tests
// exercise these lines and not a copy of them.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define EMC2_RULE __host__ __device__ __forceinline__
#else
#define EMC2_RULE inline
#endif

namespace emc2 {

// ---- fp32 operations with one rounding each, never contracted (host: built without contraction)
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float sub1(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float add1(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float mul1(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float div1(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ uint32_t bits_of(float a) { return __float_as_uint(a); }
#else
inline float sub1(float a, float b) { return a - b; }
inline float add1(float a, float b) { return a + b; }
inline float mul1(float a, float b) { return a * b; }
inline float div1(float a, float b) { return a / b; }
inline uint32_t bits_of(float a) { uint32_t u; std::memcpy(&u, &a, sizeof u); return u; }
#endif

// ---- cell of a point
// Cell index along one axis: one fp32 subtract, one IEEE fp32 divide, floor.  -1 if outside.
EMC2_RULE int axis_cell(float p, float mn, float vs, int dim) {
    const float f = floorf(div1(sub1(p, mn), vs));
    // NaN fails both comparisons; +-inf fails one of them.
    if (!(f >= 0.0f) || !(f < (float)dim)) return -1;
    return (int)f;
}

// 1 / vs in fp32 (NaN where that is not a normal number) and how far from an integer a product with it decides the
// cell without a divide, see cell_by_product.
inline float axis_inverse(float vs) {
    const float inv = 1.0f / vs;
    return std::isnormal(inv) ? inv : NAN;
}
inline float axis_margin(int dim) { return 4e-7f * (float)(dim + 2); }

// The cell along all three axes by a multiplication each; true where that provably decides it.  G has the arrays mn,
// vs, inv, margin and dims of the axes.  A divide is a subroutine of some twenty instructions and every point needs six, in two kernels, so it is
// only executed where it can matter.  q = d * RN(1 / vs) and RN(d / vs) differ by at most 3 * 2^-24 of their
// value (one rounding each of the reciprocal, the product and the quotient): unless q lies within
// `margin` = 4e-7 * (cells of the axis + 2) of an integer, both have the same floor, or both are outside.
// Adding 1.5 * 2^23 leaves the nearest integer in the low bits of the sum (values too large for that come out
// as no index of the axis, or exactly on an integer); zero, tiny and non-finite values fail the test of the
// margin.  The bits are subtracted modulo 2^32: those of a negative sum come out as no index of the axis.
template <class G>
EMC2_RULE bool cell_by_product(const G& g, const float p[3], uint32_t c[3]) {
    constexpr float kMagic = 12582912.0f;
    bool sure = true;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k) {
        const float q = mul1(sub1(p[k], g.mn[k]), g.inv[k]);
        const float t = add1(q, kMagic);
        const float e = sub1(q, sub1(t, kMagic));                 // q minus the nearest integer
        sure &= fabsf(e) > g.margin[k];
        c[k] = bits_of(t) - bits_of(kMagic) - (bits_of(e) >> 31);
    }
    return sure;
}

// Cell of a point as by subtract, divide, floor; true if inside the grid.
template <class G>
EMC2_RULE bool cell_xyz(const G& g, float x, float y, float z, int& ix, int& iy, int& iz) {
    const float p[3] = {x, y, z};
    uint32_t c[3];
    if (!cell_by_product(g, p, c)) {
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int k = 0; k < 3; ++k) c[k] = (uint32_t)axis_cell(p[k], g.mn[k], g.vs[k], g.dims[k]);
    }
    ix = (int)c[0]; iy = (int)c[1]; iz = (int)c[2];
    return (c[0] < (uint32_t)g.dims[0]) & (c[1] < (uint32_t)g.dims[1]) & (c[2] < (uint32_t)g.dims[2]);
}

// ---- frames that kTile = 256 consecutive points of a batch of B frames of N can belong to, at most
inline long long frames_of_tile(long long B, long long N) {
    const long long most = (256 - 2) / N + 2;      // a last point of one frame, then whole frames
    return B < most ? B : most;
}

// ---- which branch of a call of all stages stays on the caller's stream
// Stage 1 is a chain of four kernels.  In a small call it is the longer branch and waiting for another stream, at its begin
// and at the end of the call, costs more than it can hide: the rows go to the other stream instead.  In a large call the
// rows are the longer branch, and stage 1, which shares the chip with them, needs its stream's priority.  So they are where
// few points have wide rows: a CTA takes the rows of 256 points in a time that grows with the channels, however few CTAs
// there are.  us per call, rows on the caller's stream / stage 1 on it, both outputs of the rows unless said otherwise;
// 80 channels are nuScenes-shaped frames, other widths KITTI-shaped ones unless they have six cameras:
//   one frame of 120,000 points, 64 channels 44.6 / 37.4, dispatched rows only 38.9 / 32.4; 3 x 33,333 x 80 channels 58.4 /
//   53.9; 8 x 16,384 x 80 95.0 / 91.6.
//   Bytes: one of 240,000 x 80 (154 MB) 84.0 / 81.0, of 300,000 x 64 (154 MB) 67.8 / 65.7 or, dense, 68.3 / 69.9; 4 x 100,000
//   x 64 (205 MB) 98.9 / 104.7.  Dispatched rows only: one of 300,000 x 80 (96 MB) 83.7 / 80.3, of 480,000 x 64 (123 MB)
//   72.8 / 75.0.
//   Points: one of 300,000 x 64, dispatched rows only, 57.8 / 53.8, of 340,000 60.1 / 58.7, of 400,000 65.3 / 65.4; both
//   rows of several frames cross earlier, 4 x 40,000 x 64 61.8 / 60.0, 4 x 78,000 85.0 / 87.2, but within 3 % either way.
//   Wide rows: one of 45,000 x 128 33.2 / 35.5, of 60,000 35.0 / 36.5 (six cameras: 46.0 / 41.0), of 120,000 55.4 / 51.0; of
//   60,000 x 192 42.5 / 45.2, of 90,000 50.4 / 51.5 (six cameras: 61.3 / 60.0); of 30,000 x 256 46.0 / 50.3, of 8,000 x 512
//   41.3 / 75.  Dispatched rows only: of 30,000 x 192 30 / 34.2, of 60,000 34.0 / 35.2, of 90,000 41.4 / 37.8.
inline bool rows_on_other_stream(uint64_t points, uint64_t feat_c, bool both_rows) {
    if (feat_c >= 128 && points < feat_c * (both_rows ? 450u : 300u)) return false;
    return points <= 320000 && points * feat_c * (both_rows ? 8u : 4u) <= (both_rows ? 160000000u : 96000000u);
}

// ---- whether the gathered rows of a call stay in L2 (126 MB) until the dispatch reads them: measured at 123 and 154 MB, see
// project_gather_kernel
inline bool rows_stay_in_l2(uint64_t points, uint64_t feat_c) { return points * feat_c * 4u <= (uint64_t)128 << 20; }

// ---- notes of the tiles of a store that the marking pass touched: a bit per tile, 32 tiles to a word
// Words that hold the tiles of frame b, for frames of `cells` cells and tiles of `per_tile` cells: the first, how many, and
// at most how many of any frame.
EMC2_RULE uint32_t frame_first_word(uint32_t b, uint32_t cells, uint32_t per_tile) { return b * cells / per_tile / 32u; }
EMC2_RULE uint32_t frame_words(uint32_t b, uint32_t cells, uint32_t per_tile) {
    return (b * cells + (cells - 1u)) / per_tile / 32u - frame_first_word(b, cells, per_tile) + 1u;
}
inline uint32_t most_frame_words(uint32_t cells, uint32_t per_tile) { return cells / per_tile / 32u + 2u; }

// Whether the marking pass of a call keeps the notes: frames of which N points note in the same copy and whose stores take
// `frame_bytes` each (8 KB tiles, `words` words of notes).  The counting pass then reads the noted tiles instead of the whole
// stores, three quarters of which are empty space.  One frame's stores are read as fast as the notes come back (voxels and
// rulebooks of 30,000 points 56 and 57 us).  The more points note in one copy the longer the queues at its words: with a single
// copy notes lost from about 2^17 points on.  The 72 words hold the frames of both grid families (64 and 55 words); larger grids,
// which would need more shared memory, have not been measured with notes.
constexpr uint32_t kMarkWords = 72;
inline bool keeps_notes(uint64_t frame_bytes, uint64_t words, int B, int N) {
    return words <= kMarkWords && B * frame_bytes >= (uint64_t)24 << 20 && N <= 1 << 17;
}

// The notes are kept in this many copies, and a CTA sends its own to one of them: reductions on one word are served one after another,
// and every CTA has some for the few words of the ground plane.  us for 1, 4, 8 and 16 copies: eight KITTI-shaped frames
// 42.4, 33.8, 33.4, 33.1 (project_route; 32.1 without notes), the call 202.4, 194.3, 193.6, 193.8; vox_mark 36.5, 28.0, 27.6,
// 27.2.  Reading a word first, to send only what is new, adds to the same queue: 52.8 with one copy.
constexpr uint32_t kNoteCopies = 8;

// The same for frames of N points, which are spread over the copies: up to 2^20 points.  us per call without / with the notes:
//   voxel lists: four KITTI-shaped frames of 300,000 points 88.6 / 82.5, of 700,000 186 / 183, of 1,000,000 236 / 232; eight of
//   850,000 in firing order 421 / 410; four nuScenes-shaped ones of 300,000 127 / 121.5, of 1,000,000 381 / 376.
//   all stages, where the notes are taken by the projection: four KITTI-shaped frames of 300,000 points 207 / 200, of 524,288 334.6 /
//   332, of 700,000 441 / 441, of 850,000 525 / 528, of 1,000,000 460 / 464 (32 channels); four nuScenes-shaped ones of 300,000 257 /
//   251.5, of 700,000 551 / 551, of 850,000 665 / 670.
// So they lose up to 1 % of the calls of all stages from about 700,000 points on and gain 1 to 2 % of the voxel lists there.  Larger
// frames have not been measured.
inline bool keeps_frame_notes(uint64_t frame_bytes, uint64_t words, int B, int N) {
    return keeps_notes(frame_bytes, words, B, (N + (int)kNoteCopies - 1) / (int)kNoteCopies);
}

// ---- which tile of which frame a CTA of a marking pass takes: groups of frames, whose tiles take turns
// Marks that land in one sector of a store are served one after another, and the sector of pillars next to the sensor gets about
// a thousand of a nuScenes-shaped frame's 300,000 points.  With the frames side by side those marks are spread over the whole
// kernel.  The stores of a group should fit in L2 together: four nuScenes-shaped frames with groups of 32, 64, 128 and 256 MB
// took project_route 38.7, 37.2, 37.2 and 37.3 us, 32 KITTI-shaped ones of 262,144 points and six cameras 198, 198, 201 and 205,
// all 32 side by side 222.  us, frame after frame / groups of at most 64 MB: project_route of four nuScenes-shaped frames 44.9 /
// 37.5, their vox_mark 37.7 / 30.1, the call 301.1 / 293.3; of 32 KITTI-shaped frames of 262,144 points 167 / 161, the call 1,329 /
// 1,322, through six cameras 203.9 / 205.5 and 1,746 / 1,744; of eight of 120,000, whose first ring of points is farther away, 33.1 /
// 33.8, the call 189.6 / 189.8; voxel lists of 32 dense frames of 524,288 points 1,178 / 1,114.
// The power of two that fits:
inline int frames_side_by_side(uint64_t frame_bytes, int B) {
    int log = 0;
    while ((1 << log) < B && (frame_bytes << (log + 1)) <= (uint64_t)64 << 20) ++log;
    return log;
}

// Frames per group: as few groups as that allows, all of one size but for the last.  Groups of the power of two itself left CTAs
// without a frame, which cost nine frames in groups of four, twelve places, up to 1.6 % (us): voxel lists of uniform frames of
// 16,384 points 98.9, now 97.3, KITTI-shaped ones of 60,000 77.8, now 77.1, all stages of these 132.2, now 131.4.
inline int frames_per_group(uint64_t frame_bytes, int B) {
    const int most = 1 << frames_side_by_side(frame_bytes, B), groups = (B + most - 1) / most;
    return groups > 0 ? (B + groups - 1) / groups : 1;
}

// Four bytes that are 0 or 1 -> four bits, the lowest byte in the lowest bit.
EMC2_RULE uint32_t bits_of_bytes(uint32_t bytes) { return bytes * 0x01020408u >> 24 & 15u; }

// ---- voxels found by the rank scan: at most one per point of a call, or the store was not all zero when it began
EMC2_RULE bool voxels_possible(uint32_t voxels, uint32_t max_list) { return voxels <= max_list; }

// Rows of such a scale, and the voxels it reports: none where the store was not.
EMC2_RULE uint32_t voxels_ranked(uint32_t voxels, uint32_t max_list) { return voxels_possible(voxels, max_list) ? voxels : 0u; }

// The scan covers whole tiles, which can reach past the call's last frame; a cell found there was left over as well,
// and the caller's BEV image has no such frame.
EMC2_RULE bool frame_in_call(uint32_t frame, uint32_t frames) { return frame < frames; }

// ---- cells over the per-voxel cap (rank scan of a table store)
// A part of a tile sums the points of its cells over the cap and takes one 64-bit ticket for them, {cells, points} before
// the part.  In a store that was not all zero a word can hold anything, and a sum that wrapped would pass for a small
// one: every term and every lane's sum is clamped to kPointsClamp, which is above the points of any call
// (2^24), so that 256 cells summed by lanes of 8 and a warp of 32 stay below 2^31.
constexpr uint32_t kPointsClamp = 1u << 25;

EMC2_RULE uint32_t clamp_points(uint32_t n) { return n < kPointsClamp ? n : kPointsClamp; }

// Whether a part with `cells` cells over the cap and `points` points in them, which took the ticket `first`, finds
// room: its index lists then lie inside [0, max_list) and its cells' places inside [0, max_ovf).  No ticket may
// be taken with points > max_list.  The first ticket that does not fit is always found, because nothing has wrapped
// before it.
EMC2_RULE bool over_fits(uint64_t first, uint32_t cells, uint32_t points, uint32_t max_ovf, uint32_t max_list) {
    const uint32_t j = (uint32_t)(first >> 32), off = (uint32_t)first;
    return cells <= max_ovf && points <= max_list && j <= max_ovf - cells && off <= max_list - points;
}

EMC2_RULE uint64_t over_ticket(uint32_t cells, uint32_t points) { return (uint64_t)cells << 32 | points; }

}  // namespace emc2
