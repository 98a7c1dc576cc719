// Arithmetic that decides indices.  It runs in the kernels and compiles for the host as well, so that the CPU tests
// exercise these lines and not a copy of them.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define EMC2_RULE __host__ __device__ __forceinline__
#else
#define EMC2_RULE inline
#endif

namespace emc2 {

// ---- voxels found by the rank scan: at most one per point of a call, or the store was not all zero when it began
EMC2_RULE bool voxels_possible(uint32_t voxels, uint32_t max_list) { return voxels <= max_list; }

// The scan covers whole tiles, which can reach past the call's last frame; a cell found there was left over as well,
// and the caller's BEV image has no such frame.
EMC2_RULE bool frame_in_call(uint32_t frame, uint32_t frames) { return frame < frames; }

// ---- cells over the per-voxel cap (rank scan of a table store)
// A tile sums the points of its cells over the cap and takes one 64-bit ticket for them, {cells, points} before the
// tile.  In a store that was not all zero a word can hold anything, and a sum that wrapped would pass for a small
// one: every term and every partial sum of a tile is clamped to kPointsClamp, which is above the points of any call
// (2^24), so that 2,048 cells summed by threads of 8, warps of 32 and 8 warps stay below 2^31.
constexpr uint32_t kPointsClamp = 1u << 25;

EMC2_RULE uint32_t clamp_points(uint32_t n) { return n < kPointsClamp ? n : kPointsClamp; }

// Whether a tile with `cells` cells over the cap and `points` points in them, which took the ticket `first`, finds
// room: the tile's index lists then lie inside [0, max_list) and its cells' places inside [0, max_ovf).  No ticket may
// be taken with points > max_list.  The first ticket that does not fit is always found, because nothing has wrapped
// before it.
EMC2_RULE bool over_fits(uint64_t first, uint32_t cells, uint32_t points, uint32_t max_ovf, uint32_t max_list) {
    const uint32_t j = (uint32_t)(first >> 32), off = (uint32_t)first;
    return cells <= max_ovf && points <= max_list && j <= max_ovf - cells && off <= max_list - points;
}

EMC2_RULE uint64_t over_ticket(uint32_t cells, uint32_t points) { return (uint64_t)cells << 32 | points; }

}  // namespace emc2
