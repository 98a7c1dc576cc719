// csrc/rules.cuh for the CPU tests: its functions behind a C interface.
#include "rules.cuh"

using namespace emc2;

struct Axes {
    float mn[3], vs[3], inv[3], margin[3];
    int dims[3];
};

extern "C" {

uint32_t clamp(uint32_t n) { return clamp_points(n); }
int fits(uint64_t first, uint32_t cells, uint32_t points, uint32_t max_ovf, uint32_t max_list) {
    return over_fits(first, cells, points, max_ovf, max_list);
}
int64_t tile_frames(int64_t B, int64_t N) { return frames_of_tile(B, N); }
uint32_t first_word(uint32_t b, uint32_t cells, uint32_t per) { return frame_first_word(b, cells, per); }
uint32_t words_of_frame(uint32_t b, uint32_t cells, uint32_t per) { return frame_words(b, cells, per); }
uint32_t most_words(uint32_t cells, uint32_t per) { return most_frame_words(cells, per); }
uint32_t four_bits(uint32_t bytes) { return bits_of_bytes(bytes); }
int notes(uint64_t bytes, uint64_t words, int B, int N) { return keeps_notes(bytes, words, B, N); }
int frame_notes(uint64_t bytes, uint64_t words, int B, int N) { return keeps_frame_notes(bytes, words, B, N); }
int frames_log(uint64_t bytes, int B) { return frames_side_by_side(bytes, B); }
int frames_in_group(uint64_t bytes, int B) { return frames_per_group(bytes, B); }
int rows_aside(uint64_t points, uint64_t feat_c, int both) { return rows_on_other_stream(points, feat_c, both != 0); }
int rows_stay(uint64_t points, uint64_t feat_c) { return rows_stay_in_l2(points, feat_c); }
uint32_t ranked(uint32_t voxels, uint32_t max_list) { return voxels_ranked(voxels, max_list); }
uint64_t ticket(uint32_t cells, uint32_t points) { return over_ticket(cells, points); }

// Cells of n points (x, y, z), -1 -1 -1 outside the grid; returns for how many of them no divide was needed.
int cells(const float* pts, int n, const float* mn, const float* vs, const int* dims, int* out) {
    Axes g;
    for (int k = 0; k < 3; ++k) {
        g.mn[k] = mn[k]; g.vs[k] = vs[k]; g.dims[k] = dims[k];
        g.inv[k] = axis_inverse(vs[k]);
        g.margin[k] = axis_margin(dims[k]);
    }
    int sure = 0;
    for (int i = 0; i < n; ++i) {
        int c[3];
        uint32_t by_product[3];
        const bool in = cell_xyz(g, pts[3 * i], pts[3 * i + 1], pts[3 * i + 2], c[0], c[1], c[2]);
        for (int k = 0; k < 3; ++k) out[3 * i + k] = in ? c[k] : -1;
        sure += cell_by_product(g, pts + 3 * i, by_product);
    }
    return sure;
}

}  // extern "C"
