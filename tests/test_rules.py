"""The index arithmetic of csrc/rules.cuh, compiled for the host (CPU)."""
import os
import re

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_04123_b200", "csrc")


def test_point_sums_of_a_tile_never_wrap_and_never_pass_for_small_ones(rules):
    """2,048 words of a tile, summed as the rank scan does (8 per thread, 32 threads per warp, 8 warps), whatever they hold."""
    rng = np.random.default_rng(0)
    words = np.array([33, 1 << 24, (1 << 24) + 1, 0x80000000, 0x80000001, 0x80000005, 0xFFFFFFFF], np.uint64)
    for most in (1, 300000, 1 << 24):
        for trial in range(60):
            n = np.full(2048, 33, np.uint64) if trial == 0 else rng.choice(words[: 1 + trial % len(words)], 2048)
            n[rng.random(2048) < rng.random()] = 0
            threads = [sum(rules.clamp(int(v)) for v in t) for t in n.reshape(-1, 8)]
            assert max(threads) < 1 << 31
            warps = [sum(rules.clamp(v) for v in w) for w in np.reshape(threads, (-1, 32)).tolist()]
            assert max(warps) < 1 << 31
            tile = sum(rules.clamp(v) for v in warps)
            assert tile < 1 << 31
            true = int(n.sum())
            assert (tile > most) == (true > most)
            if true <= most:
                assert tile == true


def test_tickets_that_do_not_fit_are_found(rules):
    """A run of tickets is refused from the first one on that leaves the lists, also where 32-bit sums would wrap."""
    rng = np.random.default_rng(1)
    for max_list, max_ovf in ((300000, 9092), (1 << 24, 508401), (1, 2), (96, 4)):
        for _ in range(200):
            counter, cells, points, refused = 0, 0, 0, False
            for _ in range(60):
                c = int(rng.integers(1, 2049))
                p = int(rng.choice([c, min(33 * c, max_list), max_list, int(rng.integers(0, max_list + 1))]))
                p = min(p, max_list)
                first = counter
                counter = (counter + rules.ticket(c, p)) % (1 << 64)
                cells, points = cells + c, points + p
                ok = bool(rules.fits(first, c, p, max_ovf, max_list))
                if not refused:
                    assert ok == (cells <= max_ovf and points <= max_list)
                refused = refused or not ok
                if ok:                                      # in bounds whatever came before
                    assert (first >> 32) + c <= max_ovf and (first & 0xFFFFFFFF) + p <= max_list
            assert refused == (cells > max_ovf or points > max_list)


def test_leftover_words_do_not_make_a_small_sum(rules):
    """Two leftover words {over the cap, place 1} and {over the cap, place 5} add up to 6 in 32 bits."""
    words = [0x80000001, 0x80000005]
    assert sum(words) % (1 << 32) == 6
    assert sum(rules.clamp(w) for w in words) > 1 << 24
    assert not rules.fits(rules.ticket(0, 0x80000001), 1, 0x80000005, 1000, 300000)


def test_a_scale_with_more_voxels_than_points_is_not_ranked():
    """vox_rank leaves such a scale's tiles before it writes a rank, a list entry or one of the caller's counts."""
    text = open(os.path.join(CSRC, "voxelize.cu")).read()
    body = text[text.index("vox_rank_kernel("):text.index("pass 3: accumulate")]
    loop = body[body.index("k < listed"):]
    guard = loop.index("if (!voxels_possible(sc ? all[1] : all[0], g.max_list)) continue;")
    for write in ("a.counts[sc][m] =", "g.cell_list[m] =", "at[0] =", "atomicAdd("):
        assert guard < loop.index(write), write


def test_a_scale_that_is_not_ranked_leaves_the_callers_counts_alone(rules):
    """It has no rows: vox_rank clears no counts for it and vox_accum, which counts there for some scales, adds none."""
    for most in (0, 1, 5, 1 << 24):
        for n in {0, 1, most, most + 1, 1 << 25, 0xFFFFFFFF}:
            assert rules.ranked(n, most) == (n if n <= most else 0)
    text = open(os.path.join(CSRC, "voxelize.cu")).read()
    rank = text[text.index("vox_rank_kernel("):text.index("pass 3: accumulate")]
    clear = rank.index("a.counts[v][i] = 0")
    assert "const uint32_t voxels = voxels_ranked(all[v], g.max_list);" in rank[:clear]
    assert "i < min(voxels, (uint32_t)a.capacity[v])" in rank[clear - 120:clear]
    assert "g.totals[0] = (int)voxels_ranked(n, g.max_list);" in rank
    accum = text[text.index("vox_accum_kernel("):text.index("per-voxel cap on a bitmap scale")]
    assert accum.count("a.counts[sc]") == 1 and "if (at.m < s.totals[0]) atomicAdd(a.counts[sc] + at.m, 1);" in accum


def test_the_bev_image_is_written_for_frames_of_the_call_only():
    """A pillar scan's tiles cover cells of frames past the call's last one: every write into the image tests the frame."""
    text = open(os.path.join(CSRC, "voxelize.cu")).read()
    code = text[text.index("vox_accum_kernel("):text.index("int run_voxelize")]
    spots = [m.start() for m in re.finditer(r"a\.bev\[|dst = a\.bev \+", code)]
    assert len(spots) == 2
    for at in spots:
        assert "frame_in_call(r, a.frames)" in code[at - 300:at]


def test_frames_of_a_tile(rules):
    """256 consecutive points from any multiple of 256 on lie in no more frames than the rule says, and the rule is met."""
    for N in list(range(1, 300)) + [511, 512, 513, 1000]:
        for B in (1, 2, 3, 4, 7, 31, 32):
            total = B * N
            spans = [(min(g + 255, total - 1) // N) - g // N + 1 for g in range(0, total, 256)]
            most = rules.tile_frames(B, N)
            assert max(spans) <= most <= B
            if most > 2:
                assert N < 255
    assert rules.tile_frames(32, 1) == 32 and rules.tile_frames(32, 255) == 2 and rules.tile_frames(32, 254) == 3


def test_noted_tiles_of_a_frame_have_a_place(rules):
    """Every tile of a frame lies in the words the rule gives, frames that share a word included, and no frame has more."""
    for per in (49152, 2048):
        for cells in (1, 47, 2048, 49152, 49153, 220000, 262144, 1 << 20, 74_638_240, 90_112_000):
            most = rules.most_words(cells, per)
            for b in range(0, min(32, (1 << 32) // cells)):
                first, n = rules.first_word(b, cells, per), rules.words_of_frame(b, cells, per)
                assert first == b * cells // per // 32 and first + n - 1 == ((b + 1) * cells - 1) // per // 32
                assert 1 <= n <= most


def test_four_bytes_become_four_bits(rules):
    for v in range(16):
        assert rules.four_bits(sum((v >> k & 1) << (8 * k) for k in range(4))) == v


def test_calls_that_keep_notes(rules):
    kitti, nuscenes = 15_018_656 + 880_000, 12_439_696 + 1_048_576
    for frame, words in ((kitti, 64), (nuscenes, 55)):
        assert not rules.notes(frame, words, 1, 1000)
        assert rules.notes(frame, words, 2, 1) and rules.notes(frame, words, 32, 1 << 17)
        assert not rules.notes(frame, words, 32, (1 << 17) + 1) and not rules.notes(frame, 73, 32, 1000)


def test_frames_that_keep_notes(rules):
    """By points per frame, which the copies of the notes share: the limit that calls have."""
    kitti, nuscenes = 15_018_656 + 880_000, 12_439_696 + 1_048_576
    for frame, words in ((kitti, 64), (nuscenes, 55)):
        assert rules.frame_notes(frame, words, 2, 1) and rules.frame_notes(frame, words, 2, 1 << 20)
        assert not rules.frame_notes(frame, words, 2, (1 << 20) + 1) and not rules.frame_notes(frame, words, 1, 1000)
        assert not rules.frame_notes(frame, 73, 2, 1000)
    text = open(os.path.join(CSRC, "bridge_internal.cuh")).read()
    body = text[text.index("inline bool keeps_tile_marks("):text.index("inline TileMarks tile_marks(")]
    assert "return keeps_frame_notes(store_bytes(h), words, B, N);" in body


def test_frames_side_by_side(rules):
    """Groups are as large as the frames need or 64 MB of stores allow, and their CTAs take every tile of every frame once."""
    for frame in (0, 1, 13_488_272, 15_898_656, 32 << 20, (32 << 20) + 1, 64 << 20, 65 << 20, 700 << 20):
        for B in (1, 2, 3, 4, 5, 7, 8, 9, 31, 32):
            log = rules.frames_log(frame, B)
            G = 1 << log
            assert G == 1 or (G * frame <= 64 << 20 and G < 2 * B)
            assert G >= B or 2 * G * frame > 64 << 20
            groups = (B + G - 1) >> log
            taken = [((y << log) + (x & (G - 1)), x >> log) for y in range(groups) for x in range(3 << log)]
            assert sorted(t for t in taken if t[0] < B) == [(b, i) for b in range(B) for i in range(3)]


def test_groups_of_frames_are_as_large_as_the_batch_needs(rules):
    """No more groups than the power of two takes, fewer places without a frame than there are groups, every tile taken once."""
    for frame in (0, 1, 13_488_272, 15_898_656, 32 << 20, (32 << 20) + 1, 700 << 20):
        for B in range(0, 33):
            most, G = 1 << rules.frames_log(frame, B), rules.frames_in_group(frame, B)
            groups = -(-B // G)
            assert 1 <= G <= most and groups == -(-B // most) and (B == 0 or 0 <= groups * G - B < groups)
            taken = [(y * G + x % G, x // G) for y in range(groups) for x in range(3 * G)]
            assert sorted(t for t in taken if t[0] < B) == [(b, i) for b in range(B) for i in range(3)]
    assert rules.frames_in_group(15_898_656, 9) == 3 and rules.frames_in_group(15_898_656, 5) == 3


def test_gathered_rows_that_stay_in_l2(rules):
    for points, feat_c, stays in ((120000, 256, 1), (131072, 256, 1), (131073, 256, 0), (419430, 80, 1), (419431, 80, 0), (1, 4, 1),
                                  (1 << 24, 1020, 0)):
        assert rules.rows_stay(points, feat_c) == stays


def test_calls_whose_rows_go_to_the_other_stream(rules):
    """Either side of the limits: points, bytes of rows, and few points with wide rows."""
    for both, most_bytes, per_channel in ((1, 160_000_000, 450), (0, 96_000_000, 300)):
        width = 8 if both else 4
        for cf in (4, 64, 80, 96, 124, 128, 132, 192, 256, 512, 1024):
            least = cf * per_channel if cf >= 128 else 0
            most = min(320_000, most_bytes // (cf * width))
            for n in {1, least - 1, least, least + 1, most, most + 1, 1 << 24}:
                if n > 0:
                    assert rules.rows_aside(n, cf, both) == (least <= n <= most), (n, cf, both)
    assert rules.rows_aside(120_000, 64, 1) and rules.rows_aside(120_000, 64, 0) and rules.rows_aside(99_999, 128, 1)
    assert not rules.rows_aside(8_000, 512, 1) and not rules.rows_aside(8_000, 512, 0) and not rules.rows_aside(30_000, 256, 1)
