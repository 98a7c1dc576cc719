"""Edges of the voxel cell stores, the cell rule, the visibility test and the row kernels (needs a B200)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import emc2_gen as gen
from emc2_gen.configs import Grid
from parity import close, compare_bridge, np_, to_dev

pytestmark = pytest.mark.gpu

# A store of units of 96 cells, 8 KB tiles of 49,152 cells, groups of 128 tiles; more than 2^24 cells.
BITMAP = Grid(min=(0.0, 0.0, 0.0), voxel=(1.0, 1.0, 1.0), dims=(4099, 4099, 1))
# A store of one word per cell, tiles of 2,048 cells.
TABLE = Grid(min=(0.0, 0.0, 0.0), voxel=(1.0, 1.0, 1.0), dims=(257, 255, 1), max_points=3)


def bridge_for(w):
    import paper_2507_04123_b200 as pkg
    return pkg.Bridge(pkg.config_from_workload(w))


def check_voxels(w, pts, oracle, repeat=2, rules=False):
    br = bridge_for(w)
    d = torch.from_numpy(pts).cuda()
    for _ in range(repeat):                                    # a second call must see clean stores
        vox = br.voxelize(d)
        br.status()
        for s, g in enumerate(w.grids):
            ref = oracle.voxelize(pts, g.min, g.voxel, g.dims, g.max_points)
            M = ref["num_voxels"]
            assert int(vox["num_voxels"][s]) == M
            for k in ("coords", "counts"):
                assert np.array_equal(np_(vox[k][s])[:M], ref[k]), (k, s)
            assert np.array_equal(np_(vox["point_voxel"][s]), ref["point_voxel"]), s
            ok, mx, _ = close(np_(vox["mean"][s])[:M], ref["mean"])
            assert ok, (s, mx)
            if rules:
                out = br.rulebook(vox, s)
                br.status()
                off, rin, rout = oracle.rulebook(ref["coords"])
                assert np.array_equal(np_(out["offsets"]), off)
                assert np.array_equal(np_(out["rule_in"])[:off[27]], rin)
                assert np.array_equal(np_(out["rule_out"])[:off[27]], rout)
    br.close()


def small_images(w, h, wd):
    """The workload with images of h x wd pixels, the cameras' axes in their middle and about 77 degrees wide."""
    cams = tuple(replace(c, fx=0.63 * wd, fy=0.63 * wd, cx=wd / 2, cy=h / 2) for c in w.cameras)
    return replace(w, img_h=h, img_w=wd, feat_stride=8, cameras=cams)


def centres(ids, grid, C, rng):
    ids = np.asarray(ids, np.int64)
    x, y = ids % grid.dims[0], ids // grid.dims[0]
    pts = np.concatenate([np.stack([x + 0.5, y + 0.5, np.full(len(ids), 0.5)], 1), rng.random((len(ids), C - 3))], 1)
    return pts.astype(np.float32)


@pytest.mark.parametrize("C", [4, 5])
@pytest.mark.parametrize("which", ["edges", "full_tile", "last_cells", "one"])
def test_units_tiles_and_groups_of_the_stores(oracle, which, C):
    rng = np.random.default_rng(3)
    tile, cells = 49152, BITMAP.cells
    if which == "edges":                                       # both sides of every unit, sector, tile and group edge
        at = [e + d for e in (0, 32, 64, 96, 192, 6144, tile, 4 * tile, 127 * tile, 128 * tile, 256 * tile, 4099 * 96)
              for d in range(-3, 4)]
    elif which == "full_tile":                                 # every cell of a tile and the rows above and below
        at = list(range(tile - 4200, 2 * tile + 4200))
    elif which == "last_cells":
        at = list(range(cells - 300, cells))
    else:
        at = [cells // 2]
    at = sorted({a for a in at if 0 <= a < cells})
    fine = centres(rng.permutation(np.repeat(at, 2)), BITMAP, C, rng)
    # table cells around tile edges, some of them over their cap of 3
    few = [a for e in (0, 8, 2048, 4 * 2048, TABLE.cells) for a in range(e - 9, e + 9) if 0 <= a < TABLE.cells]
    table = centres(rng.permutation(np.repeat(few, rng.integers(1, 7, len(few)))), TABLE, C, rng)
    pts = rng.permutation(np.concatenate([fine, table]))[None]
    base = gen.KITTI if C == 4 else gen.NUSCENES
    w = replace(base.with_shape(1, pts.shape[1]), grids=(BITMAP, TABLE))
    check_voxels(w, np.ascontiguousarray(pts), oracle, rules=which in ("edges", "last_cells"))


@pytest.mark.parametrize("B", [1, 3])
@pytest.mark.parametrize("share", [1.0, 0.02])
def test_parts_of_the_tiles_of_a_table_store(oracle, B, share):
    """Parts of 32 sectors (256 cells): cells over the cap on both sides of their edges, every part or a few holding voxels."""
    rng = np.random.default_rng(11)
    frames = []
    for _ in range(B):
        few = [a for e in range(0, TABLE.cells, 256) for a in range(e - 2, e + 3) if 0 <= a < TABLE.cells and rng.random() < share]
        few += [0, TABLE.cells - 1]
        frames.append(centres(rng.permutation(np.repeat(few, rng.integers(1, 6, len(few)))), TABLE, 4, rng))
    N = max(map(len, frames))
    pts = np.full((B, N, 4), -1.0, np.float32)                 # padding outside both grids
    for b, f in enumerate(frames):
        pts[b, :len(f)] = f
    fine = Grid(min=(0.0, 0.0, 0.0), voxel=(1.0, 1.0, 1.0), dims=(4099, 4099, 1), max_points=2)      # a cap on a bitmap store
    w = replace(gen.KITTI.with_shape(B, N), grids=(fine, TABLE))
    check_voxels(w, pts, oracle)


@pytest.mark.parametrize("most", [1, 4, 5])
def test_parts_listed_by_sectors_and_by_words(oracle, most):
    """Parts (6,144 cells) whose fullest sector (192 cells) holds as many voxels as one lane lists, or one more: in the first, the
    last or any sector, in one word or at both ends of the sector, the other sectors empty or not."""
    rng = np.random.default_rng(most)
    at = []
    for part in range(24):
        p0 = 6144 * (part if part < 12 else 2700 + part)
        full = (0, 31, int(rng.integers(32)))[part % 3]
        at += [p0 + 192 * full + d for d in ([191 - k for k in range(most)] if part % 2 else [0, 95, 96, 191, 33][:most])]
        if part % 4 > 1:
            at += [p0 + 192 * s + int(rng.integers(192)) for s in range(32) if s != full]
    assert max(at) < BITMAP.cells and np.bincount(np.unique(at) // 192).max() == most
    pts = centres(rng.permutation(np.repeat(np.unique(at), 2)), BITMAP, 4, rng)[None]
    check_voxels(replace(gen.KITTI.with_shape(1, pts.shape[1]), grids=(BITMAP, TABLE)), pts, oracle)


@pytest.mark.parametrize("dims", [(1408, 1600, 40), (61, 7, 3), (2_000_000, 2, 2)])
def test_cells_of_points_on_cell_boundaries(oracle, dims):
    """Points a few ulps around multiples of the cell size, far away, and not finite: cells as by subtract, divide, floor."""
    rng = np.random.default_rng(5)
    for mn, vs in (((0.0, -40.0, -3.0), (0.05, 0.05, 0.1)), ((-51.2, -51.2, -5.0), (0.075, 1.0 / 3.0, 0.2)),
                   ((1e-3, 0.0, 0.0), (4.0, 1e-3, 1e-30)), ((0.0, 0.0, 0.0), (1e-39, 3.0, 1e30))):
        grid = Grid(min=mn, voxel=vs, dims=dims)
        pillars = Grid(min=mn, voxel=vs, dims=(dims[0] % 997 + 1, dims[1], 1))
        n = 4099
        pts = np.zeros((1, n, 4), np.float32)
        for k in range(3):
            lo, size = np.float32(mn[k]), np.float32(vs[k])
            with np.errstate(over="ignore", under="ignore"):
                v = (lo + rng.integers(-2, dims[k] + 2, n).astype(np.float32) * size).astype(np.float32)
            for _ in range(4):
                v = np.where(rng.random(n) < 0.5, np.nextafter(v, np.float32(rng.choice([-np.inf, np.inf]))), v)
            pts[0, :, k] = v
        odd = np.array([np.nan, np.inf, -np.inf, 3e38, -3e38, 1e-45, -1e-45, 0.0, -0.0, 1.2e7, 1.7e7, 3.4e7, -1.2e7], np.float32)
        pts[0, :600, :3] = rng.choice(odd, (600, 3))
        pts[0, 600:900, 0] = rng.choice(odd, 300)
        w = replace(gen.KITTI.with_shape(1, n), grids=(grid, pillars))
        br = bridge_for(w)
        vox = br.voxelize(torch.from_numpy(pts).cuda())
        br.status()
        for s, g in enumerate(w.grids):
            ref = oracle.voxelize(pts, g.min, g.voxel, g.dims, 0)
            assert int(vox["num_voxels"][s]) == ref["num_voxels"]
            assert np.array_equal(np_(vox["coords"][s])[:ref["num_voxels"]], ref["coords"])
            assert np.array_equal(np_(vox["point_voxel"][s]), ref["point_voxel"])
        br.close()


@pytest.mark.parametrize("B,N", [(1, 1), (7, 33), (3, 255), (2, 1031), (32, 1), (32, 9), (5, 254)])
def test_points_on_image_edges(oracle, B, N):
    """Pixels within a few ulps to a few hundredths of the image edges, at every depth: mask, camera and pixel as defined."""
    rng = np.random.default_rng(7)
    for base in (gen.KITTI, gen.NUSCENES):
        w = base.with_shape(B, N)
        P = np.broadcast_to(gen.make_projection(w), (B, w.K, 3, 4)).astype(np.float32).copy()
        pts = np.zeros((B, N, w.C), np.float32)
        for b in range(B):
            for i in range(N):
                k = rng.integers(w.K)
                d = 0.1 * 800 ** rng.random()
                near = rng.choice([0.0, 1e-7, 1e-5, 1e-4, 1e-3, 9e-3, 1.1e-2, 2e-2]) * rng.choice([-1, 1])
                u = rng.choice([0.0, w.img_w]) + near if rng.random() < 0.6 else rng.random() * w.img_w
                v = rng.choice([0.0, w.img_h]) + near if rng.random() < 0.6 else rng.random() * w.img_h
                M = P[b, k].astype(np.float64)
                pts[b, i, :3] = np.linalg.solve(M[:, :3], np.array([u * d, v * d, d]) - M[:, 3])
        pts[0, 0, :3] = rng.choice([np.nan, np.inf, 1e30])
        uvd, mask, cam = oracle.project(pts, P, w.img_h, w.img_w, w.min_depth)
        feat = rng.standard_normal((B, w.K, w.feat_h, w.feat_w, w.feat_c)).astype(np.float32)
        want = oracle.gather(uvd, cam, feat, w.feat_stride)
        br = bridge_for(w)
        d = [torch.from_numpy(a).cuda() for a in (pts, P, feat)]
        for got in (br.project_gather(*d), br.run(*d)["pg"]):
            br.status()
            assert np.array_equal(np_(got["vis_mask"]), mask)
            assert np.array_equal(np_(got["cam"]), cam)
            assert close(np_(got["uvd"]), uvd)[0]
            assert close(np_(got["gathered"]), want)[0]
        br.close()


@pytest.mark.parametrize("cf", [4, 32, 36, 64, 68, 80, 128, 132, 252, 256, 260, 1020, 1024, 1028])
def test_row_widths_of_the_row_kernels(oracle, cf):
    """Compiled widths, whole rows per CTA, and rows wider than a CTA; ragged tiles, four and five floats per point,
    dispatched point rows in a buffer of any alignment."""
    for base, B, N in ((gen.KITTI, 2, 259), (gen.NUSCENES, 1, 517)):
        w = replace(small_images(base.with_shape(B, N), 64, 96), feat_c=cf)
        batch = gen.make_batch(w)
        ref = oracle.bridge(w, batch)
        assert 0.1 < (ref["cam"] >= 0).mean() < 1
        d = {k: torch.from_numpy(v).cuda() for k, v in batch.items()}
        br = bridge_for(w)
        odd = torch.zeros(B * N * w.C + 1, device="cuda")[1:].view(B, N, w.C)      # 4 bytes past a 16-byte boundary
        for step in (br.run, br.run_staged):
            bufs = step(d["points"], d["proj"], d["feat"])
            bufs["rd"]["points_out"] = odd.zero_()
            bufs = step(d["points"], d["proj"], d["feat"], bufs)
            br.status()
            rd = bufs["rd"]
            assert np.array_equal(np_(rd["perm"]), ref["perm"]) and np.array_equal(np_(rd["offsets"]), ref["offsets"])
            assert np.array_equal(np_(rd["points_out"]).view(np.uint32), ref["points_out"].view(np.uint32))
            assert close(np_(rd["feat_out"]), ref["feat_out"])[0]
            assert close(np_(bufs["pg"]["gathered"]), ref["gathered"])[0]
        br.close()


@pytest.mark.parametrize("cf", [4, 12, 48, 52, 64, 80, 128, 132, 192, 260])
@pytest.mark.parametrize("hw", [(1, 3), (8, 8), (9, 63), (13, 65), (1, 127), (3, 43), (11, 13)])
def test_map_layout_and_pooling_at_tile_edges(oracle, cf, hw):
    h, wd = hw
    w = replace(gen.KITTI.with_shape(2, 16), img_h=8 * h, img_w=8 * wd, feat_stride=8, feat_c=cf)
    rng = np.random.default_rng(cf)
    planar = rng.standard_normal((2, 1, cf, h, wd)).astype(np.float32)
    br = bridge_for(w)
    last = br.features_channels_last(torch.from_numpy(planar).cuda())
    want = oracle.channels_last(planar)
    assert np.array_equal(np_(last), want)
    for p in (1, 2, 3, 4, 8):
        assert close(np_(br.pool_features(last, p)), oracle.pool(want, p))[0]
    br.status()
    br.close()


@pytest.mark.parametrize("p", [2, 4, 8, 16])
@pytest.mark.parametrize("cf,hw", [(4, (13, 21)), (68, (13, 21)), (256, (13, 21)), (64, (16, 32)), (80, (7, 9))])
def test_pooled_sampling_of_cut_windows(oracle, cf, hw, p):
    """Windows cut by both far edges, windows larger than the map, and none cut; voxels of one, two and more points."""
    h, wd = hw
    base = gen.KITTI.with_shape(2, 5001)
    cams = tuple(replace(c, fx=4.0 * wd, fy=4.0 * wd, cx=4.0 * wd, cy=4.0 * h) for c in base.cameras)
    w = replace(base, img_h=8 * h, img_w=8 * wd, feat_stride=8, feat_c=cf, cameras=cams)
    batch = gen.make_batch(w)
    again = np.random.default_rng(cf).integers(0, w.N // 3, w.N)              # about three points at every place
    batch["points"][..., :3] = batch["points"][:, again, :3]
    d = to_dev(batch)
    br = bridge_for(w)
    bufs = br.run(d["points"], d["proj"], d["feat"])
    ref = oracle.bridge(replace(w, feat_stride=8 * p, feat_offset=(p - 1) / 2 * 8), dict(batch, feat=oracle.pool(batch["feat"], p)))
    for s in range(2):
        M = ref[f"vox{s}"]["num_voxels"]
        want, cnt = oracle.voxel_image(ref[f"vox{s}"]["point_voxel"], M, ref["vis_mask"], ref["gathered"])
        assert all(int((cnt == n).sum()) > 0 for n in (0, 1, 2, 3, 4))
        out = br.voxel_image_pooled(bufs["vox"], s, bufs["pg"]["uvd"], bufs["pg"]["cam"], d["feat"], p)
        br.status()
        assert np.array_equal(np_(out["vox_img_count"])[:M], cnt)
        assert close(np_(out["vox_img"])[:M], want)[0]
    br.close()


@pytest.mark.parametrize("base,B,N", [(gen.KITTI, 3, 700), (gen.KITTI, 5, 257), (gen.NUSCENES, 9, 300), (gen.KITTI, 2, 140000),
                                      (gen.DENSE, 2, 3000)], ids=lambda v: getattr(v, "name", str(v)))
def test_frames_that_take_turns_with_notes(oracle, base, B, N):
    """Groups of frames that are not full, frames of one tile and a little, and more points per frame than one copy of the notes would
    take by itself."""
    w = replace(base.with_shape(B, N), feat_c=4)
    refs = []
    for i in range(2):
        batch = gen.make_batch(w, frames=[B * i + k for k in range(B)])
        refs.append((batch, oracle.bridge(w, batch)))
    for step in ("run", "run_staged"):
        br = bridge_for(w)
        for batch, ref in (refs[0], refs[1], refs[0]):
            d = to_dev(batch)
            bufs = getattr(br, step)(d["points"], d["proj"], d["feat"])
            br.status()
            compare_bridge(w, ref, bufs)
        br.close()


@pytest.mark.parametrize("N", [1 << 20, (1 << 20) + 1])
def test_frames_on_either_side_of_the_most_points_that_are_noted(oracle, N):
    w = replace(gen.KITTI.with_shape(2, N), feat_c=4)
    batch = gen.make_batch(w)
    ref = oracle.bridge(w, batch)
    d = to_dev(batch)
    br = bridge_for(w)
    for step in (br.run, br.run_staged, br.run):
        bufs = step(d["points"], d["proj"], d["feat"])
        br.status()
        compare_bridge(w, ref, bufs)
    br.close()


@pytest.mark.parametrize("base,B,N,cf", [(gen.KITTI, 1, 131072, 256), (gen.KITTI, 1, 131073, 256), (gen.KITTI, 2, 66000, 260),
                                         (gen.NUSCENES, 2, 209715, 80), (gen.NUSCENES, 2, 209716, 80)],
                         ids=lambda v: getattr(v, "name", str(v)))
def test_gathered_rows_on_either_side_of_l2(oracle, base, B, N, cf):
    w = replace(base.with_shape(B, N), feat_c=cf)
    batch = gen.make_batch(w)
    ref = oracle.bridge(w, batch)
    br = bridge_for(w)
    d = to_dev(batch)
    compare_bridge(w, ref, br.run_staged(d["points"], d["proj"], d["feat"]))
    br.status()
    br.close()


@pytest.mark.parametrize("cap", [1, 3, 32, 255, 256, 257, 300])
def test_cells_over_the_cap_by_the_length_of_their_lists(oracle, cap):
    """Lists around 32 and 256 entries, which a warp holds in registers, and longer ones; the first and the last points of
    the call among them, on both kinds of store."""
    rng = np.random.default_rng(cap)
    sizes = [cap, cap + 1, 31, 32, 33, 255, 256, 257, 288, 289, 600, 1025]
    for grids in ((BITMAP, replace(TABLE, max_points=cap)), (replace(BITMAP, max_points=cap), replace(TABLE, max_points=cap))):
        at = np.repeat([97 * i for i in range(len(sizes))], sizes)
        cells = np.concatenate([[0], rng.permutation(at[1:-1]), [at[-1]]])       # cell 0 has point 0, the last cell the last point
        pts = centres(cells, TABLE, 4, rng)[None]
        check_voxels(replace(gen.KITTI.with_shape(1, pts.shape[1]), grids=grids), pts, oracle)


@pytest.mark.parametrize("base,B,N,cap", [(gen.KITTI, 2, 1001, 0), (gen.KITTI, 9, 257, 0), (gen.KITTI, 32, 33, 0),
                                          (gen.NUSCENES, 3, 777, 0), (gen.DENSE, 3, 30000, 0), (gen.NUSCENES, 5, 20000, 3),
                                          (gen.KITTI, 3, 1, 0)], ids=lambda v: getattr(v, "name", str(v)))
def test_calls_that_note_the_tiles_they_mark(oracle, base, B, N, cap):
    """Only noted tiles are counted: frames that share a word of notes, the first and last cells of frames among the points,
    both kinds of store over their caps; notes are cleared for the next call, which has other points or fewer frames."""
    w = base.with_shape(B, N)
    w = replace(w, grids=(replace(w.grids[0], max_points=cap), w.grids[1]), feat_c=4)
    frames = [gen.make_batch(w, frames=[B * i + k for k in range(B)]) for i in range(2)]
    for g, at in zip(w.grids, (0, -1)):                        # a point in the first cell and one in the last
        centre = [[m + 0.5 * v for m, v in zip(g.min, g.voxel)], [m + (d - 0.5) * v for m, v, d in zip(g.min, g.voxel, g.dims)]]
        frames[0]["points"][:, at, :3] = np.float32(centre[at])
    refs = [oracle.bridge(w, f) for f in frames]
    for step in ("run", "run_staged"):
        br = bridge_for(w)
        for i in (0, 1, 0):
            d = to_dev(frames[i])
            bufs = getattr(br, step)(d["points"], d["proj"], d["feat"])
            br.status()
            compare_bridge(w, refs[i], bufs)
        w1 = w.with_shape(1, N)
        one = {k: np.ascontiguousarray(v[:1]) for k, v in frames[1].items()}
        d = to_dev(one)
        compare_bridge(w1, oracle.bridge(w1, one), getattr(br, step)(d["points"], d["proj"], d["feat"]))
        d = to_dev(frames[1])
        compare_bridge(w, refs[1], getattr(br, step)(d["points"], d["proj"], d["feat"]))
        br.close()
