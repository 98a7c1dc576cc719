"""The work whose speed counts: what a perception stack has this library do, from one small frame to a full batch.

Every case is one pass through the public entry points of ``paper_2507_04123_b200.Bridge`` on buffers, handle and
inputs that such a program holds already.  Grids, cameras and routing tables are those of ``emc2_gen.configs``; the
points follow the recipe of ``emc2_gen.frames`` (drawn on the GPU here, so that new inputs are quick).

A case is a dict:
  call    "bridge"   Bridge.run: all four stages (rows in point order stored unless ``rows`` is False)
          "staged"   voxelize, project_gather, occlusion, route_dispatch on the unoccluded mask
          "host"     Bridge.run_host: the frame lies in page-locked host memory
          "lidar"    voxelize and the 3x3x3 rulebooks of both voxel lists (the 3-D experts' input)
          "fusion"   voxel_image_sampled of both voxel lists
          "maps"     planar feature maps -> channels last -> p x p pooling
  frame   which of the frame shapes of emc2_gen.configs: tiny, kitti, nuscenes, dense, sweep
  B, N    frames per call, points per frame
  cf      channels of the feature maps
  order   "shuffled" (as the generators leave the points) or "scan" (sweep by sweep, by azimuth, as a spinning
          sensor delivers them)
"""
from __future__ import annotations

import math
from dataclasses import replace

import torch

import emc2_gen as gen
import paper_2507_04123_b200 as pkg

FRAMES = {"tiny": gen.TINY, "kitti": gen.KITTI, "nuscenes": gen.NUSCENES, "dense": gen.DENSE, "sweep": gen.SWEEP}
PAIRS_PER_POINT = 16                     # room for rulebook pairs, per point of the batch
OCCLUSION_CELL, OCCLUSION_MARGIN = 8, 0.5


def _case(name, call, frame, B, N, cf, order="shuffled", rows=True, pool=2):
    return {"name": name, "call": call, "frame": frame, "B": B, "N": N, "cf": cf, "order": order, "rows": rows,
            "pool": pool}


def listed():
    return [
        # One sparse frame, one camera: the smallest call, all latency.
        _case("tiny_frame", "bridge", "tiny", 1, 16384, 64),
        # One live frame of a spinning sensor, in firing order; only the dispatched rows are consumed.
        _case("live_frame", "bridge", "kitti", 1, 120000, 64, order="scan", rows=False),
        # Batched inference on single-camera frames.
        _case("kitti_batch", "bridge", "kitti", 8, 120000, 64),
        # Batched inference on aggregated ten-sweep clouds with six cameras: the benchmark's own workload.
        _case("nuscenes_batch", "bridge", "nuscenes", 4, 300000, 80),
        # Dense urban clutter: pillars over their point cap, many points per voxel.
        _case("dense_frame", "bridge", "dense", 1, 300000, 64),
        # The throughput end of the sweep: 32 frames through six cameras.
        _case("large_batch", "bridge", "sweep", 32, 262144, 80),
        # A ragged batch with wide feature maps (a common neck width).
        _case("ragged_wide", "bridge", "kitti", 3, 33333, 128),
        # The stage calls one by one, with the occlusion test between projection and routing.
        _case("staged_occlusion", "staged", "nuscenes", 2, 120001, 80, order="scan"),
        # LiDAR-only experts: voxel lists and the rulebooks of their sparse convolutions.
        _case("lidar_rulebooks", "lidar", "nuscenes", 4, 300000, 80),
        # Image features per voxel for the fusion expert, both scales.
        _case("voxel_fusion", "fusion", "nuscenes", 4, 300000, 80),
        # An image branch that emits planar maps, with multiscale pooling before the fusion.
        _case("feature_maps", "maps", "nuscenes", 4, 1, 80),
        # A frame that arrives in host memory.
        _case("host_frame", "host", "kitti", 1, 120000, 64, order="scan"),
    ]


def draw(rng):
    call = rng.choice(["bridge"] * 6 + ["staged", "host", "lidar", "fusion", "maps"])
    frame = rng.choice(["tiny", "kitti", "kitti", "nuscenes", "nuscenes", "dense", "sweep", "sweep"])
    most = 524288
    N = int(round(math.exp(rng.uniform(math.log(1000), math.log(most)))))
    B = int(round(math.exp(rng.uniform(0.0, math.log(32)))))
    cf = rng.choice([32, 64, 64, 68, 80, 80, 96, 128, 256])
    if call == "maps":
        N = 1
    case = _case("", call, frame, B, N, cf, order=rng.choice(["shuffled", "scan"]), rows=rng.random() < 0.7,
                 pool=rng.choice([2, 4]))
    del case["name"]
    # No dearer than the largest listed case: its rows and maps, and for the optional calls a few million points.
    w = _workload(case)
    while case["B"] > 1 and (_row_bytes(case, w) > 0.9 * 5.4e9 or
                             (call not in ("bridge", "maps") and case["B"] * N > 1500000)):
        case["B"] -= 1
        w = _workload(case)
    return case


def _row_bytes(case, w):
    return case["B"] * (case["N"] * 8 * w.feat_c + w.K * w.feat_h * w.feat_w * w.feat_c * 4)


def _workload(case):
    return replace(FRAMES[case["frame"]], B=case["B"], N=case["N"], feat_c=case["cf"])


# ------------------------------------------------------------------------------------------------ inputs
def _ground(g, dev, B, n, r0, r1, z0, square=None):
    """Ground returns: log-uniform range, full azimuth; with `square`, kept inside |x|, |y| < square."""
    def some(m):
        r = r0 * (r1 / r0) ** torch.rand((B, m), generator=g, device=dev, dtype=torch.float64)
        az = (torch.rand((B, m), generator=g, device=dev, dtype=torch.float64) * 2 - 1) * math.pi
        z = z0 + 0.05 * torch.randn((B, m), generator=g, device=dev, dtype=torch.float64)
        return torch.stack([r * torch.cos(az), r * torch.sin(az), z], dim=2)

    if square is None:
        return some(n)
    p = some(2 * n + 64)
    ok = (p[..., 0].abs() < square) & (p[..., 1].abs() < square)
    first = torch.argsort((~ok).to(torch.int8), dim=1, stable=True)[:, :n]      # those inside, in order
    return torch.gather(p, 1, first[..., None].expand(-1, -1, 3))


def _boxes(g, dev, centres, sizes, per_box, z0):
    B, nb = centres.shape[:2]
    u = torch.rand((B, nb, per_box, 3), generator=g, device=dev, dtype=torch.float64)
    yaw = (torch.rand((B, nb, 1), generator=g, device=dev, dtype=torch.float64)) * math.pi
    s = torch.tensor(sizes, device=dev, dtype=torch.float64).view(1, nb, 1, 3)
    lx, ly, lz = (u[..., 0] - 0.5) * s[..., 0], (u[..., 1] - 0.5) * s[..., 1], u[..., 2] * s[..., 2]
    c, sn = torch.cos(yaw), torch.sin(yaw)
    xyz = torch.stack([centres[..., 0:1] + c * lx - sn * ly, centres[..., 1:2] + sn * lx + c * ly, z0 + lz], dim=3)
    return xyz.reshape(B, nb * per_box, 3)


def _points(case, w, g, dev):
    """float32 [B, N, C] with the statistics of emc2_gen.frames.make_points."""
    B, n = w.B, w.N

    def uniform(shape, lo, hi):
        return lo + (hi - lo) * torch.rand(shape, generator=g, device=dev, dtype=torch.float64)

    if w.generator == "uniform":
        x0, x1, y0, y1 = w.xy_range
        xyz = torch.stack([uniform((B, n), x0, x1), uniform((B, n), y0, y1), uniform((B, n), -3.0, 1.0)], dim=2)
    elif w.generator == "dense":
        per = (6 * n // 10) // 150
        rc = 25.0 * torch.sqrt(uniform((B, 100), 0.0, 1.0))
        ac = uniform((B, 100), -math.pi / 2, math.pi / 2)
        cars = torch.stack([rc * torch.cos(ac), rc * torch.sin(ac)], dim=2)
        gx, gy = torch.meshgrid(torch.arange(0.0, 26.0, 2.0), torch.arange(-24.0, 26.0, 2.0), indexing="ij")
        sites = torch.stack([gx.ravel(), gy.ravel()], dim=1).double()
        rr = sites.norm(dim=1)
        sites = sites[(rr >= 4.0) & (rr <= 24.0)].to(dev)
        pick = torch.argsort(torch.rand((B, len(sites)), generator=g, device=dev), dim=1)[:, :50]
        centres = torch.cat([cars, sites[pick] + uniform((B, 50, 2), -0.5, 0.5)], dim=1)
        xyz = _ground(g, dev, B, n - per * 150, 2.5, 70.4, -1.7)
        if per:
            sizes = [(3.9, 1.6, 1.56)] * 100 + [(0.4, 0.4, 1.8)] * 50
            xyz = torch.cat([xyz, _boxes(g, dev, centres, sizes, per, -1.7)], dim=1)
    else:
        nus = w.generator == "nuscenes"
        nb = 40 if nus else 20
        per = (3 * n // 10) // nb
        z0 = -1.84 if nus else -1.7
        if nus:
            xyz = _ground(g, dev, B, n - per * nb, 1.5, 72.4, z0, square=51.2)
            centres = uniform((B, nb, 2), -45.0, 45.0)
        else:
            xyz = _ground(g, dev, B, n - per * nb, 2.5, 70.4, z0)
            centres = torch.stack([uniform((B, nb), 5.0, 65.0), uniform((B, nb), -35.0, 35.0)], dim=2)
        if per:
            xyz = torch.cat([xyz, _boxes(g, dev, centres, [(3.9, 1.6, 1.56)] * nb, per, z0)], dim=1)
        if nus:
            xyz[..., 2].clamp_(-5.0, 3.0)
    e = -torch.log1p(-torch.rand((7, B, n), generator=g, device=dev))              # Beta(2, 5) from exponentials
    inten = e[:2].sum(0) / e.sum(0)
    cols = [xyz.float(), inten[..., None]]
    sweep = torch.randint(0, 10, (B, n), generator=g, device=dev)
    if w.C == 5:
        cols.append((0.05 * sweep.double()).float()[..., None])
    pts = torch.cat(cols, dim=2)
    if case["order"] == "scan":
        key = torch.atan2(pts[..., 1], pts[..., 0]).double() + (sweep.double() * 10.0 if w.C == 5 else 0.0)
    else:
        key = torch.rand((B, n), generator=g, device=dev, dtype=torch.float64)
    return torch.gather(pts, 1, torch.argsort(key, dim=1)[..., None].expand_as(pts)).contiguous()


def _buffers(w, rows):
    """Output buffers of Bridge.run, zeroed once: rows past the voxels found are never written."""
    B, N, C, M = w.B, w.N, w.C, w.B * w.N
    gx, gy = w.grids[1].dims[:2]

    def z(*shape, dtype=torch.float32):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    i32 = torch.int32
    return {"vox": {"coords": [z(M, 4, dtype=i32) for _ in range(2)], "counts": [z(M, dtype=i32) for _ in range(2)],
                    "mean": [z(M, C) for _ in range(2)], "point_voxel": [z(B, N, dtype=i32) for _ in range(2)],
                    "num_voxels": z(2, dtype=i32), "bev": z(B, C, gy, gx)},
            "pg": {"uvd": z(B, N, 3), "vis_mask": z(B, N, dtype=torch.uint8), "cam": z(B, N, dtype=torch.int8),
                   "gathered": z(B, N, w.feat_c) if rows else None},
            "rd": {"expert": z(B, N, dtype=torch.uint8), "offsets": z(B, w.num_experts + 1, dtype=i32),
                   "perm": z(B, N, dtype=i32), "points_out": z(B, N, C), "feat_out": z(B, N, w.feat_c)}}


def _inputs(case, w, seed):
    """The call's inputs on the GPU: some of points [B, N, C], proj [B, K, 3, 4] and feat."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, K, call = w.B, w.K, case["call"]
    maps = (B, K, w.feat_c, w.feat_h, w.feat_w) if call == "maps" else (B, K, w.feat_h, w.feat_w, w.feat_c)
    s = {}
    if call != "lidar":
        s["feat"] = torch.randn(maps, generator=g, device="cuda")
    if call != "maps":
        s["points"] = _points(case, w, g, "cuda")
    if call not in ("lidar", "maps"):
        s["proj"] = torch.from_numpy(gen.make_projection(w)).cuda()[None].expand(B, -1, -1, -1).contiguous()
    return s


def prepare(case, seed):
    w = _workload(case)
    B, K = w.B, w.K
    s = {"case": case, "w": w, "bridge": pkg.Bridge(pkg.config_from_workload(w)), **_inputs(case, w, seed)}
    if case["call"] == "maps":
        p = case["pool"]
        s["last"] = torch.zeros((B, K, w.feat_h, w.feat_w, w.feat_c), device="cuda")
        s["pooled"] = torch.zeros((B, K, -(-w.feat_h // p), -(-w.feat_w // p), w.feat_c), device="cuda")
        return s
    s["bufs"] = _buffers(w, case["rows"] or case["call"] != "bridge")
    M = B * w.N
    if case["call"] == "staged":
        shape = (B, K, -(-w.img_h // OCCLUSION_CELL), -(-w.img_w // OCCLUSION_CELL))
        s["occ"] = {"zbuf": torch.zeros(shape, device="cuda"),
                    "occ_mask": torch.zeros((B, w.N), dtype=torch.uint8, device="cuda"),
                    "clear_mask": torch.zeros((B, w.N), dtype=torch.uint8, device="cuda")}
    elif case["call"] == "host":
        s["host"] = {k: s[k].cpu().pin_memory() for k in ("points", "proj", "feat")}
        s["h_offsets"] = torch.zeros((B, w.num_experts + 1), dtype=torch.int32).pin_memory()
        s["h_num_voxels"] = torch.zeros((2,), dtype=torch.int32).pin_memory()
        s["staging"] = {k: s.pop(k) for k in ("points", "proj", "feat")}
    elif case["call"] == "lidar":
        s["rules"] = [{"offsets": torch.zeros((28,), dtype=torch.int32, device="cuda"),
                       "rule_in": torch.zeros((PAIRS_PER_POINT * M,), dtype=torch.int32, device="cuda"),
                       "rule_out": torch.zeros((PAIRS_PER_POINT * M,), dtype=torch.int32, device="cuda")}
                      for _ in range(2)]
    elif case["call"] == "fusion":
        s["images"] = [{"vox_img": torch.zeros((M, w.feat_c), device="cuda"),
                        "vox_img_count": torch.zeros((M,), dtype=torch.int32, device="cuda")} for _ in range(2)]
        s["bridge"].run(s["points"], s["proj"], s["feat"], s["bufs"])    # the step whose outputs are fused
    return s


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    br, call = s["bridge"], s["case"]["call"]
    if call == "maps":
        return {"last": br.features_channels_last(s["feat"], out=s["last"]),
                "pooled": br.pool_features(s["last"], s["case"]["pool"], out=s["pooled"])}
    bufs = s["bufs"]
    if call == "bridge":
        return br.run(s["points"], s["proj"], s["feat"], bufs)
    if call == "host":
        br.run_host(s["host"], s["staging"], bufs, s["h_offsets"], s["h_num_voxels"])
        return {"bufs": bufs, "offsets": s["h_offsets"], "num_voxels": s["h_num_voxels"]}
    if call == "staged":
        vox = br.voxelize(s["points"], out=bufs["vox"])
        pg = br.project_gather(s["points"], s["proj"], s["feat"], out=bufs["pg"])
        occ = br.occlusion(s["points"], s["proj"], pg["vis_mask"], OCCLUSION_CELL, OCCLUSION_MARGIN, out=s["occ"])
        rd = br.route_dispatch(s["points"], occ["clear_mask"], pg["gathered"], out=bufs["rd"])
        return {"vox": vox, "pg": pg, "occ": occ, "rd": rd}
    if call == "lidar":
        vox = br.voxelize(s["points"], out=bufs["vox"])
        return {"vox": vox, "rules": [br.rulebook(vox, k, out=s["rules"][k]) for k in range(2)]}
    vox, pg = bufs["vox"], bufs["pg"]
    return [br.voxel_image_sampled(vox, k, pg["uvd"], pg["cam"], s["feat"], out=s["images"][k]) for k in range(2)]


# ------------------------------------------------------------------------------------------------ the values in 64 bits
# Which cell, camera and expert a point belongs to is decided in 32 bits by definition (one rounding per
# operation), and feature rows are sampled at the 32-bit pixel that the call returns; those are taken in 32 bits here
# too, and every value is then computed in 64 bits.
def _fma(a, b, c):
    """a * b + c of 32-bit numbers with one rounding (the product is exact in 64 bits)."""
    return (a.double() * b.double() + c.double()).float()


def _voxels64(pts, gr):
    """Per scale: row of every point's voxel (-1: outside, or past the cap), points kept per row, means, cell ids."""
    B, N, C = pts.shape
    flat = pts.reshape(-1, C)
    # a vector divisor: a plain number would be turned into a multiplication by its reciprocal
    lo, size = (torch.tensor(v, device=pts.device).expand(len(flat), 3) for v in (gr.min, gr.voxel))
    f = torch.floor((flat[:, :3] - lo) / size)
    dims = torch.tensor(gr.dims, device=pts.device)
    ok = ((f >= 0) & (f < dims)).all(1)
    c = torch.where(ok[:, None], f, torch.zeros_like(f)).long()
    frame = torch.arange(B, device=pts.device).repeat_interleave(N)
    cell = ((frame * gr.dims[2] + c[:, 2]) * gr.dims[1] + c[:, 1]) * gr.dims[0] + c[:, 0]
    at = ok.nonzero()[:, 0]
    ids, row = torch.unique(cell[at], return_inverse=True)
    if gr.max_points:                                                # the first points of every voxel, by index
        order = torch.argsort(row, stable=True)
        start = torch.searchsorted(row[order], torch.arange(len(ids), device=pts.device))
        keep = torch.arange(len(order), device=pts.device) - start[row[order]] < gr.max_points
        at, row = at[order[keep]], row[order[keep]]
    n = torch.bincount(row, minlength=len(ids))
    total = torch.zeros((len(ids), C), dtype=torch.float64, device=pts.device).index_add_(0, row, flat[at].double())
    point_row = torch.full((B * N,), -1, device=pts.device).index_put_((at,), row)
    return point_row, n, total / n[:, None], ids


def _vox64(pts, w):
    means, rows = [], []
    B, N, C = pts.shape
    gx, gy = w.grids[1].dims[:2]
    for gr in w.grids:
        point_row, _, mean, ids = _voxels64(pts, gr)
        rows.append(point_row)
        means.append(torch.zeros((B * N, C), dtype=torch.float64, device=pts.device))
        means[-1][:len(ids)] = mean
    bev = torch.zeros((B, gy * gx, C), dtype=torch.float64, device=pts.device)
    bev.view(-1, C)[ids] = mean                                      # pillars: one cell high
    bev = bev.transpose(1, 2).reshape(B, C, gy, gx)
    return {"coords": [None] * 2, "counts": [None] * 2, "mean": means, "point_voxel": [None] * 2,
            "num_voxels": None, "bev": bev}, rows


def _project64(pts, proj, w):
    """Per frame: uvd in 64 bits, the pixel in 32 bits, the lowest camera that sees each point (-1: none), and per
    camera its mask, pixel and depth."""
    x, y, z = pts[:, 0], pts[:, 1], pts[:, 2]
    N = len(pts)
    best = torch.full((N,), -1, device=pts.device)
    uvd = torch.full((N, 3), -1.0, dtype=torch.float64, device=pts.device)
    pixel = torch.zeros((N, 2), device=pts.device)
    views = []
    for k in range(w.K):
        P = proj[k]
        t = [_fma(P[r, 0], x, _fma(P[r, 1], y, _fma(P[r, 2], z, P[r, 3]))) for r in range(3)]
        u, v = t[0] / t[2], t[1] / t[2]
        vis = (t[2] > w.min_depth) & (u >= 0) & (u < w.img_w) & (v >= 0) & (v < w.img_h)
        q = pts[:, :3].double() @ P[:, :3].double().T + P[:, 3].double()
        if k == 0:
            uvd[:, 2] = q[:, 2]
        first = vis & (best < 0)
        uvd[first] = torch.stack([q[:, 0] / q[:, 2], q[:, 1] / q[:, 2], q[:, 2]], dim=1)[first]
        pixel[first] = torch.stack([u, v], dim=1)[first]
        best[first] = k
        views.append((vis, u, v, q[:, 2], t[2]))
    return uvd, pixel, best, views


def _rows64(pixel, best, feat, w):
    """Feature rows of one frame, blended in 64 bits; zeros for points that no camera sees."""
    rows = torch.zeros((len(best), w.feat_c), dtype=torch.float64, device=feat.device)
    seen = (best >= 0).nonzero()[:, 0]
    for at in seen.split(1 << 18):
        fx, fy = ((pixel[at, d].double() - w.feat_offset) / w.feat_stride for d in (0, 1))
        x0, y0 = torch.floor(fx), torch.floor(fy)
        wx, wy = (fx - x0)[:, None], (fy - y0)[:, None]

        def tap(dy, dx):
            return feat[best[at], (y0.long() + dy).clamp(0, w.feat_h - 1), (x0.long() + dx).clamp(0, w.feat_w - 1)].double()

        rows[at] = (1 - wy) * ((1 - wx) * tap(0, 0) + wx * tap(0, 1)) + wy * ((1 - wx) * tap(1, 0) + wx * tap(1, 1))
    return rows


def _experts(pts, visible, w):
    r2 = _fma(pts[:, 0], pts[:, 0], pts[:, 1] * pts[:, 1])
    bucket = torch.zeros(len(pts), dtype=torch.long, device=pts.device)
    for t in w.thresholds:
        t = torch.tensor(t, device=pts.device)                       # 32 bits, and so is its square
        bucket += (r2 >= t * t).long()
    return torch.tensor(w.lut, device=pts.device)[visible.long(), bucket]


def exact(case, seed):
    """What `run` returns, its numbers computed in 64 bits by plain torch; None for whole numbers."""
    w, call = _workload(case), case["call"]
    s = _inputs(case, w, seed)
    if call == "maps":
        last = s["feat"].permute(0, 1, 3, 4, 2).double()
        p = case["pool"]
        pooled = torch.nn.functional.avg_pool2d(s["feat"].double().flatten(0, 1), p, ceil_mode=True,
                                                count_include_pad=False)
        pooled = pooled.permute(0, 2, 3, 1).unflatten(0, last.shape[:2])
        return {"last": last.contiguous(), "pooled": pooled.contiguous()}
    pts = s["points"]
    vox, point_rows = _vox64(pts, w)
    if call == "lidar":
        return {"vox": vox, "rules": [None, None]}
    B, N, C = pts.shape
    f64 = {"dtype": torch.float64, "device": pts.device}
    uvd, rows = torch.zeros((B, N, 3), **f64), torch.zeros((B, N, w.feat_c), **f64)
    best = torch.zeros((B, N), dtype=torch.long, device=pts.device)
    views = []
    for b in range(B):
        uvd[b], pixel, best[b], v = _project64(pts[b], s["proj"][b], w)
        views.append(v if call == "staged" else None)
        rows[b] = _rows64(pixel, best[b], s["feat"][b], w)
    if call == "fusion":
        images, seen = [], (best >= 0).flatten()
        for point_row in point_rows:
            at = ((point_row >= 0) & seen).nonzero()[:, 0]
            total = torch.zeros((B * N, w.feat_c), **f64).index_add_(0, point_row[at], rows.view(B * N, -1)[at])
            n = torch.bincount(point_row[at], minlength=B * N).clamp(min=1)
            images.append({"vox_img": total / n[:, None], "vox_img_count": None})
        return images
    visible, occ = best >= 0, None
    if call == "staged":
        hz, wz = -(-w.img_h // OCCLUSION_CELL), -(-w.img_w // OCCLUSION_CELL)
        zbuf = torch.full((B, w.K, hz * wz), float("inf"), **f64)
        for b in range(B):
            visible[b] = False
            for k, (vis, u, v, depth, depth32) in enumerate(views[b]):
                cell = (v[vis] / OCCLUSION_CELL).long() * wz + (u[vis] / OCCLUSION_CELL).long()
                zbuf[b, k].scatter_reduce_(0, cell, depth[vis], "amin")
                near = torch.full((hz * wz,), float("inf"), device=pts.device).scatter_reduce_(0, cell, depth32[vis], "amin")
                visible[b, vis.nonzero()[:, 0][~(depth32[vis] > near[cell] + OCCLUSION_MARGIN)]] = True
        occ = {"zbuf": zbuf.view(B, w.K, hz, wz), "occ_mask": None, "clear_mask": None}
    points_out, feat_out = torch.zeros((B, N, C), **f64), torch.zeros((B, N, w.feat_c), **f64)
    for b in range(B):
        order = torch.argsort(_experts(pts[b], visible[b], w), stable=True)
        points_out[b], feat_out[b] = pts[b, order].double(), rows[b, order]
    pg = {"uvd": uvd, "vis_mask": None, "cam": None, "gathered": rows if case["rows"] or call != "bridge" else None}
    rd = {"expert": None, "offsets": None, "perm": None, "points_out": points_out, "feat_out": feat_out}
    out = {"vox": vox, "pg": pg, "rd": rd}
    if call == "staged":
        return {**out, "occ": occ}
    return {"bufs": out, "offsets": None, "num_voxels": None} if call == "host" else out


# ------------------------------------------------------------------------------------------------ what a pass is
def _statistics(case, w):
    """Voxels per scale, distinct texels, visible points and rulebook pairs of one frame, counted on a frame of the case."""
    one = replace(w, B=1)
    pts = _points(dict(case, order="shuffled"), one, torch.Generator().manual_seed(1), "cpu")[0].double()
    voxels, pairs = [], []
    for gr in w.grids:
        c = [torch.floor((pts[:, d] - gr.min[d]) / gr.voxel[d]).long() for d in range(3)]
        ok = torch.ones(len(pts), dtype=torch.bool)
        for d in range(3):
            ok &= (c[d] >= 0) & (c[d] < gr.dims[d])
        # one cell of margin on every side, so that a neighbour is a fixed step of the id away
        sx, sy = gr.dims[0] + 2, gr.dims[1] + 2
        ids = torch.unique((((c[2] + 1) * sy + c[1] + 1) * sx + c[0] + 1)[ok])
        voxels.append(len(ids))
        if case["call"] == "lidar":
            steps = [(z * sy + y) * sx + x for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
            pairs.append(sum(int(torch.isin(ids + d, ids, assume_unique=True).sum()) for d in steps))
    P = torch.from_numpy(gen.make_projection(w)).double()
    left, keys, seen = torch.ones(len(pts), dtype=torch.bool), [], 0
    for k in range(w.K):
        q = pts[:, :3] @ P[k, :, :3].T + P[k, :, 3]
        u, v = q[:, 0] / q[:, 2], q[:, 1] / q[:, 2]
        vis = left & (q[:, 2] > w.min_depth) & (u >= 0) & (u < w.img_w) & (v >= 0) & (v < w.img_h)
        left &= ~vis
        seen += int(vis.sum())
        x0, y0 = (u[vis] / w.feat_stride).long(), (v[vis] / w.feat_stride).long()
        for dy in (0, 1):
            for dx in (0, 1):
                keys.append((k * w.feat_h + (y0 + dy).clamp(max=w.feat_h - 1)) * w.feat_w +
                            (x0 + dx).clamp(max=w.feat_w - 1))
    return voxels, len(torch.unique(torch.cat(keys))), seen, pairs


def work(case):
    """Bytes of one pass with every input read once and every output written once, and its arithmetic."""
    w = _workload(case)
    call, B, N, C = case["call"], w.B, w.N, w.C
    pt, row = 4 * C, 4 * w.feat_c
    if call == "maps":
        p = case["pool"]
        whole = B * w.K * w.feat_h * w.feat_w * row
        pooled = B * w.K * -(-w.feat_h // p) * -(-w.feat_w // p) * row
        return {"bytes": 2 * whole + pooled, "flops": whole // 4 + pooled // 4}
    voxels, texels, seen, pairs = _statistics(case, w)
    maps = B * (texels * row + w.K * 48)
    gx, gy = w.grids[1].dims[:2]
    vox = B * (8 * N + sum(voxels) * (20 + pt) + C * gx * gy * 4) + 8            # lists, point rows, BEV image
    blend = 7 * B * seen * w.feat_c
    if call == "lidar":
        return {"bytes": B * N * pt + vox + 8 * B * sum(pairs) + 2 * 112, "flops": 2 * B * N * (C + 6)}
    if call == "fusion":
        ins = 2 * B * N * 4 + B * N * 13 + 4 * B * sum(voxels) + maps
        return {"bytes": ins + B * sum(voxels) * (row + 4), "flops": 2 * (blend + B * seen * w.feat_c)}
    out = vox + B * N * 14 + B * N * (5 + pt + row) + B * (w.num_experts + 1) * 4
    if case["rows"] or call != "bridge":
        out += B * N * row
    if call == "host":
        maps = B * w.K * (w.feat_h * w.feat_w * row + 48)                        # the whole maps cross the bus
    if call == "staged":
        out += 2 * B * N + 4 * B * w.K * -(-w.img_h // OCCLUSION_CELL) * -(-w.img_w // OCCLUSION_CELL)
    return {"bytes": B * N * pt + maps + out, "flops": B * N * (18 * w.K + 2 * (C + 6)) + blend}


def tolerance(case):
    """Integers, masks and moved rows are exact.  Pixel coordinates, means, blends and pooled texels are a few fp32
    operations each, sums in no fixed order: against 64-bit arithmetic the listed cases are off by at most 4.9e-8
    (2-norm) and 4.0e-7 (largest difference); four times that, and more for voxels of many points."""
    return {"rel": 2e-7, "max": 4e-6}
