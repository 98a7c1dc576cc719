"""Calls captured into CUDA graphs: which launches are chained to their predecessor, and replays on new frames (needs a B200)."""
import ctypes
from dataclasses import replace

import numpy as np
import pytest
import torch

import emc2_gen as gen
from parity import compare_bridge, to_dev

pytestmark = pytest.mark.gpu


def bridge_for(w, **kw):
    import paper_2507_04123_b200 as pkg
    return pkg.Bridge(pkg.config_from_workload(w, **kw))


def captured(call):
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    return graph


def chained_launches(graph):
    """Checks that every chained launch follows exactly one node, a kernel; returns how many there are."""
    cu = ctypes.CDLL("libcuda.so.1")
    g, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetEdges_v2(g, None, None, None, ctypes.byref(n)) == 0
    tails, heads = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)()
    edges = (ctypes.c_uint8 * 8 * n.value)()               # CUgraphEdgeData: from_port, to_port, type, 5 reserved bytes
    assert cu.cuGraphGetEdges_v2(g, tails, heads, edges, ctypes.byref(n)) == 0

    def is_kernel(node):
        kind = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        return kind.value == 0                               # CU_GRAPH_NODE_TYPE_KERNEL

    found = 0
    for i in range(n.value):
        if edges[i][2] == 1:                                 # CU_GRAPH_DEPENDENCY_TYPE_PROGRAMMATIC
            found += 1
            assert is_kernel(tails[i]) and is_kernel(heads[i])
            assert list(heads).count(heads[i]) == 1
    return found


def test_host_frame_replays_from_a_graph(oracle):
    """The row pass follows the copy of the feature maps there; page-locked buffers, refilled before each replay."""
    w = gen.KITTI.with_shape(2, 20001)
    frames = [gen.make_batch(w, frames=[2 * i, 2 * i + 1]) for i in range(2)]
    br = bridge_for(w)
    host = {k: torch.from_numpy(v.copy()).pin_memory() for k, v in frames[0].items()}
    staging = {k: torch.zeros_like(v, device="cuda") for k, v in host.items()}
    d = to_dev(frames[0])
    bufs = br.run(d["points"], d["proj"], d["feat"])
    h_off = torch.zeros((w.B, w.num_experts + 1), dtype=torch.int32).pin_memory()
    h_nv = torch.zeros((2,), dtype=torch.int32).pin_memory()
    torch.cuda.synchronize()
    graph = captured(lambda: br.run_host(host, staging, bufs, h_off, h_nv))
    assert chained_launches(graph) >= 3
    for batch in (frames[1], frames[0]):
        for k, v in batch.items():
            host[k].copy_(torch.from_numpy(v))
            staging[k].fill_(float("nan"))
        bufs["rd"]["feat_out"].fill_(-1.0)
        graph.replay()
        torch.cuda.synchronize()
        br.status()
        ref = oracle.bridge(w, batch)
        compare_bridge(w, ref, bufs)
        assert np.array_equal(h_off.numpy(), ref["offsets"])
        assert h_nv.tolist() == [ref["vox0"]["num_voxels"], ref["vox1"]["num_voxels"]]
    del graph
    br.close()


@pytest.mark.parametrize("overlap", [True, False])
@pytest.mark.parametrize("pinned", [True, False])
def test_host_frames_one_behind_another(oracle, overlap, pinned):
    """The maps are copied on a stream of their own: not before an earlier call's rows have read the last ones, and the results
    are back when the caller's stream is through."""
    w = gen.KITTI.with_shape(2, 20001)
    frames = [gen.make_batch(w, frames=[2 * i, 2 * i + 1]) for i in range(3)]
    br = bridge_for(w)
    br.set_overlap(overlap)
    d = to_dev(frames[0])
    buffers = [br.run(d["points"], d["proj"], d["feat"]) for _ in frames]
    hosts = [{k: torch.from_numpy(v.copy()) for k, v in f.items()} for f in frames]
    if pinned:
        hosts = [{k: v.pin_memory() for k, v in h.items()} for h in hosts]
    staging = {k: torch.zeros_like(v, device="cuda") for k, v in hosts[0].items()}
    results = [(torch.zeros((w.B, w.num_experts + 1), dtype=torch.int32).pin_memory(), torch.zeros((2,), dtype=torch.int32).pin_memory())
               for _ in frames]
    torch.cuda.synchronize()
    for host, bufs, res in zip(hosts, buffers, results):       # all enqueued before the first is through
        br.run_host(host, staging, bufs, *res)
    torch.cuda.current_stream().synchronize()
    for batch, bufs, (off, nv) in zip(frames, buffers, results):
        ref = oracle.bridge(w, batch)
        assert np.array_equal(off.numpy(), ref["offsets"])
        assert nv.tolist() == [ref["vox0"]["num_voxels"], ref["vox1"]["num_voxels"]]
        compare_bridge(w, ref, bufs)
    br.status()
    br.close()


@pytest.mark.parametrize("B", [2, 3])
@pytest.mark.parametrize("tuning", [{}, {"split_batch": 1}, {"mark_in_projection": 0}, {"split_batch": 1, "mark_in_projection": 0},
                                    {"dedup_fine": 2, "dedup_pillars": 1}], ids=str)
def test_host_frame_under_every_tuning(oracle, tuning, B):
    """The results are copied after the kernels that write them, whichever frames those are launched for: directly and from
    a graph, with nothing of an earlier call in the buffers."""
    w = gen.KITTI.with_shape(B, 20001)
    frames = [gen.make_batch(w, frames=list(range(B * i, B * i + B))) for i in range(2)]
    for overlap in (True, False):
        br = bridge_for(w)
        br.set_overlap(overlap)
        for knob, value in tuning.items():
            br.set_tuning(knob, value)
        host = {k: torch.from_numpy(v.copy()).pin_memory() for k, v in frames[0].items()}
        staging = {k: torch.zeros_like(v, device="cuda") for k, v in host.items()}
        d = to_dev(frames[0])
        bufs = br.run(d["points"], d["proj"], d["feat"])
        h_off = torch.zeros((B, w.num_experts + 1), dtype=torch.int32).pin_memory()
        h_nv = torch.zeros((2,), dtype=torch.int32).pin_memory()
        torch.cuda.synchronize()
        graph = captured(lambda: br.run_host(host, staging, bufs, h_off, h_nv))
        for call in (lambda: br.run_host(host, staging, bufs, h_off, h_nv), graph.replay):
            for batch in (frames[1], frames[0]):
                for k, v in batch.items():
                    host[k].copy_(torch.from_numpy(v))
                for t in (h_off, h_nv, bufs["rd"]["offsets"], bufs["vox"]["num_voxels"], bufs["rd"]["feat_out"]):
                    t.fill_(-1)
                torch.cuda.synchronize()
                call()
                torch.cuda.synchronize()
                br.status()
                ref = oracle.bridge(w, batch)
                assert np.array_equal(h_off.numpy(), ref["offsets"])
                assert h_nv.tolist() == [ref["vox0"]["num_voxels"], ref["vox1"]["num_voxels"]]
                compare_bridge(w, ref, bufs)
        del graph
        br.close()


@pytest.mark.parametrize("B", [2, 3])
@pytest.mark.parametrize("tuning", [{}, {"split_batch": 1}, {"mark_in_projection": 0}, {"dedup_pillars": 1},
                                    {"dedup_fine": 2, "dedup_pillars": 2}])
def test_one_call_replays_from_a_graph_under_every_tuning(oracle, tuning, B):
    """split_batch: the second half's route scan follows a wait for the other stream."""
    w = gen.NUSCENES.with_shape(B, 7001)
    w = replace(w, img_h=180, img_w=320, cameras=tuple(replace(c, fx=200.0, fy=200.0, cx=160.0, cy=90.0) for c in w.cameras))
    frames = [gen.make_batch(w, frames=list(range(B * i, B * i + B))) for i in range(2)]
    for overlap in (True, False):
        br = bridge_for(w)
        br.set_overlap(overlap)
        for knob, value in tuning.items():
            br.set_tuning(knob, value)
        d = to_dev(frames[0])
        bufs = br.run(d["points"], d["proj"], d["feat"])
        torch.cuda.synchronize()
        graph = captured(lambda: br.run(d["points"], d["proj"], d["feat"], bufs))
        assert chained_launches(graph) >= 3
        for batch in (frames[1], frames[0]):
            for k, v in batch.items():
                d[k].copy_(torch.from_numpy(v))
            bufs["rd"]["feat_out"].fill_(-1.0)
            bufs["vox"]["num_voxels"].fill_(-1)
            graph.replay()
            torch.cuda.synchronize()
            br.status()
            compare_bridge(w, oracle.bridge(w, batch), bufs)
        del graph
        br.close()


@pytest.mark.parametrize("cf,rows", [(64, True), (1024, True), (1024, False)])
def test_either_branch_of_a_call_beside_the_callers_stream(oracle, cf, rows):
    """Small calls put the rows on the other stream, calls of many row bytes stage 1: directly, and from a graph."""
    w = replace(gen.KITTI.with_shape(1, 24001), feat_c=cf)
    frames = [gen.make_batch(w, frames=[i]) for i in range(2)]
    br = bridge_for(w)
    d = to_dev(frames[0])
    bufs = br.run(d["points"], d["proj"], d["feat"])
    gathered = bufs["pg"]["gathered"]
    if not rows:
        bufs["pg"]["gathered"] = None
    torch.cuda.synchronize()
    graph = captured(lambda: br.run(d["points"], d["proj"], d["feat"], bufs))
    assert chained_launches(graph) >= 4
    for call in (lambda: br.run(d["points"], d["proj"], d["feat"], bufs), graph.replay):
        for batch in (frames[1], frames[0]):
            ref = oracle.bridge(w, batch)
            for k, v in batch.items():
                d[k].copy_(torch.from_numpy(v))
            for t in (bufs["rd"]["feat_out"], bufs["vox"]["bev"], gathered):
                t.fill_(-1.0)
            call()
            torch.cuda.synchronize()
            br.status()
            shown = {**bufs, "pg": {**bufs["pg"], "gathered": gathered if rows else torch.from_numpy(ref["gathered"])}}
            compare_bridge(w, ref, shown)
            assert rows or bool((gathered == -1.0).all())
    del graph
    br.close()


def test_stage_calls_and_calls_without_points_in_a_graph():
    """With N = 0 the route scan is the first kernel of its call: nothing is chained to what the stream held before."""
    w = gen.KITTI.with_shape(2, 1000)
    br = bridge_for(w)
    d = to_dev(gen.make_batch(w))
    bufs = br.run_staged(d["points"], d["proj"], d["feat"])
    torch.cuda.synchronize()
    graph = captured(lambda: br.run_staged(d["points"], d["proj"], d["feat"], bufs))
    assert chained_launches(graph) >= 4
    del graph
    none = br.run(d["points"][:, :0].contiguous(), d["proj"], d["feat"])
    rd = none["rd"]
    torch.cuda.synchronize()
    for call in (lambda: br.run(d["points"][:, :0].contiguous(), d["proj"], d["feat"], none),
                 lambda: br.route_dispatch(d["points"][:, :0].contiguous(), none["pg"]["vis_mask"], none["pg"]["gathered"], out=rd)):
        rd["offsets"].fill_(-1)
        torch.cuda.synchronize()

        def kernel_first():
            bufs["pg"]["uvd"].fill_(0.0)                    # a kernel of the caller's right before the call
            call()

        graph = captured(kernel_first)
        assert chained_launches(graph) == 0
        graph.replay()
        torch.cuda.synchronize()
        assert not rd["offsets"].any()
        del graph
    br.close()
