"""A path tracing call that is captured records the kernel that a session's later
calls run, also where the captured call is the session's first."""

import ctypes

import pytest

from parity import device_scene, lp_slots
from workloads import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth, pooled", [(0, False), (3, True)])
@pytest.mark.parametrize("full", [False, True])
def test_captured_kernel(V, torch_mod, tmp_path, depth, pooled, full):
    torch = torch_mod
    w = workload("random1k")
    h, keep = device_scene(V, w.scene, torch)
    s = V.vafr_session_create(V.make_session_desc(1280, 1024, 90.0, w.displays[0].poses))
    V.vafr_set_gaze(s, 0, 256.0, 256.0)
    _, n_slots, _, _ = lp_slots(V, s)
    out = torch.full((1280 * 1024 if full else n_slots, 4), -1.0, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        stream = torch.cuda.current_stream().cuda_stream
        if full:
            V.vafr_render_full_gt_pt(h, s, 0, out, 3, depth, stream)
        else:
            V.vafr_render_lp_pt(h, s, 1, out, 3, depth, None, stream)
    path = tmp_path / "graph.dot"
    dump = ctypes.CDLL("libcuda.so.1").cuGraphDebugDotPrint
    assert dump(ctypes.c_void_p(g.raw_cuda_graph()), str(path).encode(), ctypes.c_uint(1)) == 0
    dot = path.read_text()
    assert ("k_path_lanes" in dot) == (not pooled) and "k_path" in dot
    g.replay()
    torch.cuda.synchronize()
    replayed = out.clone()
    del g
    out.fill_(-1.0)
    if full:
        V.vafr_render_full_gt_pt(h, s, 0, out, 3, depth)
    else:
        V.vafr_render_lp_pt(h, s, 1, out, 3, depth)
    torch.cuda.synchronize()
    assert V.vafr_session_check(s) == 0
    assert torch.equal(out, replayed)
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)
