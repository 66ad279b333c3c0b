"""The rasteriser at the edges of its work split (warps with one triangle or
32, boxes on either side of the tile pass's limit, displays narrower than a
tile) equals the full-resolution cast's closest hits, bit for bit."""

import numpy as np
import pytest

from parity import device_scene
from workloads import random_triangles_scene

pytestmark = pytest.mark.gpu

POSE = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, -3.0]])


@pytest.mark.parametrize("width, height", [(1, 1), (15, 7), (17, 9), (333, 191), (1280, 720)])
@pytest.mark.parametrize("n, size", [(1, 1.0), (31, 0.5), (33, 0.02), (5000, 0.03), (40000, 0.01)])
def test_equals_the_cast(V, torch_mod, width, height, n, size):
    torch = torch_mod
    sc = random_triangles_scene(n, seed=n)
    rng = np.random.default_rng(n + width)
    sc.tris[:] = rng.uniform(-1, 1, (n, 1, 3)).astype(np.float32) + np.float32(size) * sc.tris
    h, keep = device_scene(V, sc, torch)
    s = V.vafr_session_create(V.make_session_desc(width, height, 50.0, [POSE]))
    vbuf = torch.full((height, width), 5, dtype=torch.int64, device="cuda")
    again = torch.zeros_like(vbuf)
    V.vafr_render_vbuffer(h, s, 0, vbuf)
    stats = V.vafr_vbuffer_stats(h, s, 0, again)
    rgba = torch.empty((height, width, 4), dtype=torch.float32, device="cuda")
    ids = torch.empty((height, width), dtype=torch.int32, device="cuda")
    V.vafr_render_full_gt(h, s, 0, rgba, ids)
    torch.cuda.synchronize()
    assert V.vafr_session_check(s) == 0
    got = torch.where(vbuf == -1, torch.full_like(vbuf, -1), vbuf & 0xFFFFFFFF).int()
    assert torch.equal(got, ids)
    assert torch.equal(vbuf, again)
    assert stats["prefilter"] >= stats["filtered"] >= stats["tests"] >= stats["atomics"] >= int((ids >= 0).sum())
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)


def test_first_call_inside_a_capture(V, torch_mod):
    """A scene's first visibility buffer and shading may be captured; eager calls
    before and after the replay give the bits of an uncaptured scene."""
    torch = torch_mod
    sc = random_triangles_scene(500, seed=3)
    pose = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, -3.0]])
    out = []
    for captured in (False, True):
        h, keep = device_scene(V, sc, torch)
        s = V.vafr_session_create(V.make_session_desc(200, 150, 70.0, [pose]))
        V.vafr_set_gaze(s, 0, 90.0, 70.0)
        slots = V.vafr_session_sizes(s)[0] // 16
        vbuf = torch.zeros(200 * 150, dtype=torch.int64, device="cuda")
        lp = torch.zeros((slots, 4), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()

        def frame(stream=None):
            V.vafr_render_vbuffer(h, s, 0, vbuf, stream)
            V.vafr_shade_lp_deferred(h, s, 0, vbuf, lp, stream)

        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                frame(torch.cuda.current_stream().cuda_stream)
            frame()
            torch.cuda.synchronize()
            out.append((vbuf.clone(), lp.clone()))
            vbuf.zero_()
            lp.zero_()
            g.replay()
        else:
            frame()
        torch.cuda.synchronize()
        assert V.vafr_session_check(s) == 0
        out.append((vbuf.clone(), lp.clone()))
        V.vafr_session_destroy(s)
        V.vafr_scene_destroy(h)
    assert (out[0][0] != -1).any()
    for vb, lp in out[1:]:
        assert torch.equal(vb, out[0][0]) and torch.equal(lp, out[0][1])
