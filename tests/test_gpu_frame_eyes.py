"""A frame's eyes share each pass's launch: the display holds the bytes of one call
per eye and pass, for both formats, with and without FXAA, at odd sizes, over
frames of the longest-first order and captured into a graph."""

import numpy as np
import pytest

from parity import device_scene
from workloads import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width, height", [(64, 33), (203, 118), (129, 257)])
@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("fxaa", [False, True])
@pytest.mark.parametrize("variant", [0, 7])
def test_frame_equals_calls_per_eye(V, torch_mod, width, height, half, fxaa, variant):
    torch = torch_mod
    w = workload("random1k")
    h, keep = device_scene(V, w.scene, torch)
    pose = w.displays[0].poses[0]
    poses = [pose, pose + np.array([[0, 0, 0, 0.06]] + [[0, 0, 0, 0]] * 2)]
    fmt = V.FMT_RGBA16F if half else V.FMT_RGBA32F
    dt = torch.float16 if half else torch.float32
    s = V.vafr_session_create(V.make_session_desc(width, height, 80.0, poses, lp_format=fmt, display_format=fmt,
                                                  lp_fxaa=fxaa))
    V.vafr_session_tuning(s, (variant, 0))
    lpb, dpb = V.vafr_session_sizes(s)[:2]
    slots = lpb // (8 if half else 16)
    disp = torch.zeros((2, height, width, 4), dtype=dt, device="cuda")
    for frame in range(3):
        for e in range(2):
            V.vafr_set_gaze(s, e, 20.0 + 9 * frame + e, 16.5)
        if lpb % 16 or dpb % 16:   # the second eye's buffers would not be aligned
            with pytest.raises(V.VafrError):
                V.vafr_render_frame(h, s, disp)
            break
        if frame < 2:
            V.vafr_render_frame(h, s, disp)
        else:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                V.vafr_render_frame(h, s, disp, torch.cuda.current_stream().cuda_stream)
            disp.zero_()
            g.replay()
            g.replay()
        lp = torch.empty((2, slots, 4), dtype=dt, device="cuda")
        V.vafr_render_lp(h, s, 3, lp)
        ref = torch.zeros_like(disp)
        for e in range(2):
            src = lp[e]
            if fxaa:
                src = torch.empty_like(lp[e])
                V.vafr_fxaa_lp(s, e, lp[e], src)
            V.vafr_reconstruct(s, e, src, ref[e])
        torch.cuda.synchronize()
        assert torch.equal(disp, ref)
    assert V.vafr_session_check(s) == 0
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)
