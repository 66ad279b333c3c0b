"""Render variant 0 picks its kernel by the scene's size: on both sides of the
line, LP casts (first frame and after a few, when the longest-first order has a
history), full-resolution casts and VaFR_Rep give the bits of variant 2."""

import numpy as np
import pytest

from parity import device_scene
from workloads import random_triangles_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4096, 4097])
@pytest.mark.parametrize("eyes", [1, 2])
def test_same_bits_on_both_sides(V, torch_mod, n, eyes):
    torch = torch_mod
    sc = random_triangles_scene(n, seed=n)
    rng = np.random.default_rng(n)
    sc.tris[:] = rng.uniform(-1, 1, (n, 1, 3)).astype(np.float32) + np.float32(0.05) * sc.tris
    h, keep = device_scene(V, sc, torch)
    pose = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, -3.0]])
    poses = [pose, pose + np.array([[0, 0, 0, 0.06]] + [[0, 0, 0, 0]] * 2)][:eyes]
    out = {}
    for variant in (2, 0):
        s = V.vafr_session_create(V.make_session_desc(203, 117, 80.0, poses))
        V.vafr_session_tuning(s, (variant, 0))
        slots = V.vafr_session_sizes(s)[0] // 16
        res = []
        for frame in range(3):
            for e in range(eyes):
                V.vafr_set_gaze(s, e, 60.0 + 20 * frame + e, 50.5)
            lp = torch.empty((eyes, slots, 4), dtype=torch.float32, device="cuda")
            ids = torch.empty((eyes, slots), dtype=torch.int32, device="cuda")
            V.vafr_render_lp(h, s, (1 << eyes) - 1, lp, ids)
            res += [lp, ids]
            if eyes == 2:
                rep = torch.zeros_like(lp)
                V.vafr_render_lp_rep(h, s, rep)
                res.append(rep)
        gt = torch.empty((117, 203, 4), dtype=torch.float32, device="cuda")
        V.vafr_render_full_gt(h, s, 0, gt)
        res.append(gt)
        torch.cuda.synchronize()
        assert V.vafr_session_check(s) == 0
        V.vafr_session_destroy(s)
        out[variant] = res
    for a, b in zip(out[2], out[0]):
        assert torch.equal(a, b)
    V.vafr_scene_destroy(h)
