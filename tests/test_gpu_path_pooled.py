"""The pooled path tracer against one path per lane (a session's first call) bit for
bit, radiance and signatures, and against the FP64 oracle: both eyes in one
launch, FP16 and FP32, remainders of a warp, displays that are no multiple of the
pixel tiles, few paths with many bounces."""

import numpy as np
import pytest

import oracle
from parity import check_guards, device_scene, lp_slots
from test_gpu_path_pool import TOL, _allowed, _oracle_paths
from workloads import workload

pytestmark = pytest.mark.gpu

LINE = 2_500_000   # bounces x paths from which a session with scratch uses the pool


@pytest.mark.parametrize("e_max, eyes, depth, half", [(10.0, 2, 5, False), (10.0, 2, 5, True), (10.0, 1, 9, False),
                                                      (5.0, 2, 15, True), (60.0, 2, 2, True)])
def test_lp(V, torch_mod, e_max, eyes, depth, half):
    torch = torch_mod
    w = workload("random1k")
    sc, disp = w.scene, w.displays[0]
    h, keep = device_scene(V, sc, torch)
    poses = [disp.poses[0], disp.poses[0] + np.array([[0, 0, 0, 0.1]] * 3)][:eyes]
    acuity = V.make_acuity([0, 10, 20, 30, 60], [40, 10, 6, 5, 4], e_max_deg=e_max)
    s = V.vafr_session_create(V.make_session_desc(512, 512, 90.0, poses, int(half), 0, acuity=acuity))
    gazes = [(200.3, 260.7), (311.0, 222.2)][:eyes]
    for e, g in enumerate(gazes):
        V.vafr_set_gaze(s, e, *g)
    lay = oracle.lp_layout(e_max=e_max)
    assert depth * eyes * lay.total >= LINE
    slot, n_slots, counts, offs = lp_slots(V, s)
    got = []
    for _ in range(2):   # one path per lane, then the pool
        lp = torch.full((eyes, n_slots, 4), -1.0, dtype=torch.float16 if half else torch.float32, device="cuda")
        sig = torch.full((eyes, n_slots, depth + 2), -7, dtype=torch.int32, device="cuda")
        V.vafr_render_lp_pt(h, s, (1 << eyes) - 1, lp, 77, depth, sig)
        got.append((lp, sig))
    torch.cuda.synchronize()
    assert V.vafr_session_check(s) == 0
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    tol = TOL + (3 * 2.0 ** -11 if half else 0.0)   # FP16 storage of values up to 3
    for e in range(eyes):
        lp, sig = (x[e].float().cpu().numpy() if k == 0 else x[e].cpu().numpy() for k, x in enumerate(got[1]))
        check_guards(lp, counts, offs)
        tex = np.unique(np.concatenate([np.random.default_rng(e).choice(lay.total, 20000), np.arange(64),
                                        lay.total - 1 - np.arange(64)]))
        o, d, _ = oracle.lp_rays(lay, 512, 512, 90.0, gazes[e], poses[e], tex)
        ref, rsig = _oracle_paths(sc, o, d, tex, 77, depth)
        same = (sig[slot][tex] == rsig).all(1)
        assert (~same).sum() <= _allowed(len(tex), depth)
        assert np.abs(lp[slot][tex][same] - ref[same]).max() <= tol
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)


@pytest.mark.parametrize("width, height, depth", [(641, 301, 15), (1003, 517, 5), (1279, 721, 3)])
def test_full_resolution(V, torch_mod, width, height, depth):
    torch = torch_mod
    w = workload("random1k")
    sc, pose = w.scene, w.displays[0].poses[0]
    h, keep = device_scene(V, sc, torch)
    s = V.vafr_session_create(V.make_session_desc(width, height, 90.0, [pose]))
    assert depth * width * height >= LINE
    got = []
    for _ in range(2):   # one path per lane, then the pool
        got.append(torch.full((height, width, 4), -1.0, dtype=torch.float32, device="cuda"))
        V.vafr_render_full_gt_pt(h, s, 0, got[-1], 9, depth)
    torch.cuda.synchronize()
    assert V.vafr_session_check(s) == 0
    assert torch.equal(got[0], got[1])
    px = np.unique(np.concatenate([np.random.default_rng(width).choice(width * height, 20000), np.arange(64),
                                   width * height - 1 - np.arange(64)]))
    o, d = oracle.pixel_rays(width, height, 90.0, pose, px)
    ref, _ = _oracle_paths(sc, o, d, px, 9, depth)
    far = np.abs(got[1].cpu().numpy().reshape(-1, 4)[px] - ref).max(1) > TOL
    assert far.sum() <= _allowed(len(px), depth)
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)
