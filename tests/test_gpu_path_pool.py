"""The path tracer at the edges of its work: fewer paths than a warp,
remainders, odd displays, both eyes in one launch, no and many bounces, on both
sides of the line between one path per lane and the pool of waiting paths
(bounces x paths >= 2.5 M), against the FP64 oracle."""

import numpy as np
import pytest

import oracle
from parity import device_scene, lp_slots
from workloads import workload

pytestmark = pytest.mark.gpu

# FP32 radiance of a few bounces with albedo <= 1 and a unit light: the bound the
# whole-buffer path tests use
TOL = 1e-4


def _oracle_paths(sc, o, d, keys, seed, depth):
    bvh = oracle.CpuBVH(sc.tris)
    rgba, sig = np.empty((len(keys), 4)), np.empty((len(keys), depth + 2), np.int32)
    keys = np.ascontiguousarray(keys, np.int64)
    light = np.ascontiguousarray(sc.light_dir, np.float64)
    alb = np.ascontiguousarray(sc.albedo, np.float32)
    oracle.lib().or_path_trace(bvh.h, oracle._p(alb), oracle._p(light), oracle._p(o), oracle._p(d), oracle._p(keys),
                               len(keys), seed, depth, oracle._p(rgba), oracle._p(sig), None)
    return rgba, sig


def _allowed(n, depth):
    """Paths that a ray-edge tie may change: 0.01 % of the rays, and at least two."""
    return 2 + int(1e-4 * n * 2 * (depth + 1))


@pytest.mark.parametrize("e_max, depth", [(0.15, 3), (0.5, 1), (1.0, 0), (3.0, 4), (10.0, 2)])
def test_small_lp_layouts(V, torch_mod, e_max, depth):
    torch = torch_mod
    w = workload("random1k")
    sc, disp = w.scene, w.displays[0]
    h, keep = device_scene(V, sc, torch)
    acuity = V.make_acuity([0, 10, 20, 30, 60], [40, 10, 6, 5, 4], e_max_deg=e_max)
    poses = [disp.poses[0], disp.poses[0] + np.array([[0, 0, 0, 0.1]] * 3)]
    s = V.vafr_session_create(V.make_session_desc(512, 512, 90.0, poses, acuity=acuity))
    gazes = [(200.3, 260.7), (311.0, 222.2)]
    for e, g in enumerate(gazes):
        V.vafr_set_gaze(s, e, *g)
    lay = oracle.lp_layout(e_max=e_max)
    slot, n_slots, _, _ = lp_slots(V, s)
    lp = torch.zeros((2, n_slots, 4), dtype=torch.float32, device="cuda")
    sig = torch.full((2, n_slots, depth + 2), -7, dtype=torch.int32, device="cuda")
    for _ in range(2):   # the second call has the pool's scratch
        V.vafr_render_lp_pt(h, s, 3, lp, 77, depth, sig)
    torch.cuda.synchronize()
    assert V.vafr_session_check(s) == 0
    for e in range(2):
        o, d, _ = oracle.lp_rays(lay, 512, 512, 90.0, gazes[e], poses[e])
        ref, rsig = _oracle_paths(sc, o, d, np.arange(lay.total), 77, depth)
        got, gsig = lp[e].cpu().numpy()[slot], sig[e].cpu().numpy()[slot]
        same = (gsig == rsig).all(1)
        assert (~same).sum() <= _allowed(lay.total, depth)
        assert np.abs(got[same] - ref[same]).max() <= TOL
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)


@pytest.mark.parametrize("width, height, depth", [(1240, 1000, 2), (1256, 1000, 2), (1781, 707, 2)])
def test_both_kernels_around_their_line(V, torch_mod, width, height, depth):
    torch = torch_mod
    w = workload("random1k")
    sc, pose = w.scene, w.displays[0].poses[0]
    h, keep = device_scene(V, sc, torch)
    s = V.vafr_session_create(V.make_session_desc(width, height, 90.0, [pose]))
    out = torch.full((height, width, 4), -1.0, dtype=torch.float32, device="cuda")
    for _ in range(2):   # the second call has the pool's scratch
        V.vafr_render_full_gt_pt(h, s, 0, out, 9, depth)
    torch.cuda.synchronize()
    assert V.vafr_session_check(s) == 0
    px = np.sort(np.random.default_rng(width).choice(width * height, 20000, replace=False))
    px = np.unique(np.concatenate([px, np.arange(64), width * height - 1 - np.arange(64)]))
    o, d = oracle.pixel_rays(width, height, 90.0, pose, px)
    ref, _ = _oracle_paths(sc, o, d, px, 9, depth)
    far = np.abs(out.cpu().numpy().reshape(-1, 4)[px] - ref).max(1) > TOL
    assert far.sum() <= _allowed(len(px), depth)
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)


def test_many_bounces_keep_the_first_segments(V, torch_mod):
    """The random numbers of a bounce depend on the texel and the bounce alone:
    at 15 bounces the first segments are those of 4 bounces, bit for bit."""
    torch = torch_mod
    w = workload("random1k")
    h, keep = device_scene(V, w.scene, torch)
    s = V.vafr_session_create(V.make_session_desc(512, 512, 90.0, w.displays[0].poses))
    V.vafr_set_gaze(s, 0, 256.0, 256.0)
    slot, n_slots, _, _ = lp_slots(V, s)
    sigs = []
    for depth in (4, 15):
        lp = torch.empty((n_slots, 4), dtype=torch.float32, device="cuda")
        sig = torch.full((n_slots, depth + 2), -7, dtype=torch.int32, device="cuda")
        for _ in range(2):   # the second call has the pool's scratch
            V.vafr_render_lp_pt(h, s, 1, lp, 3, depth, sig)
        sigs.append(sig.cpu().numpy()[slot])
    assert V.vafr_session_check(s) == 0
    assert np.array_equal(sigs[0][:, :5], sigs[1][:, :5])
    bits = 0x1f | 0x1f << 16
    assert np.array_equal(sigs[0][:, -1] & bits, sigs[1][:, -1] & bits)
    assert (sigs[1][:, 15] >= 0).any()
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)


@pytest.mark.parametrize("width, height", [(1, 1), (5, 3), (37, 21), (130, 64)])
def test_odd_displays(V, torch_mod, width, height):
    torch = torch_mod
    w = workload("random1k")
    sc, pose = w.scene, w.displays[0].poses[0]
    h, keep = device_scene(V, sc, torch)
    s = V.vafr_session_create(V.make_session_desc(width, height, 90.0, [pose]))
    out = torch.full((height, width, 4), -1.0, dtype=torch.float32, device="cuda")
    for _ in range(2):   # the second call has the pool's scratch
        V.vafr_render_full_gt_pt(h, s, 0, out, 9, 2)
    torch.cuda.synchronize()
    assert V.vafr_session_check(s) == 0
    o, d = oracle.pixel_rays(width, height, 90.0, pose)
    ref, _ = _oracle_paths(sc, o, d, np.arange(width * height), 9, 2)
    far = np.abs(out.cpu().numpy().reshape(-1, 4) - ref).max(1) > TOL
    assert far.sum() <= _allowed(width * height, 2)
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)


@pytest.mark.parametrize("depth", [0, 4])
def test_first_call_inside_a_capture(V, torch_mod, depth):
    """A session's first path tracing call may be captured: replays give the
    bits of a direct call, on either side of the line between the kernels."""
    torch = torch_mod
    w = workload("random1k")
    h, keep = device_scene(V, w.scene, torch)
    bufs = []
    for captured in (False, True):
        s = V.vafr_session_create(V.make_session_desc(512, 512, 90.0, w.displays[0].poses))
        V.vafr_set_gaze(s, 0, 256.0, 256.0)
        slot, n_slots, _, _ = lp_slots(V, s)
        lp = torch.full((n_slots, 4), -1.0, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                V.vafr_render_lp_pt(h, s, 1, lp, 3, depth, None, torch.cuda.current_stream().cuda_stream)
            assert (lp == -1.0).all()
            for _ in range(2):
                lp.fill_(-1.0)
                g.replay()
            torch.cuda.synchronize()
        else:
            for _ in range(2):   # the second call has the pool's scratch
                V.vafr_render_lp_pt(h, s, 1, lp, 3, depth)
        torch.cuda.synchronize()
        assert V.vafr_session_check(s) == 0
        bufs.append(lp.cpu().numpy()[slot])
        if captured:
            del g
        V.vafr_session_destroy(s)
    assert np.array_equal(bufs[0].view(np.int32), bufs[1].view(np.int32))
    V.vafr_scene_destroy(h)
