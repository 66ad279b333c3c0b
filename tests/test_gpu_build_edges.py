"""Scene build at the edges of its tiles: the refit's blocks of 512 leaves, the
clustering rounds' tiles of 488, the 2,048 clusters that one block finishes,
and more than 4,096 tiles, whose counts are scanned by a launch of their own."""

import ctypes

import numpy as np
import pytest

import oracle
from parity import device_scene
from test_gpu_lbvh import check_tree4
from workloads import random_triangles_scene

pytestmark = pytest.mark.gpu


def _soup(n, seed, size):
    """n triangles of the given size spread over the unit cube."""
    sc = random_triangles_scene(n, seed=seed)
    rng = np.random.default_rng(seed)
    sc.tris[:] = rng.uniform(-1, 1, (n, 1, 3)).astype(np.float32) + (size * sc.tris).astype(np.float32)
    return sc


def _check(V, torch, sc, lbvh=True):
    h, keep = device_scene(V, sc, torch)
    try:
        check_tree4(*V.vafr_scene_export_tree4(h), sc.tris.reshape(-1, 3, 3))
        if lbvh:
            codes, ids, child, nb, lb = V.vafr_scene_export_lbvh(h)
            ref = oracle.lbvh(sc.tris)
            assert np.array_equal(codes, ref.codes) and np.array_equal(ids, ref.sorted_ids)
            assert np.array_equal(child, ref.child)
            assert np.array_equal(nb.view(np.uint32), ref.node_box.view(np.uint32))
            assert np.array_equal(lb.view(np.uint32), ref.leaf_box.view(np.uint32))
    finally:
        V.vafr_scene_destroy(h)


@pytest.mark.parametrize("n", [2, 488, 489, 511, 512, 513, 1025, 2047, 2048, 2049, 2441, 4097, 9761])
def test_tile_edges(V, torch_mod, n):
    _check(V, torch_mod, _soup(n, n, 0.05))


@pytest.mark.parametrize("n", [2050, 30001])
def test_equal_boxes(V, torch_mod, n):
    """All clusters of a round are equal: every tie goes to the partner i ^ 1."""
    sc = _soup(n, 4, 0.05)
    sc.tris[:] = sc.tris[:1]
    _check(V, torch_mod, sc)


def test_more_tiles_than_a_block_sums(V, torch_mod):
    _check(V, torch_mod, _soup(4096 * 488 + 12345, 6, 0.003), lbvh=False)


def test_binary_tree_casts_the_same_hits(V, torch_mod):
    """The radix tree's two-child nodes (render variant 3) and the 4-wide ones
    give the same hits, bit for bit."""
    torch = torch_mod
    sc = _soup(20000, 8, 0.05)
    h, keep = device_scene(V, sc, torch)
    pose = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, -3.0]])
    s = V.vafr_session_create(V.make_session_desc(640, 480, 70.0, [pose]))
    V.vafr_set_gaze(s, 0, 320.0, 240.0)
    slots = V.vafr_session_sizes(s)[0] // 16
    out = []
    for variant in (0, 3):
        V.vafr_session_tuning(s, (variant, 0))
        lp = torch.empty((slots, 4), dtype=torch.float32, device="cuda")
        ids = torch.empty(slots, dtype=torch.int32, device="cuda")
        V.vafr_render_lp(h, s, 1, lp, ids)
        out.append((lp, ids))
    torch.cuda.synchronize()
    assert V.vafr_session_check(s) == 0
    assert (out[0][1] >= 0).any()
    assert torch.equal(out[0][1], out[1][1]) and torch.equal(out[0][0], out[1][0])
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 4, 8])
def test_device_inputs_at_any_address(V, torch_mod, shift):
    """Triangles and albedo in device memory at any byte address build the tree of
    host inputs."""
    torch = torch_mod
    sc = _soup(1000, 9, 0.05)
    light = (ctypes.c_float * 3)(*[float(v) for v in sc.light_dir])
    ref = V.vafr_build_scene(sc.tris.reshape(-1, 9), sc.albedo, sc.light_dir)
    held = []
    for x in (sc.tris, sc.albedo):
        raw = torch.from_numpy(np.frombuffer(np.ascontiguousarray(x, np.float32).tobytes(), np.uint8).copy())
        buf = torch.zeros(raw.numel() + 16, dtype=torch.uint8, device="cuda")
        buf[shift:shift + raw.numel()] = raw.cuda()
        held.append(buf)
    torch.cuda.synchronize()
    out = ctypes.c_void_p()
    lib = V.load()
    assert lib.vafr_build_scene(held[0].data_ptr() + shift, held[1].data_ptr() + shift, 1000,
                                ctypes.cast(light, ctypes.c_void_p), None, ctypes.byref(out)) == 0
    for a, b in zip(V.vafr_scene_export_tree4(ref), V.vafr_scene_export_tree4(out.value)):
        assert np.array_equal(a.view(np.int32), b.view(np.int32))
    V.vafr_scene_destroy(ref)
    V.vafr_scene_destroy(out.value)
