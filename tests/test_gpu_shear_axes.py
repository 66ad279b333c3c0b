"""The triangle test takes one of three shears by the ray's largest axis: views along
every axis and diagonal, where rays of all three meet, against the FP64 oracle,
for the casts and for the visibility buffer."""

import numpy as np
import pytest

import oracle
from parity import compare_hits_and_colours, device_scene
from workloads import random_triangles_scene
from workloads.views import look_at_pose

pytestmark = pytest.mark.gpu

VIEWS = [(1, 0, 0), (-1, 0, 0), (0, 1, 1e-3), (0, -1, 1e-3), (0, 0, 1), (0, 0, -1),
         (1, 1, 1), (-1, 1, 1), (1, -1, 1), (1, 1, -1)]


@pytest.mark.parametrize("view", VIEWS)
def test_views(V, torch_mod, view):
    torch = torch_mod
    sc = random_triangles_scene(3000, seed=11)
    lo, hi = sc.tris.reshape(-1, 3).min(0), sc.tris.reshape(-1, 3).max(0)
    centre, size = 0.5 * (lo + hi), float(np.linalg.norm(hi - lo))
    eye = centre - 0.6 * size * np.asarray(view, np.float64) / np.linalg.norm(view)
    pose = look_at_pose(tuple(eye), tuple(centre))
    w, hgt, fov = 160, 121, 95.0
    h, keep = device_scene(V, sc, torch)
    s = V.vafr_session_create(V.make_session_desc(w, hgt, fov, [pose]))
    out = torch.empty((hgt, w, 4), dtype=torch.float32, device="cuda")
    ids = torch.empty(hgt * w, dtype=torch.int32, device="cuda")
    V.vafr_render_full_gt(h, s, 0, out, ids)
    vbuf = torch.empty(hgt * w, dtype=torch.int64, device="cuda")
    V.vafr_render_vbuffer(h, s, 0, vbuf)
    torch.cuda.synchronize()
    assert V.vafr_session_check(s) == 0
    rgba, oid, ot, o, d = oracle.render_gt(sc.tris, sc.albedo, sc.light_dir, w, hgt, fov, pose)
    got = ids.cpu().numpy()
    compare_hits_and_colours(sc.tris, o, d, got, out.cpu().numpy().reshape(-1, 4), oid, ot, rgba, 1e-3, tie_budget=1e-3)
    key = vbuf.cpu().numpy()
    assert np.array_equal(np.where(key == -1, -1, key & 0xffffffff), got)
    V.vafr_session_destroy(s)
    V.vafr_scene_destroy(h)
