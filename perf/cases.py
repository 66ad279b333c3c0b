"""Performance cases of the renderer: what a user's program has it do.

Each case goes through the public entry points of ``paper_2503_23410_gb300.vafr``
on inputs made from a seed: a triangle scene (random soup, or an fBm terrain
with boxes and spheres), a display with its pose(s), and a gaze point per eye.

kinds
  frame        vafr_render_frame: LP cast of every eye, FXAA if asked for, and
               reconstruction, into a device display
  cast         vafr_render_lp with hit ids
  reconstruct  vafr_reconstruct of one eye from a given LP buffer
  fxaa         vafr_fxaa_lp of one eye's LP buffer
  batch        several binocular sessions in one vafr_batch_render (or the
               replay of a captured graph), as the serving loop does
  gt           vafr_render_full_gt: one ray per display pixel, with hit ids
  pathtrace    vafr_render_lp_pt
  rep          vafr_render_lp_rep: right eye warped from the left
  deferred     vafr_render_vbuffer, then vafr_shade_lp_deferred
  build        vafr_build_scene and the first cast of the new scene
"""

import math

import numpy as np
import torch

from paper_2503_23410_gb300 import vafr as V

DEV = "cuda"
LIGHT = (-0.4, -1.0, 0.6)
TERRAIN = {"scene": "terrain", "nx": 512, "nz": 1024, "boxes": 2000, "spheres": 0}     # 1,069,506 triangles
OBJECTS = {"scene": "terrain", "nx": 829, "nz": 1024, "boxes": 4000, "spheres": 4000}  # 1,998,088 triangles
EXTENT = (200.0, 400.0)
SERVED = ((1920, 1080), (2560, 1440), (3840, 2160), (7680, 4320))   # displays of the served mix


def listed():
    return [
        # a small scene on a small display: a whole frame whose launches are short
        {"name": "frame_512", "kind": "frame", "scene": "random", "tris": 1024, "width": 512, "height": 512,
         "fov": 90.0, "eyes": 1, "half": False, "acuity": "paper", "fxaa": False, "tuned": False},
        # the headline: binocular 8K frames of a 2 M triangle scene, half-precision buffers, autotuned
        {"name": "frame_8k_binocular", "kind": "frame", **OBJECTS, "width": 7680, "height": 4320, "fov": 100.0,
         "eyes": 2, "half": True, "acuity": "paper", "fxaa": False, "tuned": True},
        # the LP cast alone on a 4K display (1 M triangles, FP32, with hit ids)
        {"name": "cast_4k", "kind": "cast", **TERRAIN, "width": 3840, "height": 2160, "fov": 100.0, "eyes": 1,
         "half": False, "acuity": "paper"},
        # the inverse mapping alone, 4K FP32 and one 8K FP16 eye
        {"name": "reconstruct_4k", "kind": "reconstruct", "width": 3840, "height": 2160, "fov": 100.0,
         "half": False, "acuity": "paper"},
        {"name": "reconstruct_8k_half", "kind": "reconstruct", "width": 7680, "height": 4320, "fov": 100.0,
         "half": True, "acuity": "paper"},
        # anti-aliasing inside the LP buffer
        {"name": "fxaa", "kind": "fxaa", "half": False, "acuity": "paper"},
        # a step of the serving loop: eight binocular sessions from 1080p to 8K in one batch
        {"name": "batch_served_mix", "kind": "batch", **TERRAIN, "sessions": 8, "first": 0, "graph": False},
        # the full-resolution cast that foveated frames are compared with
        {"name": "gt_1440p", "kind": "gt", **TERRAIN, "width": 2560, "height": 1440, "fov": 100.0, "half": False},
        # one path per LP texel, three diffuse bounces
        {"name": "pathtrace_4k", "kind": "pathtrace", **TERRAIN, "width": 3840, "height": 2160, "fov": 100.0,
         "eyes": 1, "half": False, "acuity": "paper", "depth": 3},
        # the right eye warped from the left one, holes cast
        {"name": "rep_8k", "kind": "rep", **OBJECTS, "width": 7680, "height": 4320, "fov": 100.0, "half": True,
         "acuity": "paper"},
        # native-resolution visibility buffer, lighting by 31 point lights in the LP buffer
        {"name": "deferred_4k", "kind": "deferred", **TERRAIN, "width": 3840, "height": 2160, "fov": 100.0,
         "half": False, "acuity": "paper", "lights": 31},
        # a new scene (loaded, or rebuilt because its geometry moved) and its first cast
        {"name": "build_1m", "kind": "build", **TERRAIN, "width": 3840, "height": 2160, "fov": 100.0, "half": False},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["frame", "cast", "reconstruct", "fxaa", "batch", "gt", "pathtrace", "rep", "deferred",
                       "build"])
    c = {"kind": kind}
    width = _log_int(rng, 320, 3840 if kind in ("gt", "deferred") else 7680)
    height = max(180, int(width * rng.uniform(0.5, 0.6)))
    display = {"width": width, "height": height, "fov": round(rng.uniform(80.0, 110.0), 1),
               "half": rng.random() < 0.5}
    acuity = {"acuity": rng.choice(["paper", "anisotropic", "display"])}
    nx = _log_int(rng, 40, 512)
    nz = _log_int(rng, 80, 1024)
    terrain = {"scene": "terrain", "nx": nx, "nz": nz, "boxes": _log_int(rng, 20, 2000),
               "spheres": _log_int(rng, 10, 200)}
    soup = {"scene": "random", "tris": _log_int(rng, 1, 4096)}
    if kind == "frame":
        c.update(rng.choice([terrain, soup]), **display, **acuity, eyes=rng.choice([1, 2]),
                 fxaa=rng.random() < 0.5, tuned=rng.random() < 0.5)
    elif kind == "cast":
        c.update(rng.choice([terrain, soup]), **display, **acuity, eyes=rng.choice([1, 2]))
    elif kind == "reconstruct":
        c.update(**display, **acuity)
    elif kind == "fxaa":
        c.update(half=display["half"], seam=rng.randrange(1 << 16), **acuity)
    elif kind == "batch":
        c.update(terrain, sessions=rng.randint(1, 8), first=rng.randrange(len(SERVED)), graph=rng.random() < 0.5)
    elif kind == "gt":
        c.update(rng.choice([terrain, soup]), **display)
    elif kind == "pathtrace":
        c.update(terrain, **display, **acuity, eyes=1, depth=rng.randint(0, 3))
    elif kind == "rep":
        c.update(terrain, **display, **acuity)
    elif kind == "deferred":
        c.update(terrain, **display, **acuity, lights=rng.choice([0, 1, 8, 31]))
    else:
        c.update(rng.choice([terrain, soup]), **display)
    return c


# ---- inputs --------------------------------------------------------------------------

class _Owned:
    """Library handles that live as long as the state that holds them."""

    def __init__(self):
        self.handles = []

    def take(self, destroy, handle):
        self.handles.append((destroy, handle))
        return handle

    def __del__(self):
        for destroy, handle in reversed(self.handles):
            destroy(handle)


def _rng(seed, salt):
    return np.random.default_rng([int(seed), salt])


def _heights(case, seed):
    """fBm value-noise heights (nz, nx) of the terrain, 20 m amplitude."""
    rng = _rng(seed, 1)
    ex, ez = EXTENT
    xs = torch.linspace(-ex / 2, ex / 2, case["nx"], dtype=torch.float64, device=DEV)
    zs = torch.linspace(-ez / 2, ez / 2, case["nz"], dtype=torch.float64, device=DEV)
    h = torch.zeros(case["nz"], case["nx"], dtype=torch.float64, device=DEV)
    freq, amp, norm = 1.0 / 80.0, 1.0, 0.0
    for _ in range(6):
        lat = torch.from_numpy(rng.uniform(-1.0, 1.0, (256, 256))).to(DEV)
        x, z = xs * freq + 17.0, zs * freq + 31.0
        xi, zi = x.floor(), z.floor()
        fx, fz = x - xi, z - zi
        sx = (fx * fx * fx * (fx * (fx * 6 - 15) + 10))[None, :]
        sz = (fz * fz * fz * (fz * (fz * 6 - 15) + 10))[:, None]
        x0, z0 = (xi.long() % 256)[None, :], (zi.long() % 256)[:, None]
        x1, z1 = (x0 + 1) % 256, (z0 + 1) % 256
        h += amp * ((lat[x0, z0] * (1 - sx) + lat[x1, z0] * sx) * (1 - sz) +
                    (lat[x0, z1] * (1 - sx) + lat[x1, z1] * sx) * sz)
        norm += amp
        freq *= 2.0
        amp *= 0.5
    return h / norm * 20.0


def _box():
    v = np.array([[-1, 0, -1], [1, 0, -1], [1, 0, 1], [-1, 0, 1], [-1, 2, -1], [1, 2, -1], [1, 2, 1], [-1, 2, 1]],
                 np.float64) * 0.5
    f = [(0, 1, 2), (0, 2, 3), (4, 6, 5), (4, 7, 6), (0, 4, 5), (0, 5, 1), (1, 5, 6), (1, 6, 2), (2, 6, 7),
         (2, 7, 3), (3, 7, 4), (3, 4, 0)]
    return v[np.array(f)]


def _sphere(slices=8, stacks=5):
    def p(i, j):
        th, ph = math.pi * i / stacks, 2 * math.pi * j / slices
        return (0.5 * math.sin(th) * math.cos(ph), 0.5 * (math.cos(th) + 1.0), 0.5 * math.sin(th) * math.sin(ph))
    tris = []
    for i in range(stacks):
        for j in range(slices):
            a, b, c, d = p(i, j), p(i, j + 1), p(i + 1, j + 1), p(i + 1, j)
            if i < stacks - 1:
                tris.append((a, c, d))
            if i > 0:
                tris.append((a, b, c))
    return np.array(tris, np.float64)


def _instances(proto, n, smax, rng, h):
    ex, ez = EXTENT
    px, pz = rng.uniform(-0.475 * ex, 0.475 * ex, n), rng.uniform(-0.475 * ez, 0.475 * ez, n)
    s, yaw = rng.uniform(1.0, smax, n), rng.uniform(0.0, 2 * math.pi, n)
    iz = np.rint((pz / ez + 0.5) * (h.shape[0] - 1)).astype(np.int64)
    ix = np.rint((px / ex + 0.5) * (h.shape[1] - 1)).astype(np.int64)
    py = h[iz, ix] - 0.1 * s
    v = proto[None] * s[:, None, None, None]
    c, q = np.cos(yaw)[:, None, None], np.sin(yaw)[:, None, None]
    out = np.stack([c * v[..., 0] + q * v[..., 2] + px[:, None, None], v[..., 1] + py[:, None, None],
                    c * v[..., 2] - q * v[..., 0] + pz[:, None, None]], -1)
    return out.reshape(-1, 3, 3)


def _scene_inputs(case, seed):
    """(triangles (n, 9), albedo (n, 3), both FP32 on the device; camera pose (3, 4))."""
    if case["scene"] == "random":
        rng = _rng(seed, 2)
        tris = torch.from_numpy(rng.uniform(-1.0, 1.0, (case["tris"], 9)).astype(np.float32)).to(DEV)
        alb = torch.from_numpy(rng.uniform(0.2, 1.0, (case["tris"], 3)).astype(np.float32)).to(DEV)
        pose = np.zeros((3, 4))
        pose[:, :3] = np.eye(3)
        pose[2, 3] = -3.0
        return tris, alb, pose
    h = _heights(case, seed)
    nz, nx = h.shape
    ex, ez = EXTENT
    xs = torch.linspace(-ex / 2, ex / 2, nx, dtype=torch.float64, device=DEV)
    zs = torch.linspace(-ez / 2, ez / 2, nz, dtype=torch.float64, device=DEV)
    v = torch.stack([xs[None, :].expand(nz, nx), h, zs[:, None].expand(nz, nx)], -1)
    a, b, c, d = v[:-1, :-1], v[:-1, 1:], v[1:, 1:], v[1:, :-1]
    ground = torch.stack([torch.stack([a, b, c], -2), torch.stack([a, c, d], -2)], 2).reshape(-1, 9).float()
    rng = _rng(seed, 3)
    hn = h.cpu().numpy()
    parts, colours = [ground], []
    g = torch.from_numpy(rng.normal(0.0, 0.05, (4096, 3)).astype(np.float32)).to(DEV)
    rep = g[torch.arange(ground.shape[0], device=DEV) * 2654435761 % 4096]
    colours.append((torch.tensor([0.35, 0.55, 0.25], device=DEV) + rep).clamp(0.2, 1.0))
    for proto, n, smax in ((_sphere(), case["spheres"], 6.0), (_box(), case["boxes"], 8.0)):
        if n:
            parts.append(torch.from_numpy(_instances(proto, n, smax, rng, hn).reshape(-1, 9).astype(np.float32)).to(DEV))
            col = torch.from_numpy(rng.uniform(0.2, 1.0, (n, 3)).astype(np.float32)).to(DEV)
            colours.append(col.repeat_interleave(len(proto), 0))
    z0 = -ez / 2 + 20.0
    y0 = float(hn[int(round((z0 / ez + 0.5) * (nz - 1))), nx // 2])
    fwd = np.array([0.0, -10.0, 60.0]) / math.hypot(10.0, 60.0)
    right = np.array([1.0, 0.0, 0.0])
    pose = np.stack([right, np.cross(fwd, right), fwd, np.array([0.0, y0 + 10.0, z0])], 1)
    return torch.cat(parts), torch.cat(colours), pose


def _eyes(pose, eyes):
    if eyes == 1:
        return [pose]
    left, right = pose.copy(), pose.copy()
    left[:, 3] -= pose[:, 0] * 0.0315
    right[:, 3] += pose[:, 0] * 0.0315
    return [left, right]


def _gaze(seed, salt, width, height, eyes):
    """Gaze points of the eyes: within the middle 70 % of the display, a few pixels apart."""
    rng = _rng(seed, salt)
    x, y = rng.uniform(0.15, 0.85) * width, rng.uniform(0.15, 0.85) * height
    return [(x + e * rng.uniform(-0.01, 0.01) * width, y + e * rng.uniform(-0.01, 0.01) * height)
            for e in range(eyes)]


def _acuity(name):
    if name == "anisotropic":
        return V.vafr_acuity_anisotropic()
    if name == "display":
        return V.vafr_acuity_display_limited(12.0)
    return V.vafr_acuity_default()


def _fmt(half):
    return V.FMT_RGBA16F if half else V.FMT_RGBA32F


def _pixels(half, *shape):
    return torch.empty(*shape, 4, dtype=torch.float16 if half else torch.float32, device=DEV)


def _session(own, case, poses, fxaa=False):
    half = case["half"]
    d = V.make_session_desc(case["width"], case["height"], case["fov"], poses, _fmt(half), _fmt(half),
                            acuity=_acuity(case.get("acuity", "paper")), lp_fxaa=fxaa)
    return own.take(V.vafr_session_destroy, V.vafr_session_create(d))


def _slots(session, half):
    return V.vafr_session_sizes(session)[0] // (8 if half else 16)


# ---- the log-polar layout and forward map in FP64 (inputs and exact results) ---------

class _Layout:
    def __init__(self, acuity):
        E = np.array([0.0, 10.0, 20.0, 30.0, 60.0])
        f = np.array([40.0, 10.0, 6.0, 5.0, 4.0])
        if acuity == "display":
            f = np.minimum(f, 12.0)
        delta = np.array([1.0, 5 / 6, 2 / 3, 0.5, 0.5]) if acuity == "anisotropic" else np.ones(5)
        self.e_max = 60.0
        w = 1.0 / f
        self.E, self.w, self.m = E[:-1], w[:-1], np.diff(w) / np.diff(E)
        self.U = np.concatenate([[0.0], np.cumsum([self._du(i, E[i + 1] - E[i]) for i in range(4)])])[:4]
        u_max = float(self.u_of_e(np.array([self.e_max]))[0])
        self.n_cols = int(math.ceil(u_max - 0.5))
        e = self.e_of_u(np.arange(self.n_cols) + 0.5)
        i = self._seg(e)
        l = 360.0 * np.sin(np.radians(2 * e)) / (self.m[i] * e + self.w[i] - self.m[i] * self.E[i])
        self.n = np.maximum(1, np.floor(np.interp(e, E, delta) * l + 0.5)).astype(np.int64)
        self.off = np.concatenate([[0], np.cumsum(self.n + 2)[:-1]]) + 1
        self.slots = int((self.n + 2).sum())
        self.e = e

    def _seg(self, e):
        return np.clip(np.searchsorted(self.E, e, side="right") - 1, 0, 3)

    def _du(self, i, de):
        return 2 * de / self.w[i] if self.m[i] == 0 else 2 / self.m[i] * math.log1p(self.m[i] * de / self.w[i])

    def e_of_u(self, u):
        i = np.clip(np.searchsorted(self.U, u, side="right") - 1, 0, 3)
        m, w, du = self.m[i], self.w[i], u - self.U[i]
        safe = np.where(m == 0, 1.0, m)
        return self.E[i] + np.where(m == 0, du * w / 2, np.expm1(m * du / 2) * w / safe)

    def u_of_e(self, e):
        """e: numpy array or torch tensor, degrees."""
        if isinstance(e, np.ndarray):
            return self.u_of_e(torch.from_numpy(e)).numpy()
        E, m, w, U = (torch.from_numpy(np.ascontiguousarray(a)).to(e.device) for a in (self.E, self.m, self.w, self.U))
        i = (torch.searchsorted(E, e.contiguous(), right=True) - 1).clamp(0, 3)
        mi, wi, de = m[i], w[i], e - E[i]
        safe = torch.where(mi == 0, torch.ones_like(mi), mi)
        return U[i] + torch.where(mi == 0, 2 * de / wi, 2 / safe * torch.log1p(mi * de / wi))

    def device(self):
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
        col = torch.repeat_interleave(torch.arange(self.n_cols, device=DEV), t(self.n + 2))
        j = torch.arange(self.slots, device=DEV) - t(self.off)[col]
        return t(self.n), t(self.off), t(self.e), col, j % t(self.n)[col]     # guards wrap


def _lp_image(case, seed):
    """A rendered-looking LP buffer: sky above a noisy horizon, shaded patches with hard edges below."""
    n, _, e, col, row = _Layout(case["acuity"]).device()
    rng = _rng(seed, 5)
    te = torch.tan(torch.deg2rad(e))[col]
    ph = 2 * math.pi * (row + 0.5) / n[col]
    x, y = te * torch.cos(ph), -te * torch.sin(ph)
    cells = torch.from_numpy(rng.uniform(0.05, 1.0, (64, 64, 3))).to(DEV)
    k = 4.0 + 12.0 * rng.random() + case.get("seam", 0) / 65536.0
    horizon = 0.1 * torch.sin(3.0 * x + rng.uniform(0, 6)) + rng.uniform(-0.2, 0.2)
    depth = 1.0 / (horizon - y).clamp(min=0.02)
    ground = cells[(x * depth * k).floor().long() % 64, (depth * k).floor().long() % 64]
    grain = torch.from_numpy(rng.normal(0.0, 0.02, (65536, 1))).to(DEV)
    ground = ground * (0.9 + grain[(97 * row + 31 * col) % 65536])
    s = 0.5 + 0.5 * y / torch.sqrt(x * x + y * y + 1.0)
    sky = torch.stack([1.0 - 0.5 * s, 1.0 - 0.3 * s, torch.ones_like(s)], -1)
    rgb = torch.where((y > horizon)[:, None], sky, ground)
    lp = torch.ones(len(col), 4, dtype=torch.float64, device=DEV)
    lp[:, :3] = rgb
    return lp.to(torch.float16 if case["half"] else torch.float32)


# ---- the cases -----------------------------------------------------------------------

def prepare(case, seed):
    own = _Owned()
    kind = case["kind"]
    st = {"case": case, "own": own}
    if kind in ("reconstruct", "fxaa"):
        size = {"width": 1920, "height": 1080, "fov": 100.0, **case}
        pose = np.eye(4)[:3]
        st["session"] = _session(own, size, [pose])
        st["lp"] = _lp_image(case, seed)
        if kind == "fxaa":
            st["out"] = torch.empty_like(st["lp"])
        else:
            st["gaze"] = _gaze(seed, 4, case["width"], case["height"], 1)
            st["out"] = _pixels(case["half"], case["height"], case["width"])
        return st
    tris, alb, pose = _scene_inputs(case, seed)
    if kind == "build":
        st["tris"], st["albedo"] = tris, alb
        scene = None
    else:
        scene = st["scene"] = own.take(V.vafr_scene_destroy, V.vafr_build_scene(tris, alb, LIGHT))
    if kind == "batch":
        st["sessions"], st["frames"], st["gaze"] = [], [], []
        for k in range(case["sessions"]):
            w, h = SERVED[(case["first"] + k) % len(SERVED)]
            c = {"width": w, "height": h, "fov": 100.0, "half": True}
            s = _session(own, c, _eyes(pose, 2))
            lp, disp = _pixels(True, 2, _slots(s, True)), _pixels(True, 2, h, w)
            gaze = _gaze(seed, 100 + k, w, h, 2)
            for e in range(2):
                V.vafr_set_gaze(s, e, *gaze[e])
                st["frames"].append((s, e, lp[e], disp[e]))
                st["gaze"].append((s, e, *gaze[e]))
        st["batch"] = own.take(V.vafr_batch_destroy, V.vafr_batch_create(scene, len(st["frames"])))
        V.vafr_batch_autotune(st["batch"], st["frames"], iters=2)
        if case["graph"]:
            V.vafr_batch_capture(st["batch"], st["frames"])
        return st
    eyes = 2 if kind == "rep" else case.get("eyes", 1)
    half, w, h = case["half"], case["width"], case["height"]
    s = st["session"] = _session(own, case, _eyes(pose, eyes), case.get("fxaa", False))
    st["gaze"] = _gaze(seed, 4, w, h, eyes)
    for e, (x, y) in enumerate(st["gaze"]):
        V.vafr_set_gaze(s, e, x, y)
    if kind in ("frame", "gt"):
        st["out"] = _pixels(half, eyes, h, w)
    if kind == "frame" and case["tuned"]:
        V.vafr_session_autotune(scene, s, _pixels(half, eyes, _slots(s, half)), st["out"], warm=3, iters=5)
    if kind == "gt":
        st["ids"] = torch.empty(eyes, h, w, dtype=torch.int32, device=DEV)
    if kind in ("cast", "build", "pathtrace", "rep", "deferred"):
        st["lp"] = _pixels(half, eyes, _slots(s, half))
        st["ids"] = torch.empty(eyes, _slots(s, half), dtype=torch.int32, device=DEV)
    if kind == "rep":
        st["ids"] = torch.full_like(st["ids"][1], -1)   # guard slots are not written
    if kind == "pathtrace":
        st["seed"] = int(seed) * 7919 + 17
    if kind == "deferred":
        rng = _rng(seed, 6)
        n = case["lights"]
        pos = np.stack([rng.uniform(-60, 60, n), pose[1, 3] + rng.uniform(-5, 10, n), rng.uniform(-170, -60, n)], 1)
        V.vafr_scene_set_point_lights(scene, pos, rng.uniform(2.0, 30.0, (n, 3)))
        st["vbuf"] = torch.empty(h, w, dtype=torch.int64, device=DEV)
    return st


def run(st):
    kind = st["case"]["kind"]
    if kind == "fxaa":
        V.vafr_fxaa_lp(st["session"], 0, st["lp"], st["out"])
        return st["out"]
    if kind == "batch":
        for s, e, x, y in st["gaze"]:
            V.vafr_set_gaze(s, e, x, y)
        if st["case"]["graph"]:
            V.vafr_batch_replay(st["batch"])
        else:
            V.vafr_batch_render(st["batch"], st["frames"])
        return [f[2] for f in st["frames"]] + [f[3] for f in st["frames"]]
    s = st["session"]
    for e, (x, y) in enumerate(st["gaze"]):
        V.vafr_set_gaze(s, e, x, y)
    if kind == "reconstruct":
        V.vafr_reconstruct(s, 0, st["lp"], st["out"])
        return st["out"]
    if kind == "frame":
        V.vafr_render_frame(st["scene"], s, st["out"])
        return st["out"]
    if kind == "cast":
        V.vafr_render_lp(st["scene"], s, (1 << len(st["gaze"])) - 1, st["lp"], st["ids"])
        return st["lp"], st["ids"]
    if kind == "gt":
        V.vafr_render_full_gt(st["scene"], s, 0, st["out"], st["ids"])
        return st["out"], st["ids"]
    if kind == "pathtrace":
        V.vafr_render_lp_pt(st["scene"], s, 1, st["lp"], st["seed"], st["case"]["depth"])
        return st["lp"]
    if kind == "rep":
        V.vafr_render_lp_rep(st["scene"], s, st["lp"], st["ids"])
        return st["lp"], st["ids"]
    if kind == "deferred":
        V.vafr_render_vbuffer(st["scene"], s, 0, st["vbuf"])
        V.vafr_shade_lp_deferred(st["scene"], s, 0, st["vbuf"], st["lp"])
        return st["vbuf"], st["lp"]
    scene = V.vafr_build_scene(st["tris"], st["albedo"], LIGHT)
    V.vafr_render_lp(scene, s, 1, st["lp"], st["ids"])
    V.vafr_scene_destroy(scene)
    return st["lp"], st["ids"]


# ---- the work that a pass cannot do without ------------------------------------------

def _n_tris(case):
    if case["scene"] == "random":
        return case["tris"]
    return 2 * (case["nx"] - 1) * (case["nz"] - 1) + 64 * case["spheres"] + 12 * case["boxes"]


def _rays(case, rays):
    """Bytes and operations of a cast: each ray descends one binary path of log2(n)
    levels (two boxes of 12 operations each), tests one triangle (30) and is set
    up and shaded (60); the triangles and colours that can be hit are read once."""
    n = _n_tris(case)
    return min(n, rays) * 48, rays * (90 + 24 * math.ceil(math.log2(n + 1)))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        texels = _Layout("paper").n.sum()
        px = sum(SERVED[(case["first"] + k) % len(SERVED)][0] * SERVED[(case["first"] + k) % len(SERVED)][1]
                 for k in range(case["sessions"])) * 2
        b, f = _rays(case, 2 * case["sessions"] * texels)
        return {"bytes": int(b + 2 * case["sessions"] * texels * 16 + px * 8), "flops": int(f + 50 * px)}
    bpp = 8 if case["half"] else 16
    lay = _Layout(case.get("acuity", "paper"))
    texels = int(lay.n.sum())
    if kind == "fxaa":
        return {"bytes": 2 * lay.slots * bpp, "flops": texels * 40}
    px = case["width"] * case["height"]
    eyes = 2 if kind == "rep" else case.get("eyes", 1)
    if kind == "reconstruct":
        return {"bytes": lay.slots * bpp + px * bpp, "flops": px * 50}
    if kind == "frame":
        b, f = _rays(case, texels * eyes)
        return {"bytes": int(b + eyes * px * bpp), "flops": int(f + eyes * px * 50)}
    if kind == "gt":
        b, f = _rays(case, px)
        return {"bytes": int(b + px * (bpp + 4)), "flops": int(f)}
    if kind == "pathtrace":    # about one further segment or shadow ray per bounce, paths leaving early
        b, f = _rays(case, texels * (1 + min(case["depth"], 2)))
        return {"bytes": int(b + texels * bpp), "flops": int(f)}
    if kind == "rep":          # the left eye cast, the right one interpolated
        b, f = _rays(case, texels)
        return {"bytes": int(b + texels * (2 * bpp + 4)), "flops": int(f + texels * 150)}
    n = _n_tris(case)
    if kind == "deferred":
        return {"bytes": n * 36 + px * 8 + texels * (8 + bpp),
                "flops": n * 100 + px * 60 + texels * (60 + 20 * case["lights"])}
    b, f = _rays(case, texels * eyes)
    if kind == "build":        # triangles and colours in; sorted triangles, colours and a binary tree out
        return {"bytes": int(b + n * (48 + 64 + 32) + texels * (bpp + 4)), "flops": int(f + n * 200)}
    return {"bytes": int(b + texels * eyes * (bpp + 4)), "flops": int(f)}


# ---- exact results (plain FP64) ------------------------------------------------------

def _shade_exact(tris, alb, org, dirs):
    """FP64 closest hits by testing every triangle, and their shading: (rgba, ids)."""
    t9 = tris.double()
    a, e1, e2 = t9[:, 0:3] - org, t9[:, 3:6] - t9[:, 0:3], t9[:, 6:9] - t9[:, 0:3]
    nrm = torch.linalg.cross(e1, e2)
    an = (a * nrm).sum(-1)
    q1, q2 = torch.linalg.cross(a, e2), torch.linalg.cross(e1, a)
    light = torch.tensor(LIGHT, dtype=torch.float64, device=DEV)
    light = light / light.norm()
    out = torch.ones(len(dirs), 4, dtype=torch.float64, device=DEV)
    ids = torch.full((len(dirs),), -1, dtype=torch.int32, device=DEV)
    step = max(1, (1 << 27) // max(1, len(t9)))
    for i in range(0, len(dirs), step):
        d = dirs[i:i + step]
        det = d @ nrm.T
        t = an / det
        # barycentrics from the Cramer's rule of o + t d = a + u e1 + v e2
        u = -(d @ q1.T) / det
        v = -(d @ q2.T) / det
        miss = (u < 0) | (v < 0) | (u + v > 1) | ~(t > 0)
        t = torch.where(miss, torch.full_like(t, math.inf), t)
        best, k = t.min(1)
        hit = torch.isfinite(best)
        n = nrm[k] / nrm[k].norm(dim=1, keepdim=True)
        n = torch.where(((n * d).sum(1) > 0)[:, None], -n, n)
        lam = (-(n @ light)).clamp(min=0.0)
        rgb = alb.double()[k] * (0.1 + 0.9 * lam)[:, None]
        s = 0.5 * (d[:, 1] / d.norm(dim=1) + 1.0)
        sky = torch.stack([1.0 - 0.5 * s, 1.0 - 0.3 * s, torch.ones_like(s)], 1)
        out[i:i + step, :3] = torch.where(hit[:, None], rgb, sky)
        ids[i:i + step] = torch.where(hit, k.int(), torch.full_like(ids[i:i + step], -1))
    return out, ids


def _lp_exact(case, seed):
    """Exact LP buffers (eyes, slots, 4) and hit ids of a scene small enough to test every triangle."""
    tris, alb, pose = _scene_inputs(case, seed)
    eyes = case.get("eyes", 1)
    n, off, e, col, row = _Layout(case.get("acuity", "paper")).device()
    cr = 2.0 * math.tan(math.radians(case["fov"]) / 2) / case["height"]
    te, ph = torch.tan(torch.deg2rad(e))[col], 2 * math.pi * (row + 0.5) / n[col]
    rgba, ids = [], []
    for P, (x0, y0) in zip(_eyes(pose, eyes), _gaze(seed, 4, case["width"], case["height"], eyes)):
        gx, gy = cr * (x0 - 0.5 * case["width"]), cr * (0.5 * case["height"] - y0)
        d = torch.stack([te * torch.cos(ph) + gx, -te * torch.sin(ph) + gy, torch.ones_like(te)], 1)
        P = torch.from_numpy(P).to(DEV)
        a, b = _shade_exact(tris, alb, P[:, 3], d @ P[:, :3].T)
        rgba.append(a)
        ids.append(b)
    return torch.stack(rgba), torch.stack(ids)


def _reconstruct_exact(case, lp, gaze):
    """Exact display (height, width, 4) of one eye's LP buffer (slots, 4)."""
    lay = _Layout(case["acuity"])
    n, off, _, _, _ = lay.device()
    lp = lp.double()
    w, h = case["width"], case["height"]
    cr = 2.0 * math.tan(math.radians(case["fov"]) / 2) / h
    out = torch.empty(h, w, 4, dtype=torch.float64, device=DEV)
    dx = (torch.arange(w, device=DEV, dtype=torch.float64) + 0.5 - gaze[0])[None, :]
    rows = max(1, (1 << 23) // w)
    for y in range(0, h, rows):
        dy = (torch.arange(y, min(h, y + rows), device=DEV, dtype=torch.float64) + 0.5 - gaze[1])[:, None]
        e = torch.rad2deg(torch.atan(cr * torch.sqrt(dx * dx + dy * dy))).clamp(max=lay.e_max)
        uf = lay.u_of_e(e) - 0.5
        frac = torch.atan2(dy.expand_as(uf), dx.expand_as(uf)) / (2 * math.pi)
        frac = torch.where(frac < 0, frac + 1, frac)
        c0 = uf.floor()
        wu = (uf - c0)[..., None]
        v = []
        for k in (0, 1):
            c = (c0.long() + k).clamp(0, lay.n_cols - 1)
            r = frac * n[c] - 0.5
            j = r.floor()
            wr = (r - j)[..., None]
            j = j.long()
            v.append(lp[off[c] + j % n[c]] * (1 - wr) + lp[off[c] + (j + 1) % n[c]] * wr)
        out[y:y + rows] = v[0] * (1 - wu) + v[1] * wu
    return out


def _fxaa_exact(case, lp):
    """FXAA of one eye's LP buffer (slots, 4): the published method on the LP grid, in FP64."""
    lay = _Layout(case["acuity"])
    n, off, _, col, row = lay.device()
    lp = lp.double()
    lum = 0.299 * lp[:, 0] + 0.587 * lp[:, 1] + 0.114 * lp[:, 2]
    nc = n[col]

    def at(c2, j=row):      # slot of the texel of column c2 (clamped) at the angle of row j
        c2 = c2.clamp(0, lay.n_cols - 1)
        j2 = torch.where(c2 == col, j, (2 * j + 1) * n[c2] // (2 * nc))
        return off[c2] + j2

    t = off[col] + row
    sE, sW = at(col + 1), at(col - 1)
    M, N, S, E, W = lum[t], lum[t + 1], lum[t - 1], lum[sE], lum[sW]
    NE, SE, NW, SW = lum[sE + 1], lum[sE - 1], lum[sW + 1], lum[sW - 1]
    five = torch.stack([M, N, S, E, W])
    lo, hi = five.amin(0), five.amax(0)
    rng = hi - lo
    skip = rng < torch.clamp(hi / 6, min=1 / 12)
    kA = 2 * (N + S - 2 * M).abs() + (NE + SE - 2 * E).abs() + (NW + SW - 2 * W).abs()
    kR = 2 * (E + W - 2 * M).abs() + (NE + NW - 2 * N).abs() + (SE + SW - 2 * S).abs()
    across = kR >= kA
    Ln, Lp = torch.where(across, W, S), torch.where(across, E, N)
    gn, gp = (Ln - M).abs(), (Lp - M).abs()
    pos = gp >= gn
    avg = 0.5 * (M + torch.where(pos, Lp, Ln))
    thr = 0.25 * torch.maximum(gn, gp)
    side = torch.where(pos, 1, -1)
    dist, end = [], []
    for sgn in (-1, 1):
        d = torch.full_like(col, 12)
        last = torch.zeros_like(M)
        going = torch.ones_like(across)
        for k in range(1, 13):
            jk = (row + sgn * k) % nc
            ta = torch.where(across, off[col] + jk, at(col + sgn * k))
            tb = torch.where(across, at(col + side, jk), ta + side)
            s = 0.5 * (lum[ta] + lum[tb])
            last = torch.where(going, s, last)
            stop = going & ((s - avg).abs() >= thr)
            d = torch.where(stop, k, d)
            going &= ~stop
        dist.append(d)
        end.append(last)
    near = dist[0] < dist[1]
    dn, lend = torch.where(near, dist[0], dist[1]), torch.where(near, end[0], end[1])
    good = ((lend - avg) < 0) != ((M - avg) < 0)
    edge = torch.where(good, 0.5 - dn.double() / (dist[0] + dist[1]).double(), torch.zeros_like(M))
    l3 = (2 * (N + S + E + W) + NE + NW + SE + SW) / 12
    a = ((l3 - M).abs() / torch.where(rng > 0, rng, torch.ones_like(rng))).clamp(max=1.0)
    b = (3 - 2 * a) * a * a
    wgt = torch.maximum(edge, 0.75 * b * b)
    q = torch.where(across, torch.where(pos, sE, sW), t + side)
    out = lp[t] + torch.where(skip, torch.zeros_like(wgt), wgt)[:, None] * (lp[q] - lp[t])
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "reconstruct":
        return _reconstruct_exact(case, _lp_image(case, seed), _gaze(seed, 4, case["width"], case["height"], 1)[0])
    if kind == "fxaa":
        return _fxaa_exact(case, _lp_image(case, seed))
    if case.get("scene") != "random":
        return None              # testing every triangle would take minutes
    if kind in ("cast", "build"):
        return _lp_exact(case, seed)
    if kind == "gt":
        tris, alb, pose = _scene_inputs(case, seed)
        w, h = case["width"], case["height"]
        cr = 2.0 * math.tan(math.radians(case["fov"]) / 2) / h
        y, x = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
        d = torch.stack([cr * (x + 0.5 - 0.5 * w), cr * (0.5 * h - y - 0.5), torch.ones_like(x).double()],
                        -1).double().reshape(-1, 3)
        P = torch.from_numpy(pose).to(DEV)
        rgba, ids = _shade_exact(tris, alb, P[:, 3], d @ P[:, :3].T)
        return rgba.reshape(1, h, w, 4), ids.reshape(1, h, w)
    if case["fxaa"]:
        return None
    lp, _ = _lp_exact(case, seed)
    gaze = _gaze(seed, 4, case["width"], case["height"], case["eyes"])
    return torch.stack([_reconstruct_exact(case, lp[e], gaze[e]) for e in range(case["eyes"])])
