"""The work that a program has this library do, as cases that can be timed and checked.

Each case is one pass through the public entry points: a frame of probe update and query, a
query alone, a texel gradient, a training step, a camera G-buffer.  Scenes are made of
axis-aligned boxes and rectangles (a city, a room, an interior) or a heightfield with boxes
(the tracking cascades), drawn from the seed; sizes are those of the library's own workloads
and tests, and smaller, larger and odd ones around them.

``exact`` evaluates the same pass in 64-bit floating point with plain torch: rays against
every box, sums over every ray, the eight-probe query.  It starts from the state that
``prepare`` leaves (atlases, probe states, points), so it computes the one pass that ``run``
makes.
"""
import math

import numpy as np
import torch

import paper_2009_10796_gb300 as ddgi

FP32, FP16, RGB9E5 = 0, 1, 2
BLEND = {"fp32": 0, "tf32": 1, "bf16": 2, "tf32x3": 3}
OFF, SLEEPING, NEWLY, VIGILANT = 1, 2, 3, 4


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # one room, few probes and rays: every launch is short, latency and launches count
        dict(name="room_frame", kind="frame", scene="room", boxes=32, nx=8, ny=8, nz=8, spacing=1.25, rays=64,
             irr_n=6, dist_n=14, blend="fp32", fmt=FP32, hysteresis=0.9, width=64, height=64),
        # the frame of a game: a level around the camera, full-precision blend, 1080p
        dict(name="city_frame", kind="frame", scene="city", boxes=16384, nx=32, ny=16, nz=32, spacing=2.0, rays=256,
             irr_n=6, dist_n=14, blend="fp32", fmt=FP32, hysteresis=0.97, width=1920, height=1080),
        # the memory-saving settings: FP16 atlases and the tensor-core blend, an odd grid, half resolution
        dict(name="city_mixed", kind="frame", scene="city", boxes=4096, nx=29, ny=13, nz=31, spacing=2.0, rays=200,
             irr_n=6, dist_n=14, blend="tf32", fmt=FP16, hysteresis=0.97, width=959, height=541),
        # the paper's own tile resolution (8 x 8 irradiance, 16 x 16 visibility)
        dict(name="paper_tiles", kind="frame", scene="city", boxes=4096, nx=24, ny=12, nz=20, spacing=2.0, rays=192,
             irr_n=8, dist_n=16, blend="fp32", fmt=FP32, hysteresis=0.97, width=1280, height=720),
        # a renderer that owns all its memory: the allocation-free update
        dict(name="noalloc_update", kind="noalloc", scene="city", boxes=4096, nx=16, ny=8, nz=16, spacing=2.0,
             rays=128, irr_n=6, dist_n=14, hysteresis=0.97),
        # a level is entered: every probe is new, the position optimizer and classification run
        dict(name="level_load", kind="load", scene="city", boxes=4096, nx=24, ny=12, nz=24, spacing=2.0, rays=128,
             irr_n=6, dist_n=14, iters=5),
        # an open world: four nested volumes that follow the camera, replayed as a graph, and their query
        dict(name="cascade_frame", kind="cascade", quads=256, boxes=10000, n=32, levels=4, rays=288, blend="fp32",
             fmt=FP32, width=1280, height=720),
        # a few thousand points (particles, agents) looked up: the smallest call
        dict(name="query_points", kind="query", nx=8, ny=8, nz=8, spacing=1.25, irr_n=6, dist_n=14, gamma=5.0,
             fmt=FP32, glossy=False, width=64, height=64),
        # second-order glossy reflections at half resolution
        dict(name="glossy_half", kind="query", nx=16, ny=8, nz=16, spacing=2.5, irr_n=6, dist_n=14, gamma=5.0,
             fmt=FP32, glossy=True, width=960, height=540),
        # texels fitted to target irradiance: query and its gradient
        dict(name="texel_gradient", kind="texels", nx=16, ny=8, nz=16, spacing=2.5, irr_n=6, dist_n=14, gamma=5.0,
             width=1280, height=720),
        # materials and emitters fitted to target irradiance: two frames, query, reverse pass
        dict(name="field_training", kind="train", boxes=16000, objects=256, emitters=64, nx=16, ny=8, nz=16,
             spacing=2.5, rays=128, gamma=1.0, frames=2, points=1000000),
        # the camera's G-buffer traced instead of rasterised
        dict(name="gbuffer", kind="gbuffer", scene="city", boxes=16384, width=1920, height=1080),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    kind = rng.choice(["frame", "frame", "frame", "noalloc", "load", "cascade", "query", "query", "texels", "train",
                       "gbuffer"])
    grid = dict(nx=rng.randint(6, 28), ny=rng.randint(4, 14), nz=rng.randint(6, 28), spacing=2.0)
    pixels = dict(width=_log(rng, 48, 1920), height=_log(rng, 40, 1080))
    city = dict(scene="city", boxes=rng.randint(24, 96) ** 2)
    tiles = dict(zip(("irr_n", "dist_n"), rng.choice([(6, 14), (6, 14), (8, 16), (5, 12)])))
    if kind == "frame":
        blend = rng.choice(["fp32", "fp32", "tf32", "bf16", "tf32x3"])
        fmt = rng.choice([FP32, FP32, FP16])
        if rng.random() < 0.3:
            city = dict(scene="room", boxes=rng.randint(12, 200))
            grid = dict(nx=rng.randint(4, 12), ny=rng.randint(4, 12), nz=rng.randint(4, 12), spacing=0.75)
        return dict(kind=kind, **city, **grid, rays=_log(rng, 48, 288), **tiles, blend=blend, fmt=fmt,
                    hysteresis=rng.choice([0.0, 0.9, 0.97]), **pixels)
    if kind == "noalloc":
        return dict(kind=kind, **city, nx=rng.randint(6, 20), ny=rng.randint(4, 10), nz=rng.randint(6, 20),
                    spacing=2.0, rays=_log(rng, 48, 250), **tiles, hysteresis=rng.choice([0.0, 0.9, 0.97]))
    if kind == "load":
        return dict(kind=kind, **city, nx=rng.randint(6, 24), ny=rng.randint(4, 12), nz=rng.randint(6, 24),
                    spacing=2.0, rays=_log(rng, 32, 128), **tiles, iters=rng.randint(0, 5))
    if kind == "cascade":
        return dict(kind=kind, quads=rng.randint(64, 256), boxes=_log(rng, 500, 10000), n=rng.choice([16, 20, 24, 32]),
                    levels=rng.randint(2, 4), rays=4 * rng.randint(16, 64), blend=rng.choice(["fp32", "tf32x3"]),
                    fmt=rng.choice([FP32, FP32, FP16]), **pixels)
    if kind == "query":
        return dict(kind=kind, nx=rng.randint(4, 30), ny=rng.randint(4, 12), nz=rng.randint(4, 30), spacing=1.5,
                    **tiles, gamma=rng.choice([5.0, 5.0, 5.0, 2.2, 1.0]), fmt=rng.choice([FP32, FP32, FP16, RGB9E5]),
                    glossy=rng.random() < 0.4, **pixels)
    if kind == "texels":
        return dict(kind=kind, nx=rng.randint(4, 16), ny=rng.randint(4, 8), nz=rng.randint(4, 16), spacing=2.0,
                    **tiles, gamma=rng.choice([5.0, 5.0, 1.0]), width=_log(rng, 48, 1280), height=_log(rng, 40, 720))
    if kind == "train":
        return dict(kind=kind, boxes=_log(rng, 500, 16000), objects=rng.randint(8, 256), emitters=rng.randint(4, 64),
                    nx=rng.randint(6, 16), ny=rng.randint(4, 8), nz=rng.randint(6, 16), spacing=2.5,
                    rays=_log(rng, 48, 128), gamma=rng.choice([1.0, 1.0, 5.0]), frames=rng.randint(1, 2),
                    points=_log(rng, 5000, 1000000))
    return dict(kind=kind, **city, **pixels)


# ---------------------------------------------------------------------------
# Scenes: axis-aligned boxes and rectangles, or a heightfield with boxes
# ---------------------------------------------------------------------------

class Scene:
    """Boxes lo / hi [B, 3] (fronts outside), an optional shell (fronts inside), rectangles
    (axis, sign of the normal, lo, hi with lo[axis] = hi[axis]); object and emitter of each."""

    def __init__(self, rng):
        self.rng = rng
        self.lo = self.hi = np.zeros((0, 3), np.float32)
        self.box_obj = np.zeros(0, np.int32)
        self.shell = None        # (lo, hi), object 0
        self.rects = []          # (axis, sign, lo, hi, object, emitter)
        self.field = None        # (verts, tris), object 0
        self.albedo = np.zeros((0, 3), np.float32)
        self.casts = np.zeros(0, np.int32)
        self.emit = np.zeros((0, 3), np.float32)

    def _box_tris(self, lo, hi):
        c = np.array([[x, y, z] for x in (0, 1) for y in (0, 1) for z in (0, 1)])
        v = np.where(c[None], hi[:, None], lo[:, None]).astype(np.float32)
        # counter-clockwise seen from outside
        q = np.array([[0, 1, 3, 2], [4, 6, 7, 5], [0, 4, 5, 1], [2, 3, 7, 6], [0, 2, 6, 4], [1, 5, 7, 3]])
        t = np.concatenate([q[:, [0, 1, 2]], q[:, [0, 2, 3]]])
        return v.reshape(-1, 3), (8 * np.arange(len(lo))[:, None, None] + t[None]).reshape(-1, 3)

    def arrays(self):
        vs, ts, ob, em = [], [], [], []
        n = 0

        def add(v, t, o, e):
            nonlocal n
            vs.append(v); ts.append(t + n); ob.append(o); em.append(e)
            n += len(v)

        for axis, sign, lo, hi, obj, e in self.rects:
            u, w = (axis + 1) % 3, (axis + 2) % 3
            p = np.tile(np.asarray(lo, np.float32), (4, 1))
            p[1, u] = p[2, u] = hi[u]
            p[2, w] = p[3, w] = hi[w]
            t = np.array([[0, 1, 2], [0, 2, 3]])
            add(p, t if sign > 0 else t[:, ::-1], np.full(2, obj), np.full(2, e))
        if self.field is not None:
            add(self.field[0], self.field[1], np.zeros(len(self.field[1])), np.full(len(self.field[1]), -1))
        if self.shell is not None:
            v, t = self._box_tris(*[np.asarray(a, np.float32)[None] for a in self.shell])
            add(v, t[:, ::-1], np.zeros(12), np.full(12, -1))
        if len(self.lo):
            v, t = self._box_tris(self.lo, self.hi)
            add(v, t, np.repeat(self.box_obj, 12), np.full(len(t), -1))
        return (np.concatenate(vs), np.concatenate(ts).astype(np.int32), np.concatenate(ob).astype(np.int32),
                self.albedo, self.casts, np.concatenate(em).astype(np.int32), self.emit)

    def upload(self):
        return ddgi.Scene(*self.arrays())


class Light:
    def __init__(self, sun_dir, sun, a, b):
        d = np.asarray(sun_dir, np.float64)
        self.sun_dir = (d / np.linalg.norm(d)).astype(np.float32)
        self.sun_irradiance = np.full(3, sun, np.float32)
        self.sky_a = np.full(3, a, np.float32)
        self.sky_b = np.full(3, b, np.float32)
        self.sky_up = np.array([0.0, 1.0, 0.0], np.float32)


def _city(rng, boxes):
    """One tower per 4 m lot (footprint 2 to 3.5 m, 4 to 40 m high), founded below the ground."""
    s, side = Scene(rng), int(round(math.sqrt(boxes)))
    half = 2.0 * side
    s.rects.append((1, 1, (-half, 0.0, -half), (half, 0.0, half), 0, -1))
    iz, ix = np.divmod(np.arange(side * side), side)
    c = np.stack([-half + 4.0 * (ix + 0.5), -half + 4.0 * (iz + 0.5)], 1)
    f = rng.uniform(1.0, 1.75, (side * side, 2))
    top = rng.uniform(4.0, 40.0, side * side)
    s.lo = np.stack([c[:, 0] - f[:, 0], np.full(len(c), -0.5), c[:, 1] - f[:, 1]], 1).astype(np.float32)
    s.hi = np.stack([c[:, 0] + f[:, 0], top, c[:, 1] + f[:, 1]], 1).astype(np.float32)
    s.box_obj = rng.integers(1, 8, len(c)).astype(np.int32)
    s.albedo = rng.uniform(0.5, 0.9, (8, 3)).astype(np.float32)
    s.casts = np.ones(8, np.int32)
    return s, Light((0.3, -1.0, 0.5), 3.0, 0.2, 0.1)


def _room(rng, boxes):
    """A 10 m room with box occluders and one 2 m lamp on a wall; its shell lets the sun in."""
    s = Scene(rng)
    s.shell = ((0.0, 0.0, 0.0), (10.0, 10.0, 10.0))
    c, h = rng.uniform(1.0, 9.0, (boxes, 3)), rng.uniform(0.15, 0.8, (boxes, 3))
    s.lo, s.hi = (c - h).astype(np.float32), (c + h).astype(np.float32)
    s.box_obj = 1 + np.arange(boxes, dtype=np.int32) % 32
    s.rects.append((0, 1, (0.01, 4.0, 4.0), (0.01, 6.0, 6.0), 33, 0))
    s.albedo = rng.uniform(0.5, 0.9, (34, 3)).astype(np.float32)
    s.casts = np.ones(34, np.int32)
    s.casts[0] = 0
    s.emit = np.full((1, 3), 5.0, np.float32)
    return s, Light((0.3, -1.0, 0.2), 3.0, 0.0, 0.0)


def _interior(rng, boxes, objects, emitters):
    """A 40 x 20 x 40 m hall with boxes grouped into objects and lamps on the ceiling and a wall."""
    s = Scene(rng)
    s.shell = ((-20.0, 0.0, -20.0), (20.0, 20.0, 20.0))
    c = np.stack([rng.uniform(-19, 19, boxes), rng.uniform(0.5, 18, boxes), rng.uniform(-19, 19, boxes)], 1)
    h = rng.uniform(0.1, 0.6, (boxes, 3))
    s.lo, s.hi = (c - h).astype(np.float32), (c + h).astype(np.float32)
    s.box_obj = (1 + np.arange(boxes) % (objects - 1)).astype(np.int32)
    # each lamp in a cell of its own: 8 x 8 cells of the ceiling, 4 x 8 of the wall
    ceiling, wall = rng.permutation(64), rng.permutation(32)
    for k in range(emitters):
        dx, dz = rng.uniform(0.0, 2.5, 2)
        if k % 2 == 0:
            u, v = -17 + 4.25 * (ceiling[k // 2] // 8) + dx, -17 + 4.25 * (ceiling[k // 2] % 8) + dz
            s.rects.append((1, -1, (u, 19.99, v), (u + 1.5, 19.99, v + 1.5), objects, k))
        else:
            y, v = 1.0 + 4.25 * (wall[k // 2] // 8) + dx, -17 + 4.25 * (wall[k // 2] % 8) + dz
            s.rects.append((0, 1, (-19.99, y, v), (-19.99, y + 1.5, v + 1.5), objects, k))
    s.rects = [(a, g, np.asarray(lo, np.float32), np.asarray(hi, np.float32), o, e) for a, g, lo, hi, o, e in s.rects]
    s.albedo = rng.uniform(0.2, 0.9, (objects + 1, 3)).astype(np.float32)
    s.casts = np.ones(objects + 1, np.int32)
    s.emit = np.repeat(rng.uniform(0.1, 2.0, (emitters, 1)), 3, 1).astype(np.float32)
    return s, Light((0.3, -1.0, 0.2), 3.0, 0.0, 0.0)


class _Hills:
    """Height of a sum of eight sinusoid products, 20 m at most."""

    def __init__(self, rng):
        self.fx, self.fz = rng.uniform(0.002, 0.02, (2, 8))
        self.px, self.pz = rng.uniform(0.0, 2 * np.pi, (2, 8))
        self.amp = rng.uniform(0.5, 1.0, 8)

    def __call__(self, x, z):
        x, z = np.asarray(x)[..., None], np.asarray(z)[..., None]
        h = (self.amp * np.sin(self.fx * x + self.px) * np.cos(self.fz * z + self.pz)).sum(-1)
        return 20.0 * h / self.amp.sum()


def _terrain(rng, quads, boxes):
    s, hills, size = Scene(rng), _Hills(rng), 2.0 * quads
    n = quads + 1
    x, z = np.meshgrid(*[np.linspace(-size / 2, size / 2, n)] * 2, indexing="ij")
    v = np.stack([x, hills(x, z), z], -1).reshape(-1, 3).astype(np.float32)
    i, j = np.divmod(np.arange(quads * quads), quads)
    a = i * n + j
    s.field = (v, np.concatenate([np.stack([a, a + 1, a + n + 1], 1), np.stack([a, a + n + 1, a + n], 1)]))
    c = rng.uniform(-size / 2 + 10, size / 2 - 10, (boxes, 2))
    f, top = rng.uniform(1.0, 4.0, (boxes, 2)), rng.uniform(3.0, 20.0, boxes)
    y = hills(c[:, 0], c[:, 1])
    s.lo = np.stack([c[:, 0] - f[:, 0], y - 3.0, c[:, 1] - f[:, 1]], 1).astype(np.float32)
    s.hi = np.stack([c[:, 0] + f[:, 0], y + top, c[:, 1] + f[:, 1]], 1).astype(np.float32)
    s.box_obj = np.ones(boxes, np.int32)
    s.albedo = np.full((2, 3), 0.7, np.float32)
    s.casts = np.ones(2, np.int32)
    return s, hills, Light((0.3, -1.0, 0.5), 3.0, 0.2, 0.1)


def _scene_of(case, rng):
    return _city(rng, case["boxes"]) if case["scene"] == "city" else _room(rng, case["boxes"])


def _camera(scene):
    if scene.shell is not None:
        return (5.0, 5.0, 1.0), (0.1, -0.15, 1.0)
    at = 2.0 * (int(round(math.sqrt(len(scene.lo)))) % 2)      # a crossing of two streets
    return (at, 12.0, -28.0 + at), (0.0, -0.1736, 0.9848)


class Desc:
    """A volume descriptor (the fields that the library reads)."""

    def __init__(self, case, seed, **kw):
        n, s = (case["nx"], case["ny"], case["nz"]), float(case["spacing"])
        self.counts, self.spacing = n, (s, s, s)
        self.origin = tuple(float(np.float32(-0.5 * s * (k - 1))) for k in n)
        self.rays_per_probe = case.get("rays", 64)
        self.irr_n, self.dist_n = case.get("irr_n", 6), case.get("dist_n", 14)
        self.hysteresis_irr = self.hysteresis_vis = case.get("hysteresis", 0.0)
        self.gamma = case.get("gamma", 5.0)
        self.irr_format = case.get("fmt", FP32)
        self.dist_format = FP16 if self.irr_format == FP16 else FP32
        self.self_shadow_bias, self.dist_cos_power, self.t_max = 0.3, 50.0, 2.0 * s * math.sqrt(3.0)
        self.thr_low, self.thr_high, self.thr_step = 0.25, 0.8, 0.15
        self.state_machine, self.seed, self.tracking = 1, seed, 0
        self.optimizer_iters, self.offset_limit, self.converge_batches = 0, 0.45, 0
        for k, v in kw.items():
            setattr(self, k, v)


def _place(desc, case):
    """Over the ground of a city, inside a room."""
    n, s = desc.counts, desc.spacing[0]
    if case.get("scene") == "city":
        desc.origin = (desc.origin[0], 1.0, desc.origin[2])
    elif case.get("scene") == "room":
        desc.spacing = tuple(float(np.float32(10.0 / k)) for k in n)
        desc.origin = tuple(float(np.float32(0.5 * d)) for d in desc.spacing)
        desc.t_max = 2.0 * math.sqrt(sum(d * d for d in desc.spacing))
    else:
        desc.origin = (desc.origin[0], 0.5 * s, desc.origin[2])
    return desc


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------

class State:
    pass


def _buffers(s, vol, extra=False):
    """The caller's copies of a volume's atlases and states, as a renderer or a checkpoint keeps them."""
    d, N, M = vol.desc, vol.desc.irr_n + 2, vol.desc.dist_n + 2
    half = d.irr_format == FP16
    s.irr = torch.zeros((vol.n_probes, N, N, 4), dtype=torch.float16 if half else torch.float32, device="cuda")
    s.dist = torch.zeros((vol.n_probes, M, M, 2), dtype=torch.float16 if half else torch.float32, device="cuda")
    s.states = torch.zeros(vol.n_probes, dtype=torch.uint8, device="cuda")
    if extra:
        s.offsets = torch.zeros((vol.n_probes, 4), dtype=torch.float32, device="cuda")


def prepare(case, seed):
    s = State()
    s.case, rng, kind = case, np.random.default_rng(seed), case["kind"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if kind in ("frame", "noalloc", "load", "gbuffer"):
        s.model, s.lights = _scene_of(case, rng)
        s.scene = s.model.upload()
        s.cam, s.fwd = _camera(s.model)
        s.frame = 0
    if kind == "gbuffer":
        s.cam = tuple(float(v) for v in np.float32(np.asarray(s.cam) + rng.uniform(-1, 1, 3) * (0.2, 4.0, 0.2)))
    elif kind == "frame":
        s.desc = _place(Desc(case, seed), case)
        s.vol = ddgi.Volume(s.desc)
        s.pos, s.nrm = s.scene.raycast_gbuffer(s.cam, s.fwd, (0.0, 1.0, 0.0), 60.0, case["width"], case["height"])
        s.out = torch.empty_like(s.pos)
        _buffers(s, s.vol)
        for _ in range(3):      # classified and lit, as every frame but the first finds it
            run(s)
    elif kind == "noalloc":
        s.desc = _place(Desc(case, seed), case)
        P = case["nx"] * case["ny"] * case["nz"]
        N, M = s.desc.irr_n + 2, s.desc.dist_n + 2
        s.irr = torch.zeros((P, N, N, 4), device="cuda")
        s.dist = torch.zeros((P, M, M, 2), device="cuda")
        s.states = torch.zeros(P, dtype=torch.uint8, device="cuda")
        for _ in range(3):
            run(s)
    elif kind == "load":
        s.desc = _place(Desc(case, seed, optimizer_iters=case["iters"]), case)
        s.vol = ddgi.Volume(s.desc)
        _buffers(s, s.vol, extra=True)
        s.zero = [torch.zeros_like(t) for t in (s.irr, s.dist, s.states, s.offsets)]
    elif kind == "cascade":
        s.model, hills, s.lights = _terrain(rng, case["quads"], case["boxes"])
        s.scene = s.model.upload()
        # a walk round a circle, 0.6 m a frame, 10 m above the ground
        k = np.arange(105)
        x, z = 10.0 * np.cos(2 * np.pi * k / 105), 10.0 * np.sin(2 * np.pi * k / 105)
        s.path = [tuple(float(v) for v in p) for p in np.float32(np.stack([x, hills(x, z) + 10.0, z], 1))]
        c, n = dict(case, nx=case["n"], ny=case["n"], nz=case["n"], hysteresis=0.97), case["n"]
        s.vol = ddgi.Cascade([Desc(dict(c, spacing=2.0 ** k), seed, tracking=1) for k in range(case["levels"])])
        s.pos, s.nrm = s.scene.raycast_gbuffer(s.path[0], (0.9, -0.3, 0.3), (0.0, 1.0, 0.0), 60.0, case["width"],
                                               case["height"])
        s.out, s.frame = torch.empty_like(s.pos), 0
        for _ in range(4):
            run(s)
    elif kind in ("query", "texels"):
        s.desc = Desc(case, seed)
        s.vol = ddgi.Volume(s.desc)
        _lit_hall(s, gen)
        if kind == "texels":
            s.atlas = s.irr.clone().requires_grad_(True)
            s.dE = torch.randn(s.pos.shape, generator=gen, device="cuda")
    elif kind == "train":
        s.model, s.lights = _interior(rng, case["boxes"], case["objects"], case["emitters"])
        s.scene = s.model.upload()
        s.desc = _place(Desc(case, seed, state_machine=0), case)
        s.vol = ddgi.Volume(s.desc)
        s.cam = (0.0, 10.0, 0.0)
        s.pos, s.nrm = _surface_points(s.model, case["points"], gen)
        s.albedo = torch.tensor(s.model.albedo, device="cuda").requires_grad_(True)
        s.emit = torch.tensor(s.model.emit, device="cuda").requires_grad_(True)
        s.target = 0.5 + torch.rand(s.pos.shape, generator=gen, device="cuda")
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "frame":
        s.vol.update(s.scene, s.lights, s.frame, precision=BLEND[case["blend"]])
        s.vol.query(s.pos, s.nrm, s.cam, out=s.out)
        s.frame += 1
        for which, t in enumerate((s.irr, s.dist, s.states)):
            s.vol.copy_buffer(which, t)
        return {"E": s.out, "irr": s.irr[..., :3], "dist": s.dist, "states": s.states}
    if kind == "noalloc":
        ddgi.update_noalloc(s.scene, s.desc, s.lights, s.frame, s.states, s.irr, s.dist)
        s.frame += 1
        return {"irr": s.irr[..., :3], "dist": s.dist, "states": s.states}
    if kind == "load":
        for which, t in enumerate(s.zero):
            s.vol.set_buffer(which, t)
        s.vol.update(s.scene, s.lights, s.frame)
        s.frame += 1
        for which, t in enumerate((s.irr, s.dist, s.states, s.offsets)):
            s.vol.copy_buffer(which, t)
        return {"irr": s.irr[..., :3], "dist": s.dist, "states": s.states, "offsets": s.offsets}
    if kind == "cascade":
        s.cam = s.path[s.frame % len(s.path)]
        s.vol.update(s.scene, s.lights, s.frame, s.cam, precision=BLEND[case["blend"]], use_graph=True)
        s.vol.query(s.pos, s.nrm, s.cam, out=s.out)
        s.frame += 1
        dt = torch.float16 if case["fmt"] == FP16 else torch.float32
        return {"E": s.out, "volumes": [[s.vol.buffer(k, 0).view(dt), s.vol.buffer(k, 1).view(dt), s.vol.states(k)]
                                        for k in range(case["levels"])]}
    if kind == "query":
        if case["glossy"]:
            return s.vol.query_glossy(s.pos, s.nrm, s.dirs, out=s.out)
        return s.vol.query(s.pos, s.nrm, s.cam, out=s.out)
    if kind == "texels":
        s.atlas.grad = None
        E = ddgi.ProbeQuery.apply(s.atlas, s.vol, s.pos, s.nrm, s.cam)
        E.backward(s.dE)
        return {"E": E, "grad": s.atlas.grad}
    if kind == "train":
        s.albedo.grad = s.emit.grad = None
        E = ddgi.IrradianceField.apply(s.albedo, s.emit, s.vol, s.scene, s.lights, s.pos, s.nrm, s.cam, 0,
                                       case["frames"])
        ((E - s.target) ** 2).mean().backward()
        return {"E": E, "albedo": s.albedo.grad, "emit": s.emit.grad}
    return s.scene.raycast_gbuffer(s.cam, s.fwd, (0.0, 1.0, 0.0), 60.0, case["width"], case["height"])


def work(case):
    """Bytes: inputs and atlases read once, outputs written once.  Operations: box and triangle
    tests of a walk down the hierarchy (a ray cannot do without a path to its hit), the weighted
    sums, about 400 for each of a point's eight probes."""
    kind = case["kind"]
    n = case.get("points", case.get("width", 0) * case.get("height", 0))
    P = case.get("nx", 0) * case.get("ny", 0) * case.get("nz", 0)
    if kind == "cascade":
        P = case["levels"] * case["n"] ** 3
    tris = 12 * case.get("boxes", 0) + 2 * case.get("quads", 0) ** 2 + 2
    ray = 100 * max(1.0, math.log(tris, 4)) + 60
    ni, nd = case.get("irr_n", 6), case.get("dist_n", 14)
    half = 0.5 if case.get("fmt") in (FP16, RGB9E5) else 1.0
    tile = half * (16 * (ni + 2) ** 2 + 8 * (nd + 2) ** 2)
    # shares seen in these scenes: a quarter of a city's or landscape's probes are active, most of a room's
    share = {"frame": 0.9 if case.get("scene") == "room" else 0.25, "noalloc": 0.25, "load": 0.25, "cascade": 0.15,
             "train": 1.0}.get(kind, 0.0)
    traced = share * P * case.get("rays", 0)
    rays = traced * 1.5 + (n if kind == "gbuffer" else 0)
    frames = case.get("frames", 1)
    flops = frames * (rays * ray + traced * 8 * 400 + traced * 2 * (3 * ni * ni + 2 * nd * nd)) + (0 if kind == "gbuffer" else n * 8 * 400)
    bytes_ = n * (24 if kind == "gbuffer" else 36) + frames * share * P * tile * 2 + min(tris * 64, rays * 100)
    if kind in ("frame", "load"):
        bytes_ += 2 * P * tile                       # the caller's copies
    if kind == "load":
        flops += (1 + case["iters"]) * P * case["rays"] * ray
        bytes_ += 2 * P * tile
    if kind in ("query", "texels"):
        bytes_ += P * tile
    if kind == "cascade":
        bytes_ += 2 * P * tile
    if kind == "texels":
        flops *= 2
        bytes_ += n * 36 + 4 * P * tile
    if kind == "train":
        flops *= 2
        bytes_ += n * 48
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# A lit hall in closed form: probes, points and atlases without a trace
# ---------------------------------------------------------------------------

def _texel_dirs(n):
    u = (2.0 * torch.arange(n, dtype=torch.float64, device="cuda") + 1.0) / n - 1.0
    y, x = torch.meshgrid(u, u, indexing="ij")
    z = 1.0 - x.abs() - y.abs()
    sx, sy = torch.where(x >= 0, 1.0, -1.0), torch.where(y >= 0, 1.0, -1.0)
    v = torch.stack([torch.where(z < 0, (1 - y.abs()) * sx, x), torch.where(z < 0, (1 - x.abs()) * sy, y), z], -1)
    return v / v.norm(dim=-1, keepdim=True)


def _bordered(t):
    """[..., n, n, C] interior texels to [..., n + 2, n + 2, C] tiles (the octahedral border)."""
    n = t.shape[-2]
    at = torch.empty((n + 2, n + 2), dtype=torch.long)
    inner = torch.arange(n * n).view(n, n)
    at[1:-1, 1:-1] = inner
    at[1:-1, 0], at[1:-1, -1] = inner[:, 0].flip(0), inner[:, -1].flip(0)
    at[0, 1:-1], at[-1, 1:-1] = inner[0].flip(0), inner[-1].flip(0)
    at[0, 0], at[0, -1], at[-1, 0], at[-1, -1] = inner[-1, -1], inner[-1, 0], inner[0, -1], inner[0, 0]
    f = t.reshape(*t.shape[:-3], n * n, t.shape[-1])
    return f[..., at.view(-1).to(t.device), :].view(*t.shape[:-3], n + 2, n + 2, t.shape[-1])


def _grid(desc):
    ax = [torch.arange(k, dtype=torch.float64, device="cuda") * float(np.float32(s)) + float(np.float32(o))
          for k, s, o in zip(desc.counts, desc.spacing, desc.origin)]
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    return torch.stack([x, y, z], -1).view(-1, 3)


def _lit_hall(s, gen):
    """A box hall around the volume: distances to its walls, a smooth seeded radiance, a tenth of
    the probes asleep, and the points that a camera inside it sees."""
    d, case = s.desc, s.case
    probes = _grid(d)
    lo, hi = probes[0] - 0.45 * d.spacing[0], probes[-1] + 0.45 * d.spacing[0]
    P = len(probes)

    def wall(o, v):
        t = torch.maximum((lo - o) / v, (hi - o) / v)
        return t.min(-1)

    rnd = lambda *shape: torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    k, ph = 0.4 * (rnd(3, 3) - 0.5), 6.28 * rnd(3)
    v = _texel_dirs(d.irr_n)
    m = 0.6 + 0.3 * torch.sin(probes @ k + ph)[:, None, None] + 0.25 * (v @ (2 * rnd(3, 3) - 1))[None].clamp(-0.9, 0.9)
    e = _bordered((m.clamp_min(0.02) * (0.9 + 0.2 * rnd(P, d.irr_n, d.irr_n, 1))) ** (1.0 / d.gamma))
    v = _texel_dirs(d.dist_n)
    t = wall(probes[:, None, None], v[None])[0] * (0.6 + 0.4 * rnd(P, d.dist_n, d.dist_n))   # something may stand before the wall
    t = t.clamp_max(d.t_max)
    mom = _bordered(torch.stack([t, t * t * (1.0 + 0.05 * rnd(*t.shape))], -1))
    s.irr = torch.zeros((P, d.irr_n + 2, d.irr_n + 2, 4), device="cuda")
    s.irr[..., :3] = e
    s.dist = mom.float()
    if d.irr_format == FP16:
        s.irr, s.dist = s.irr.half(), s.dist.half()
    stored = s.irr
    if d.irr_format == RGB9E5:      # shared exponent 15 + 1: steps of 2^-8
        q = (s.irr[..., :3].double() * 256.0).round().clamp(0, 511).long()
        stored = (q[..., 0] | (q[..., 1] << 9) | (q[..., 2] << 18) | (16 << 27)).to(torch.int64)
        stored = torch.where(stored >= 2 ** 31, stored - 2 ** 32, stored).to(torch.int32)
        s.irr = torch.nn.functional.pad(q.double() / 256.0, (0, 1))
    s.states = torch.where(rnd(P) < 0.1, SLEEPING, VIGILANT).to(torch.uint8)
    for which, b in enumerate((stored, s.dist, s.states)):
        s.vol.set_buffer(which, b)
    mid, ext = 0.5 * (lo + hi), hi - lo
    cam = (mid + 0.2 * ext * (rnd(3) - 0.5)).float().double()
    s.cam = tuple(float(c) for c in cam)
    w, h = case["width"], case["height"]
    y, x = torch.meshgrid((torch.arange(h, device="cuda") + 0.5) / h * 2 - 1, (torch.arange(w, device="cuda") + 0.5) / w * 2 - 1, indexing="ij")
    a = 6.28 * rnd(1)[0]
    th = math.tan(math.radians(30.0))
    right, fwd = torch.stack([a.cos(), 0 * a, -a.sin()]), torch.stack([a.sin(), 0 * a - 0.2, a.cos()])
    up = torch.tensor([0.0, 1.0, 0.0], dtype=torch.float64, device="cuda")
    dirs = (fwd + x.double().reshape(-1, 1) * th * w / h * right - y.double().reshape(-1, 1) * th * up)
    dirs = dirs / dirs.norm(dim=-1, keepdim=True)
    t, axis = wall(cam[None], dirs)
    n = -torch.nn.functional.one_hot(axis, 3).double() * torch.sign(dirs)
    s.pos = (cam + t[:, None] * dirs).float().contiguous()
    s.nrm = n.float().contiguous()
    s.dirs = dirs.float().contiguous()
    s.out = torch.empty_like(s.pos)


def _surface_points(model, n, gen):
    """Points spread over the boxes and the shell by area, a millimetre off the surface."""
    v, t = (torch.tensor(a, device="cuda") for a in model.arrays()[:2])
    p = v[t.long()]
    c = torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
    area = c.norm(dim=-1)
    cdf = area.double().cumsum(0)
    pick = torch.searchsorted(cdf, torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * cdf[-1]).clamp_max(len(t) - 1)
    u = torch.rand((n, 2), generator=gen, device="cuda")
    u = torch.where((u.sum(-1) > 1)[:, None], 1 - u, u)
    p, nn = p[pick], c[pick] / area[pick][:, None]
    x = p[:, 0] + u[:, :1] * (p[:, 1] - p[:, 0]) + u[:, 1:] * (p[:, 2] - p[:, 0]) + 1e-3 * nn
    return x.contiguous(), nn.contiguous()


# ---------------------------------------------------------------------------
# The same pass in 64 bits
# ---------------------------------------------------------------------------

def _t64(a):
    return torch.as_tensor(np.asarray(a, np.float32), device="cuda").double()


class _Boxes:
    """Closest hit of rays with a box scene, every ray against every box."""

    def __init__(self, m):
        self.lo, self.hi = _t64(m.lo), _t64(m.hi)
        self.obj = torch.as_tensor(m.box_obj, device="cuda").long()
        self.casts = torch.as_tensor(m.casts, device="cuda").bool()
        self.shell = None if m.shell is None else (_t64(m.shell[0]), _t64(m.shell[1]))
        self.rects = [(a, g, _t64(lo), _t64(hi), o, e) for a, g, lo, hi, o, e in m.rects]

    def _slabs(self, o, inv):
        tn = tf = None
        for a in range(3):
            p = (self.lo[:, a] - o[:, a:a + 1]) * inv[:, a:a + 1]
            q = (self.hi[:, a] - o[:, a:a + 1]) * inv[:, a:a + 1]
            n, f = torch.minimum(p, q), torch.maximum(p, q)
            tn, tf = (n, f) if a == 0 else (torch.maximum(tn, n), torch.minimum(tf, f))
        return tn, tf

    def _rect(self, o, d, r):
        a, g, lo, hi, _, _ = r
        t = (lo[a] - o[:, a]) / d[:, a]
        x = o + t[:, None] * d
        u, w = (a + 1) % 3, (a + 2) % 3
        ok = (t > 0) & (x[:, u] >= lo[u]) & (x[:, u] <= hi[u]) & (x[:, w] >= lo[w]) & (x[:, w] <= hi[w])
        return torch.where(ok, t, math.inf)

    def _pieces(self, n):
        step = max(1, (1 << 25) // max(1, len(self.lo)))
        return [slice(k, k + step) for k in range(0, n, step)]

    def closest(self, o, d):
        """t (inf on a miss), the surface's normal, whether the front was hit, object, emitter."""
        n = len(o)
        t, nrm = torch.full((n,), math.inf, dtype=torch.float64, device="cuda"), torch.zeros_like(d)
        front, obj = torch.zeros(n, dtype=torch.bool, device="cuda"), torch.zeros(n, dtype=torch.long, device="cuda")
        em = torch.full((n,), -1, dtype=torch.long, device="cuda")
        for c in self._pieces(n) if len(self.lo) else []:
            tn, tf = self._slabs(o[c], 1.0 / d[c])
            k = torch.where((tn <= tf) & (tf > 0), torch.where(tn > 0, tn, tf), math.inf)
            t[c], i = k.min(1)
            front[c] = tn.gather(1, i[:, None])[:, 0] > 0
            obj[c] = self.obj[i]
            p, q = (self.lo[i] - o[c]) / d[c], (self.hi[i] - o[c]) / d[c]
            axis = torch.where(front[c], torch.minimum(p, q).argmax(-1), torch.maximum(p, q).argmin(-1))
            out = torch.nn.functional.one_hot(axis, 3).double() * torch.sign(d[c])
            nrm[c] = torch.where(front[c][:, None], -out, out)      # entered from outside, or left from inside
        if self.shell is not None:
            q = torch.maximum((self.shell[0] - o) / d, (self.shell[1] - o) / d)
            k, axis = q.min(-1)
            near = k < t
            t = torch.where(near, k, t)
            front, obj = front | near, torch.where(near, 0, obj)
            nrm = torch.where(near[:, None], -torch.nn.functional.one_hot(axis, 3).double() * torch.sign(d), nrm)
        for r in self.rects:
            k = self._rect(o, d, r)
            near = k < t
            t, obj, em = torch.where(near, k, t), torch.where(near, r[4], obj), torch.where(near, r[5], em)
            front = torch.where(near, d[:, r[0]] * r[1] < 0, front)
            axis = torch.zeros(3, dtype=torch.float64, device="cuda")
            axis[r[0]] = r[1]
            nrm = torch.where(near[:, None], axis, nrm)
        return t, nrm, front, obj, em

    def blocked(self, o, d):
        """Whether a ray of the one direction d meets anything that casts shadows."""
        got = torch.zeros(len(o), dtype=torch.bool, device="cuda")
        d = d.expand_as(o)
        for c in self._pieces(len(o)) if len(self.lo) else []:
            tn, tf = self._slabs(o[c], 1.0 / d[c])
            got[c] = ((tn <= tf) & (tf > 0) & self.casts[self.obj]).any(1)
        if self.shell is not None and self.casts[0]:
            got |= True
        for r in self.rects:
            if self.casts[r[4]]:
                got |= torch.isfinite(self._rect(o, d, r))
        return got


_M64 = (1 << 64) - 1


def _mix(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _frame_dirs(seed, frame, R):
    """Spherical Fibonacci under the frame's random rotation (SplitMix64, Shoemake's quaternion)."""
    st, u = _mix((seed & _M64) ^ _mix((frame + 0x9E3779B97F4A7C15) & _M64)), []
    for _ in range(3):
        st = (st + 0x9E3779B97F4A7C15) & _M64
        u.append((_mix(st) >> 11) / 9007199254740992.0)
    a, b = math.sqrt(1 - u[0]), math.sqrt(u[0])
    x, y = a * math.sin(2 * math.pi * u[1]), a * math.cos(2 * math.pi * u[1])
    z, w = b * math.sin(2 * math.pi * u[2]), b * math.cos(2 * math.pi * u[2])
    m = torch.tensor([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                      [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                      [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]],
                     dtype=torch.float64, device="cuda")
    i = torch.arange(R, dtype=torch.float64, device="cuda")
    phi = 2 * math.pi * torch.frac(i * 0.61803398874989484820)
    c = 1 - (2 * i + 1) / R
    r = (1 - c * c).clamp_min(0).sqrt()
    return torch.stack([phi.cos() * r, phi.sin() * r, c], -1) @ m.T


def _oct(v):
    p = v[:, :2] / v.abs().sum(-1, keepdim=True)
    f = (1 - p.abs().flip(-1)) * torch.where(p >= 0, 1.0, -1.0)
    return torch.where(v[:, 2:] < 0, f, p)


def _taps(v, n):
    """Texel indices [N, 4] and weights [N, 4] of a bilinear lookup in a bordered tile."""
    s = (0.5 + (_oct(v) + 1) * 0.5 * n).nan_to_num()       # no direction (a background pixel): any texel
    f = s.floor().clamp(0, n)
    t, f = s - f, f.long()
    at = f[:, 1] * (n + 2) + f[:, 0]
    x, y = t[:, 0], t[:, 1]
    return (torch.stack([at, at + 1, at + n + 2, at + n + 3], -1),
            torch.stack([(1 - x) * (1 - y), x * (1 - y), (1 - x) * y, x * y], -1))


def _query(desc, irr, dist, active, x, n, wo, look=None):
    """Mean radiance M at points; irr [P, tile, 3], dist [P, tile, 2], 64 bits."""
    sp, org = _t64(desc.spacing), _t64(desc.origin)
    cnt = torch.tensor(desc.counts, device="cuda")
    D = sp.min()
    xb = x + (0.2 * n + 0.8 * wo) * (0.75 * D * float(np.float32(desc.self_shadow_bias)))
    g = ((xb - org) / sp).nan_to_num()
    base = torch.minimum(g.floor().clamp_min(0), (cnt - 2).double())
    fr = (g - base).clamp(0, 1)
    at, w4 = _taps(n if look is None else look, desc.irr_n)
    den, acc = 0.0, 0.0
    for c in range(8):
        o = torch.tensor([c & 1, (c >> 1) & 1, c >> 2], device="cuda")
        k = base.long() + o
        p = k[:, 0] + cnt[0] * (k[:, 1] + cnt[1] * k[:, 2])
        xp = org + k.double() * sp
        wt = torch.where(o.bool(), fr, 1 - fr).prod(-1)
        dp = xp - x
        ld = dp.norm(dim=-1)
        cw = torch.where(ld > 0, (n * dp).sum(-1) / ld, 1.0)
        wb = ((1 + cw) * 0.5) ** 2 + 0.2
        pv = xb - xp
        r = pv.norm(dim=-1)
        da, dw = _taps(pv / r[:, None].clamp_min(1e-300), desc.dist_n)
        mom = (dist[p[:, None], da] * dw[..., None]).sum(1)
        var = (mom[:, 1] - mom[:, 0] ** 2).clamp_min(0)
        dr = r - mom[:, 0]
        ch = torch.where((r > 0) & (dr > 0), var / (var + dr * dr).clamp_min(1e-300), 1.0)
        w = wt * wb * ch.clamp_min(1e-6) * active[p]
        e = (irr[p[:, None], at] * w4[..., None]).sum(1)
        e = torch.where(e > 0, e.clamp_min(1e-300) ** (0.5 * desc.gamma), 0.0)
        acc, den = acc + w[:, None] * e, den + w
    return torch.where(den[:, None] > 0, acc / den[:, None].clamp_min(1e-300), 0.0) ** 2


def _irradiance(desc, irr, dist, active, pos, nrm, cam):
    out = torch.zeros((len(pos), 3), dtype=torch.float64, device="cuda")
    for c in range(0, len(pos), 1 << 18):
        x, n = pos[c:c + (1 << 18)].double(), nrm[c:c + (1 << 18)].double()
        wo = _t64(cam) - x
        l = wo.norm(dim=-1, keepdim=True)
        M = _query(desc, irr, dist, active, x, n, torch.where(l < 1e-6, n, wo / l))
        out[c:c + (1 << 18)] = math.pi * torch.where((n != 0).any(-1, keepdim=True), M, 0.0)
    return out


def _flat(t, c):
    return t[..., :c].double().reshape(len(t), -1, c)


def _records(desc, model, lights, boxes, dirs, probes, query, albedo=None, emit=None):
    """Radiance [A, R, 3] and distance [A, R] of every ray of the probes (positions [A, 3]);
    query(x, n, wo) is the previous frame's mean radiance, or None where it is zero."""
    albedo = _t64(model.albedo) if albedo is None else albedo
    emit = _t64(model.emit) if emit is None else emit
    A, R = len(probes), len(dirs)
    o, d = probes.repeat_interleave(R, 0), dirs.repeat(A, 1)
    t, n, front, obj, em = boxes.closest(o, d)
    miss = torch.isinf(t)
    rad = torch.zeros((A * R, 3), dtype=torch.float64, device="cuda")
    rad[miss] = _t64(lights.sky_a) + _t64(lights.sky_b) * (d[miss] @ _t64(lights.sky_up))[:, None]
    depth = torch.where(front | miss, t, 0.2 * t).clamp_max(float(np.float32(desc.t_max)))
    h = (front & ~miss).nonzero()[:, 0]
    dh, nh = d[h], n[h]
    x = o[h] + t[h, None] * dh
    tol = -_t64(lights.sun_dir)
    cosl = nh @ tol
    s = (cosl > 0).nonzero()[:, 0]
    lit = torch.zeros(len(h), dtype=torch.bool, device="cuda")
    lit[s] = ~boxes.blocked(x[s] + 1e-4 * (1 + x[s].norm(dim=-1, keepdim=True)) * nh[s], tol)
    direct = torch.where(lit, cosl, 0.0)[:, None] * _t64(lights.sun_irradiance) / math.pi
    M = 0.0 if query is None else torch.cat([query(x[c], nh[c], -dh[c]) for c in torch.arange(len(h), device="cuda").split(1 << 18)])
    Le = torch.where((em[h] >= 0)[:, None], emit[em[h].clamp_min(0)], 0.0) if len(emit) else 0.0
    rad = rad.index_copy(0, h, Le + albedo[obj[h]] * (direct + M))
    return rad.view(A, R, 3), depth.view(A, R)


def _blend(desc, dirs, rad, depth):
    """Encoded irradiance [A, n, n, 3] and distance moments [A, m, m, 2] of this frame's rays, and
    whether any ray reaches a texel."""
    wi = (_texel_dirs(desc.irr_n) @ dirs.T).clamp_min(0)
    wd = (_texel_dirs(desc.dist_n) @ dirs.T).clamp_min(0) ** float(np.float32(desc.dist_cos_power))
    si, sd = wi.sum(-1), wd.sum(-1)
    m = torch.einsum("yxr,arc->ayxc", wi, rad) / si.clamp_min(1e-300)[..., None]
    # the root of zero has no derivative that counts
    e = m if desc.gamma == 1.0 else torch.where(m > 0, m.clamp_min(1e-300) ** (1.0 / desc.gamma), 0.0)
    mom = torch.einsum("yxr,arc->ayxc", wd, torch.stack([depth, depth ** 2], -1)) / sd.clamp_min(1e-300)[..., None]
    return e, mom, si > 0, sd > 0


def _exact_update(s, frame):
    """Atlases [P, tile, C] and states after the frame that run() makes from this state."""
    d = s.desc
    boxes, states = _Boxes(s.model), s.states
    irr, dist = _flat(s.irr, 3), _flat(s.dist, 2)
    active = ((states == NEWLY) | (states == VIGILANT)).double()
    act = active.nonzero()[:, 0]
    dirs = _frame_dirs(d.seed, frame, d.rays_per_probe)
    rad, depth = _records(d, s.model, s.lights, boxes, dirs, _grid(d)[act],
                          lambda x, n, wo: _query(d, irr, dist, active, x, n, wo))
    e, mom, ri, rd = _blend(d, dirs, rad, depth)
    newly = (states[act] == NEWLY)[:, None, None]
    N, M = d.irr_n + 2, d.dist_n + 2
    old = irr.view(-1, N, N, 3)[act, 1:-1, 1:-1]
    change = (e - old).abs().amax(-1)
    hyst = float(np.float32(d.hysteresis_irr))
    a = torch.where(newly, 0.0, torch.full_like(change, hyst))
    a = torch.where(change > float(np.float32(d.thr_low)), (a - float(np.float32(d.thr_step))).clamp_min(0), a)
    a = torch.where(change > float(np.float32(d.thr_high)), 0.0, a)[..., None]
    irr = irr.view(-1, N, N, 3).clone()
    irr[act] = _bordered(torch.where(ri[..., None], (1 - a) * e + a * old, old))
    old = dist.view(-1, M, M, 2)[act, 1:-1, 1:-1]
    b = torch.where(newly, 0.0, torch.full_like(old[..., 0], hyst))[..., None]
    dist = dist.view(-1, M, M, 2).clone()
    dist[act] = _bordered(torch.where(rd[..., None], (1 - b) * mom + b * old, old))
    return irr, dist, active


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits.  None for the cascades (millions of rays
    against a landscape's triangles) and for a level's first frame (10^11 box tests, and the
    optimizer moves a probe to another place when two hits are within rounding)."""
    kind = case["kind"]
    if kind in ("cascade", "load"):
        return None
    s = prepare(case, seed)
    if kind in ("frame", "noalloc"):
        irr, dist, active = _exact_update(s, s.frame)
        got = {"irr": irr, "dist": dist, "states": None}
        if kind == "frame":
            got["E"] = _irradiance(s.desc, irr.flatten(1, 2), dist.flatten(1, 2), active, s.pos, s.nrm, s.cam)
        return got
    if kind in ("query", "texels"):
        irr, dist, active = _flat(s.irr, 3), _flat(s.dist, 2), (s.states == VIGILANT).double()
        if kind == "texels":
            irr.requires_grad_(True)
            E = []
            for c in range(0, len(s.pos), 1 << 17):
                x, n = s.pos[c:c + (1 << 17)].double(), s.nrm[c:c + (1 << 17)].double()
                wo = _t64(s.cam) - x
                e = math.pi * _query(s.desc, irr, dist, active, x, n, wo / wo.norm(dim=-1, keepdim=True))
                (e * s.dE[c:c + (1 << 17)].double()).sum().backward()
                E.append(e.detach())
            return {"E": torch.cat(E), "grad": torch.nn.functional.pad(irr.grad, (0, 1)).view(s.irr.shape)}
        if not case["glossy"]:
            return _irradiance(s.desc, irr, dist, active, s.pos, s.nrm, s.cam)
        out = []
        for x, n, w in zip(*[t.double().split(1 << 18) for t in (s.pos, s.nrm, s.dirs)]):
            r = w - 2 * (w * n).sum(-1, keepdim=True) * n
            out.append(_query(s.desc, irr, dist, active, x, n, -w, r / r.norm(dim=-1, keepdim=True)))
        return torch.cat(out)
    if kind == "train":
        d, boxes = s.desc, _Boxes(s.model)
        alb, em = (t.detach().double().requires_grad_(True) for t in (s.albedo, s.emit))
        probes = _grid(d)
        on = torch.ones(len(probes), dtype=torch.float64, device="cuda")
        irr = dist = None
        for f in range(case["frames"]):
            dirs = _frame_dirs(d.seed, f, d.rays_per_probe)
            prev = (irr, dist)
            rad, depth = _records(d, s.model, s.lights, boxes, dirs, probes,
                                  None if f == 0 else lambda x, n, wo: _query(d, *prev, on, x, n, wo), alb, em)
            e, mom, _, _ = _blend(d, dirs, rad, depth)
            irr, dist = _bordered(e).flatten(1, 2), _bordered(mom).flatten(1, 2)
        leaf, E = irr.detach().requires_grad_(True), []
        for x, n, y in zip(*[t.double().split(1 << 17) for t in (s.pos, s.nrm, s.target)]):
            wo = _t64(s.cam) - x
            c = math.pi * _query(d, leaf, dist, on, x, n, wo / wo.norm(dim=-1, keepdim=True))
            (((c - y) ** 2).sum() / s.target.numel()).backward()
            E.append(c.detach())
        irr.backward(leaf.grad)
        return {"E": torch.cat(E), "albedo": alb.grad, "emit": em.grad}
    # the camera's rays, as a pinhole's definition has them
    f = _t64(s.fwd)
    f = f / f.norm()
    r = torch.linalg.cross(f, _t64((0.0, 1.0, 0.0)))
    r = r / r.norm()
    u = torch.linalg.cross(r, f)
    w, h, th = case["width"], case["height"], math.tan(math.radians(30.0))
    ar = lambda k: (torch.arange(k, dtype=torch.float64, device="cuda") + 0.5) / k * 2 - 1  # noqa: E731
    y, x = torch.meshgrid(ar(h), ar(w), indexing="ij")
    d = f + x.reshape(-1, 1) * th * (w / h) * r - y.reshape(-1, 1) * th * u
    d = d / d.norm(dim=-1, keepdim=True)
    o = _t64(s.cam).expand_as(d)
    t, n, _, _, _ = _Boxes(s.model).closest(o, d)
    hit = torch.isfinite(t)[:, None]
    return [torch.where(hit, o + torch.where(hit, t[:, None], 0.0) * d, 0.0), torch.where(hit, n, 0.0)]
