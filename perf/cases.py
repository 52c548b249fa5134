"""The work that a user of this ray tracer has it do, as measurable cases.

A program that uses the library loads meshes into a scene (rg_blas_build),
places and moves instances (rg_tlas_build, rg_tlas_refit), asks ray queries
(rg_trace_rays), renders frames (rg_render), filters them (rg_fxaa), serves
many render requests at once (rg_server_*), and sorts pairs
(rg_radix_sort_pairs).  listed() holds one or more cases of each, from the
smallest calls to the largest workload of bench.py; draw() gives others of
the same ranges.

Scenes follow the repository's own configurations (scenegen): the tiny room
(ground and cubes, 64x64), the medium scene (64 instances of four meshes,
about 158,000 triangles, four lights, 1920x1080 at depth 4), the large one
(4,096 instances of 16 meshes, 1.94M triangles, 2^24 rays), and the serving
requests.  Everything is made from the seed, on the GPU.
"""
import math

import numpy as np
import torch

import paper_2001_09792_gb300 as rg

DEV = "cuda"


def listed():
    return [
        # a pick under the cursor, a line of sight, a footstep probe: a handful of rays, all latency
        dict(name="pick 64 rays", kind="query", instances=3, tris=26, meshes=2, rays=64, mode="closest", update="none",
             compressed=False),
        # one bounce of a lighting bake or a lidar sweep over a medium scene: incoherent closest hits
        dict(name="bounce 1M rays", kind="query", instances=64, tris=158000, meshes=4, rays=1 << 20, mode="closest",
             update="none", compressed=False),
        # a simulation tick: 4,096 moved instances, the tree rebuilt, an odd number of short visibility rays
        dict(name="tick 4096 instances", kind="query", instances=4096, tris=500000, meshes=16, rays=65537, mode="any",
             update="rebuild", compressed=False),
        # the benchmark's step: 4,096 moved instances, rebuild, 2^24 closest hits and 2^24 any hits
        dict(name="large step", kind="query", instances=4096, tris=1940000, meshes=16, rays=1 << 24, mode="both",
             update="rebuild", compressed=False),
        # closest and any hits against the compressed BVH, for a program that keeps its scenes in that form
        dict(name="compressed 2M rays", kind="query", instances=64, tris=158000, meshes=4, rays=1 << 21, mode="both",
             update="none", compressed=True),
        # a thumbnail or preview frame of the tiny room, moved since the last one
        dict(name="frame 64x64", kind="frame", instances=3, tris=26, meshes=2, width=64, height=64, depth=1,
             update="refit", compressed=False),
        # the medium frame: instances moved, the tree rebuilt, 1920x1080 at depth 4
        dict(name="frame 1920x1080", kind="frame", instances=64, tris=158000, meshes=4, width=1920, height=1080, depth=4,
             update="rebuild", compressed=False),
        # the anti-aliasing pass of a 4K frame
        dict(name="fxaa 3840x2160", kind="fxaa", width=3840, height=2160),
        # a mesh that changes its shape (cloth, destruction): fast build, then a query against it
        dict(name="load 20480 fast", kind="build", tris=20480, meshes=1, sah=False, morton63=False, compressed=False,
             rays=16384),
        # loading the medium scene's meshes for trace speed, then a query against them
        dict(name="load 158000 sah", kind="build", tris=158000, meshes=4, sah=True, morton63=False, compressed=False,
             rays=65536),
        # render requests of several scenes, sizes and depths that arrive together
        dict(name="serve 8 requests", kind="serve", scenes=3, requests=8, largest=3),
        # sorting (key, value) pairs, a ragged million
        dict(name="sort 1000003 pairs", kind="sort", pairs=1000003, bits=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind, and sizes spread over the logarithm of its range."""
    kind = rng.choice(["query", "query", "query", "frame", "frame", "fxaa", "build", "build", "serve", "sort"])
    if kind == "query":
        big = rng.random() < 0.5
        return dict(kind="query", instances=_log_int(rng, 512, 4096) if big else _log_int(rng, 3, 511),
                    tris=_log_int(rng, 26, 1900000), meshes=16 if big else 4, rays=_log_int(rng, 64, 1 << 23) | 1,
                    mode=rng.choice(["closest", "any", "both"]), update=rng.choice(["none", "rebuild", "refit"]),
                    compressed=rng.random() < 0.2)
    if kind == "frame":
        return dict(kind="frame", instances=_log_int(rng, 3, 256), tris=_log_int(rng, 26, 400000), meshes=4,
                    width=_log_int(rng, 64, 1920), height=_log_int(rng, 64, 1080), depth=rng.randint(1, 5),
                    update=rng.choice(["rebuild", "refit"]), compressed=rng.random() < 0.2)
    if kind == "fxaa":
        return dict(kind="fxaa", width=_log_int(rng, 64, 3840), height=_log_int(rng, 64, 2160))
    if kind == "build":
        return dict(kind="build", tris=_log_int(rng, 100, 400000), meshes=rng.randint(1, 4), sah=rng.random() < 0.5,
                    morton63=rng.random() < 0.3, compressed=rng.random() < 0.2, rays=_log_int(rng, 64, 65536))
    if kind == "serve":
        return dict(kind="serve", scenes=rng.randint(1, 4), requests=rng.randint(1, 10), largest=rng.randint(0, 3))
    return dict(kind="sort", pairs=_log_int(rng, 1000, 1 << 24), bits=rng.choice([32, 32, 64]))


# ---------------------------------------------------------------- geometry

def _bumps(gen, x, y, z, octaves=4):
    """Smooth seeded noise in [-1, 1] at points (sums of plane waves of doubling frequency)."""
    total, amp_sum = torch.zeros_like(x), 0.0
    for k in range(octaves):
        for _ in range(3):
            w = torch.randn(4, generator=gen, dtype=torch.float64).tolist()
            f = 2.0 * 2 ** k
            total += 0.5 ** k * torch.sin(f * (w[0] * x + w[1] * y + w[2] * z) + 6.28 * w[3])
            amp_sum += 0.5 ** k
    return total / amp_sum


def _surface(kind, tris, radius, gen):
    """A mesh of about `tris` triangles of a grid of quads: a bumpy ball (poles
    of degenerate triangles, as a UV sphere has), a ring, or a patch of
    terrain; centred, of the given bounding radius.  (vertices, indices) on
    the GPU."""
    nv = max(3, int(math.sqrt(tris / 4)))
    nu = max(3, tris // (2 * nv))
    u = torch.arange(nu + 1, device=DEV, dtype=torch.float64) / nu
    w = torch.arange(nv + 1, device=DEV, dtype=torch.float64) / nv
    U, W = torch.meshgrid(u, w, indexing="ij")
    if kind == "terrain":
        x, z = 2 * U - 1, 2 * W - 1
        p = torch.stack([x, 0.125 * _bumps(gen, x, 0 * x, z), z], -1)
    elif kind == "ring":
        a, b = 2 * math.pi * U, 2 * math.pi * W
        r = 1 + 0.35 * torch.cos(b)
        p = torch.stack([r * torch.cos(a), 0.35 * torch.sin(b), r * torch.sin(a)], -1)
    else:
        a, b = 2 * math.pi * U, math.pi * W
        p = torch.stack([torch.sin(b) * torch.cos(a), torch.cos(b), torch.sin(b) * torch.sin(a)], -1)
        p = p * (1 + 0.1 * _bumps(gen, p[..., 0], p[..., 1], p[..., 2]))[..., None]
    p = p.reshape(-1, 3)
    p = p - (p.amin(0) + p.amax(0)) / 2
    p = p * (radius / p.norm(dim=1).max())
    i = torch.arange(nu, device=DEV)[:, None] * (nv + 1) + torch.arange(nv, device=DEV)[None, :]
    a, b, c, d = i, i + 1, i + nv + 2, i + nv + 1
    idx = torch.stack([torch.stack([a, b, c], -1), torch.stack([a, c, d], -1)], -2)
    return p.float().contiguous(), idx.reshape(-1, 3).int().contiguous()


def _room_meshes():
    """The tiny room's meshes: a unit cube and a 10x10 ground quad at y = -0.5."""
    v = np.array([[x, y, z] for x in (-.5, .5) for y in (-.5, .5) for z in (-.5, .5)], np.float32)
    quads = [(0, 1, 3, 2), (4, 6, 7, 5), (0, 4, 5, 1), (2, 3, 7, 6), (0, 2, 6, 4), (1, 5, 7, 3)]
    i = np.array([t for q in quads for t in ((q[0], q[1], q[2]), (q[0], q[2], q[3]))], np.int32)
    gv = np.array([[-5, -.5, -5], [-5, -.5, 5], [5, -.5, 5], [5, -.5, -5]], np.float32)
    gi = np.array([[0, 1, 2], [0, 2, 3]], np.int32)
    return [(torch.from_numpy(v).to(DEV), torch.from_numpy(i).to(DEV)),
            (torch.from_numpy(gv).to(DEV), torch.from_numpy(gi).to(DEV))]


def _meshes(case, seed, radius):
    """case["meshes"] meshes whose triangle counts fall geometrically and add up to about case["tris"]."""
    gen = torch.Generator().manual_seed(seed)
    m = case["meshes"]
    ratio = 0.2 if m <= 4 else 0.66
    w = [ratio ** k for k in range(m)]
    return [_surface(("terrain", "ball", "ring")[k % 3], max(18, int(case["tris"] * w[k] / sum(w))), radius, gen)
            for k in range(m)]


def _rotations(rng, n):
    q = rng.normal(size=(n, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    w, x, y, z = q.T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).reshape(n, 3, 3)


class Scene:
    """A built scene with its tables, as a program keeps it; freed with the object."""

    def __init__(self, case, seed):
        rng = np.random.default_rng(seed)
        n = case["instances"]
        room = n == 3 and case["tris"] <= 26
        if room:
            self.half = 5.0
            self.meshes = _room_meshes()
            ang = rng.uniform(0, 2 * math.pi, 2)
            M = np.zeros((3, 3, 4), np.float32)
            M[0, :, :3] = np.eye(3)
            for k, x in ((1, -0.6), (2, 1.6)):
                c, s = math.cos(ang[k - 1]), math.sin(ang[k - 1])
                M[k, :, :3] = [[c, 0, s], [0, 1, 0], [-s, 0, c]]
                M[k, :, 3] = [x + rng.uniform(-.3, .3), 0, rng.uniform(-1, .5)]
            mesh_id = np.array([1, 0, 0])
            self.mats = (np.zeros(3, np.uint32), np.full((3, 3), 0.8, np.float32), np.ones(3, np.float32))
            self.lights = (np.array([[2, 4, 3]], np.float32), np.ones((1, 3), np.float32))
            self.camera = dict(eye=(0, 2, 5), target=(0, 0, 0), up=(0, 1, 0), vfov=60.0)
        else:
            radius = 10.0 if n <= 512 else 5.0
            self.half = (50.0 if n <= 512 else 100.0) * (n / (64.0 if n <= 512 else 512.0)) ** (1 / 3)
            self.meshes = _meshes(case, seed, radius)
            # a scene of many instances places its small meshes more often
            p = np.array([i.shape[0] for _, i in self.meshes], float) ** (-0.77 if n > 512 else 0.0)
            mesh_id = rng.choice(len(self.meshes), n, p=p / p.sum())
            M = np.zeros((n, 3, 4), np.float32)
            M[:, :, :3] = _rotations(rng, n) * rng.uniform(0.5, 2.0, (n, 1, 1))
            M[:, :, 3] = rng.uniform(-self.half, self.half, (n, 3))
            r = rng.random(n)
            t = np.where(r < 0.6, 0, np.where(r < 0.8, 1, 2)).astype(np.uint32)
            alb = np.where(t[:, None] == 0, rng.uniform(0.2, 0.9, (n, 3)), 0.9).astype(np.float32)
            self.mats = (t, alb, np.where(t == 2, 1.5, 1.0).astype(np.float32))
            lp = rng.uniform(-1, 1, (4, 3)) * self.half
            lp[:, 1] = rng.uniform(0.8, 1.2, 4) * self.half
            self.lights = (lp.astype(np.float32), np.full((4, 3), 0.25, np.float32))
            self.camera = dict(eye=(0, 0, 2 * self.half), target=(0, 0, 0), up=(0, 1, 0), vfov=60.0)
        self.room, self.M, self.mesh_id = room, M, mesh_id
        flags = (rg.RG_SCENE_COMPRESSED if case.get("compressed") else 0) | rg.RG_SCENE_SAH_TLAS * (n > 512)
        self.h = rg.rg_scene_create(flags=flags)
        ids = [rg.rg_blas_build(self.h, v, i, rg.RG_BLAS_SAH) for v, i in self.meshes]
        host = rg.pack_instances(M, [ids[m] for m in mesh_id], np.arange(n))
        self.inst = torch.from_numpy(host).to(DEV)
        rg.rg_tlas_build(self.h, self.inst)
        # the transforms of the next frame: every instance a little moved and turned
        moved = M.copy()
        if not room:
            moved[:, :, 3] += rng.normal(0, 1, (n, 3)).astype(np.float32)
        else:
            moved[1:, 0, 3] += rng.uniform(-.1, .1, 2).astype(np.float32)
        self.moved = moved
        host2 = host.copy()
        host2[:, :12] = moved.reshape(n, 12)
        self.inst_next = torch.from_numpy(host2).to(DEV)
        rg.rg_scene_set_materials(self.h, *self.mats)
        rg.rg_scene_set_lights(self.h, *self.lights)
        rg.rg_sync(self.h)

    def update(self, how):
        if how == "rebuild":
            rg.rg_tlas_build(self.h, self.inst_next)
        elif how == "refit":
            rg.rg_tlas_refit(self.h, self.inst_next)

    def __del__(self):
        if getattr(self, "h", None):
            rg.rg_scene_destroy(self.h)


def _rays(n, half, seed, reach=None):
    """n rays from points of the scene's box in all directions, unbounded or of lengths in `reach`."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    r = torch.empty((n, 8), device=DEV)
    r[:, 0:3] = (2 * torch.rand((n, 3), device=DEV, generator=g) - 1) * half
    d = torch.randn((n, 3), device=DEV, generator=g)
    r[:, 4:7] = d / d.norm(dim=1, keepdim=True)
    r[:, 3] = 0
    r[:, 7] = math.inf if reach is None else reach[0] + (reach[1] - reach[0]) * torch.rand(n, device=DEV, generator=g)
    return r


def _room_rays(r):
    """Rays over the tiny room start above its ground."""
    r[:, 1] = r[:, 1].abs() + 1.0
    r[:, 5] = -r[:, 5].abs()
    return r


def _picture(w, h, seed):
    """An image with what frames hold: flat regions, shading ramps, straight and curved edges, thin lines."""
    g = torch.Generator().manual_seed(seed)
    rnd = lambda *s: torch.rand(*s, generator=g).tolist()  # noqa: E731
    y, x = torch.meshgrid(torch.linspace(0, 1, h, device=DEV), torch.linspace(0, w / h, w, device=DEV), indexing="ij")
    img = torch.stack([0.2 + 0.1 * y, 0.3 + 0.1 * y, 0.5 + 0.2 * y], -1)
    for k in range(24):
        a = rnd(10)
        cx, cy, s = a[0] * w / h, a[1], 0.02 + 0.2 * a[2]
        if k % 3 == 0:
            m = (x - cx) ** 2 + (y - cy) ** 2 < s * s
        elif k % 3 == 1:
            c, q = math.cos(6.28 * a[3]), math.sin(6.28 * a[3])
            m = ((c * (x - cx) + q * (y - cy)).abs() < s) & ((c * (y - cy) - q * (x - cx)).abs() < 0.5 * s)
        else:
            c, q = math.cos(6.28 * a[3]), math.sin(6.28 * a[3])
            m = (c * (x - cx) + q * (y - cy)).abs() < 0.003
        col = torch.tensor(a[4:7], device=DEV) * (0.6 + 0.4 * torch.sin(3 * x + 6 * a[7] + 2 * y))[..., None]
        img = torch.where(m[..., None], col, img)
    return torch.cat([img, torch.ones_like(img[..., :1])], -1).contiguous()


# ---------------------------------------------------------------- a pass

SIZES = [(320, 240), (640, 480), (1280, 720), (1920, 1080), (3840, 2160)]


def _requests(case):
    """(scene, width, height, depth) of each request: the sizes and depths of the serving workload, in turn."""
    return [(k % case["scenes"], *SIZES[k % (case["largest"] + 1)], 1 + (3 * k) % 8) for k in range(case["requests"])]


class Server:
    """Resident scenes and a server over them; freed with the object."""

    def __init__(self, case, seed):
        spec = [dict(instances=64, tris=158000, meshes=4), dict(instances=3, tris=26, meshes=2)]
        self.scenes = [Scene(spec[k % 2 if k < 2 else 0], seed * 8 + k) for k in range(case["scenes"])]
        self.h = rg.rg_server_create()
        self.ids = [rg.rg_server_add_scene(self.h, s.h) for s in self.scenes]
        self.images = [torch.empty((h, w, 4), device=DEV) for _, w, h, _ in _requests(case)]

    def __del__(self):
        if getattr(self, "h", None):
            torch.cuda.synchronize()
            rg.rg_server_destroy(self.h)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "query":
        s = st["scene"] = Scene(case, seed)
        if case["mode"] != "any":
            st["rays"] = _rays(case["rays"], s.half, seed)
        if case["mode"] != "closest":
            st["short"] = _rays(case["rays"], s.half, seed + 7919, (1.0, 50.0))
        if s.room:
            for k in ("rays", "short"):
                if k in st:
                    _room_rays(st[k])
    elif kind == "frame":
        st["scene"] = Scene(case, seed)
    elif kind == "fxaa":
        st["image"] = _picture(case["width"], case["height"], seed)
    elif kind == "build":
        rng = np.random.default_rng(seed)
        m = case["meshes"]
        st["meshes"] = _meshes(case, seed, 10.0)
        M = np.zeros((m, 3, 4), np.float32)
        M[:, :, :3] = _rotations(rng, m)
        M[:, :, 3] = rng.uniform(-10, 10, (m, 3))
        st["M"] = M
        st["inst"] = torch.from_numpy(rg.pack_instances(M, np.arange(m))).to(DEV)  # BLAS ids count from 0
        st["rays"] = _rays(case["rays"], 15.0, seed)
    elif kind == "serve":
        st["server"] = Server(case, seed)
    elif kind == "sort":
        g = torch.Generator(device=DEV).manual_seed(seed)
        lo, hi, t = (-2 ** 31, 2 ** 31, torch.int32) if case["bits"] == 32 else (-2 ** 63, 2 ** 63 - 1, torch.int64)
        st["keys"] = torch.randint(lo, hi, (case["pairs"],), device=DEV, dtype=t, generator=g)
        st["vals"] = torch.arange(case["pairs"], device=DEV, dtype=torch.int32)
    return st


def _records(hits):
    """A closest-hit record: two ids, then t, u, v as float32 (views, no copies)."""
    return dict(ids=hits[:, :2], tuv=hits.view(torch.float32)[:, 2:])


def _query(h, st):
    out = {}
    if "rays" in st:
        out.update(_records(rg.rg_trace_rays(h, st["rays"], rg.RG_CLOSEST)))
    if "short" in st:
        # an any-hit query says occluded or not; which hit its record names is open
        out["occluded"] = rg.rg_trace_rays(h, st["short"], rg.RG_ANY)[:, 0] != -1
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "query":
        state["scene"].update(case["update"])
        return _query(state["scene"].h, state)
    if kind == "frame":
        s = state["scene"]
        s.update(case["update"])
        return rg.rg_render(s.h, s.camera, case["width"], case["height"], case["depth"])
    if kind == "fxaa":
        return rg.rg_fxaa(state["image"])
    if kind == "build":
        h = rg.rg_scene_create(flags=rg.RG_SCENE_COMPRESSED if case["compressed"] else 0)
        flags = (rg.RG_BLAS_SAH if case["sah"] else 0) | (rg.RG_MORTON63 if case["morton63"] else rg.RG_MORTON30)
        try:
            for v, i in state["meshes"]:
                rg.rg_blas_build(h, v, i, flags)
            rg.rg_tlas_build(h, state["inst"])
            out = _query(h, state)
            rg.rg_sync(h)
        finally:
            rg.rg_scene_destroy(h)
        return out
    if kind == "serve":
        sv = state["server"]
        for (k, w, h, depth), image in zip(_requests(case), sv.images):
            rg.rg_server_submit(sv.h, sv.ids[k], sv.scenes[k].camera, w, h, depth, image, sv.scenes[k].moved)
        rg.rg_server_drain(sv.h)
        rg.rg_server_poll(sv.h)
        return list(sv.images)
    return list(rg.rg_radix_sort_pairs(state["keys"], state["vals"]))


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Rays and records moved once, the tables and the trees read (or written)
    once, and per ray one descent of a perfectly separating tree: the slab
    tests (about 24 operations a box, two boxes a level) and one triangle."""
    kind = case["kind"]
    if kind == "sort":
        return dict(bytes=2 * case["pairs"] * (case["bits"] // 8 + 4), flops=0)
    if kind == "fxaa":
        px = case["width"] * case["height"]
        return dict(bytes=32 * px, flops=40 * px)
    if kind == "serve":
        px = [w * h for _, w, h, _ in _requests(case)]
        return dict(bytes=16 * sum(px) + 110 * 158000, flops=sum(px) * 60 * 24 * 2)
    tree = 110 * case["tris"]  # a triangle's 48 B and a node's 64 B
    if kind == "build":
        return dict(bytes=18 * case["tris"] + tree + 52 * case["rays"], flops=100 * case["tris"])
    levels = math.log2(case["instances"] + 1) + math.log2(max(2, case["tris"] / case["meshes"]))
    per_ray = 48 * levels + 60
    if kind == "frame":
        px = case["width"] * case["height"]
        return dict(bytes=16 * px + tree + 64 * case["instances"], flops=px * per_ray)
    n = case["rays"] * (2 if case["mode"] == "both" else 1)
    return dict(bytes=52 * n + min(tree, 110 * n * 2) + 64 * case["instances"], flops=n * per_ray)


# ---------------------------------------------------------------- in 64 bits

PAIRS = 1 << 23  # (ray, triangle) pairs tested at a time
MOST_TESTS = 2e10


def _soup(meshes, M, mesh_id):
    """Per instance: world-space triangles (n, 3, 3) in float64."""
    for m, k in zip(torch.from_numpy(np.asarray(M, np.float64)).to(DEV), mesh_id):
        v, i = meshes[int(k)]
        yield (v.double() @ m[:, :3].T + m[:, 3])[i.long()]


def _brute(soup, rays):
    """Nearest hit of each ray by testing every triangle of the instances
    whose bounding sphere it meets: (t, u, v, instance, primitive) in 64 bits,
    distances compared as float32, then by instance and primitive.  None when
    that is too much work."""
    r = rays.double()
    o, tmin, d, tmax = r[:, :3], r[:, 3], r[:, 4:7], r[:, 7]
    n = r.shape[0]
    best = torch.full((n, 3), 0.0, device=DEV, dtype=torch.float64)
    best[:, 0] = math.inf
    ids = torch.full((n, 2), -1, device=DEV)
    tests = 0
    for inst, tri in enumerate(soup):
        c = (tri.amin((0, 1)) + tri.amax((0, 1))) / 2
        rad = (tri - c).norm(dim=2).max() * 1.0001
        oc = o - c
        b, dd = (oc * d).sum(1), (d * d).sum(1)
        disc = b * b - dd * ((oc * oc).sum(1) - rad * rad)
        far = (-b + disc.clamp(min=0).sqrt()) / dd
        near = (-b - disc.clamp(min=0).sqrt()) / dd
        pick = ((disc >= 0) & (far >= tmin) & (near <= tmax) & (near.float() <= best[:, 0].float())).nonzero()[:, 0]
        tests += pick.numel() * tri.shape[0]
        if tests > MOST_TESTS:
            return None
        a, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
        step_t = min(tri.shape[0], 1 << 20)
        for p in pick.split(max(1, PAIRS // step_t)):
            for t0 in range(0, tri.shape[0], step_t):
                A, E1, E2 = a[t0:t0 + step_t][None], e1[t0:t0 + step_t][None], e2[t0:t0 + step_t][None]
                D, S = d[p][:, None], o[p][:, None] - A
                P = torch.linalg.cross(D.expand(-1, E2.shape[1], -1), E2.expand(p.numel(), -1, -1))
                det = (E1 * P).sum(2)
                Q = torch.linalg.cross(S, E1.expand_as(S))
                u, v, t = (S * P).sum(2) / det, (D * Q).sum(2) / det, (E2 * Q).sum(2) / det
                ok = (det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t >= tmin[p][:, None]) & (t <= tmax[p][:, None])
                t32 = torch.where(ok, t.float(), math.inf)
                m = t32.amin(1)
                at = torch.where(t32 == m[:, None], torch.arange(t32.shape[1], device=DEV), t32.shape[1]).amin(1)
                at = at.clamp(max=t32.shape[1] - 1)
                won = m < best[p, 0].float()  # instances and primitives come in ascending order
                q, w = p[won], at[won]
                row = won.nonzero()[:, 0]
                best[q] = torch.stack([t[row, w], u[row, w], v[row, w]], 1)
                ids[q] = torch.stack([torch.full_like(w, inst), t0 + w], 1)
    return best, ids


def _exact_room_frame(s, w, h):
    """The diffuse room at depth 1: ambient, and the Lambert term of the light
    where no triangle stands between; background where nothing is hit."""
    cam, f64 = s.camera, dict(device=DEV, dtype=torch.float64)
    eye, tgt, up = (torch.tensor(cam[k], **f64) for k in ("eye", "target", "up"))
    unit = lambda a: a / a.norm(dim=-1, keepdim=True)  # noqa: E731
    F = unit(tgt - eye)
    R = unit(torch.linalg.cross(F, up))
    U = torch.linalg.cross(R, F)
    th = math.tan(math.radians(cam["vfov"]) / 2)
    y, x = torch.meshgrid(torch.arange(h, **f64), torch.arange(w, **f64), indexing="ij")
    px, py = (2 * (x + 0.5) / w - 1) * (w / h) * th, (1 - 2 * (y + 0.5) / h) * th
    d = unit(px[..., None] * R + py[..., None] * U + F).reshape(-1, 3)
    n = d.shape[0]
    pack = lambda o, dd, t0, t1: torch.cat([o, torch.full((o.shape[0], 1), t0, **f64), dd, t1[:, None]], 1)  # noqa: E731
    rays = pack(eye.expand(n, 3), d, 0.0, torch.full((n,), math.inf, **f64))
    soup = list(_soup(s.meshes, s.moved, s.mesh_id))
    best, ids = _brute(soup, rays)
    hit = ids[:, 0] >= 0
    rgba = torch.zeros((n, 4), **f64)
    rgba[:, :3] = torch.tensor([0.2, 0.3, 0.5], device=DEV).double()
    k = hit.nonzero()[:, 0]
    tri = torch.stack([soup[i][p] for i, p in ids[k].tolist()])
    nrm = unit(torch.linalg.cross(tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]))
    nf = torch.where(((d[k] * nrm).sum(1) < 0)[:, None], nrm, -nrm)
    p = eye + best[k, :1] * d[k]
    eps = 1e-4 * p.abs().amax(1).clamp(min=1.0)
    os = p + eps[:, None] * nf
    alb = torch.from_numpy(s.mats[1]).to(DEV).double()[ids[k, 0]]
    col = alb * float(np.float32(0.1))
    for lp, li in zip(*(torch.from_numpy(a).to(DEV).double() for a in s.lights)):
        lv = lp - os
        dist = lv.norm(dim=1)
        cl = (nf * lv).sum(1) / dist
        shadow = _brute(soup, pack(os, lv / dist[:, None], 0.0, dist - eps))[1][:, 0] >= 0
        col += torch.where(((cl > 0) & ~shadow)[:, None], alb * li * cl[:, None], 0.0)
    rgba[k, :3], rgba[k, 3] = col, 1.0
    return rgba.reshape(h, w, 4)


def _exact_fxaa(img):
    """The filter as rg.h states it, in 64 bits."""
    c = img.double()
    h, w = c.shape[:2]
    lum = (0.299 * c[..., 0] + 0.587 * c[..., 1] + 0.114 * c[..., 2]).clamp(min=0).sqrt()
    Y, X = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
    at = lambda a, y, x: a[y.clamp(0, h - 1), x.clamp(0, w - 1)]  # noqa: E731

    def bilinear(a, py, px):
        fy, fx = py.floor(), px.floor()
        y0, x0, dy, dx = fy.long(), fx.long(), py - fy, px - fx
        if a.dim() == 3:
            dy, dx = dy[..., None], dx[..., None]
        top = torch.lerp(at(a, y0, x0), at(a, y0, x0 + 1), dx)
        return torch.lerp(top, torch.lerp(at(a, y0 + 1, x0), at(a, y0 + 1, x0 + 1), dx), dy)

    L = {(dy, dx): at(lum, Y + dy, X + dx) for dy in (-1, 0, 1) for dx in (-1, 0, 1)}
    M, N, S, W, E = L[0, 0], L[-1, 0], L[1, 0], L[0, -1], L[0, 1]
    five = torch.stack([M, N, S, W, E])
    rng_, hi = five.amax(0) - five.amin(0), five.amax(0)
    y, x = (rng_ >= (0.125 * hi).clamp(min=0.0312)).nonzero(as_tuple=True)
    L = {k: v[y, x] for k, v in L.items()}
    M, N, S, W, E, rng_ = L[0, 0], L[-1, 0], L[1, 0], L[0, -1], L[0, 1], rng_[y, x]
    sd = lambda a, m, b: (a + b - 2 * m).abs()  # noqa: E731
    eh = sd(L[-1, -1], W, L[1, -1]) + 2 * sd(N, M, S) + sd(L[-1, 1], E, L[1, 1])
    ev = sd(L[-1, -1], N, L[-1, 1]) + 2 * sd(W, M, E) + sd(L[1, -1], S, L[1, 1])
    hz = eh >= ev
    l1, l2 = torch.where(hz, N, W), torch.where(hz, S, E)
    neg = (l1 - M).abs() >= (l2 - M).abs()
    gs = 0.25 * torch.maximum((l1 - M).abs(), (l2 - M).abs())
    edge = 0.5 * (torch.where(neg, l1, l2) + M)
    sgn = torch.where(neg, -1.0, 1.0).double()
    fy, fx = y.double(), x.double()
    sx, sy = torch.where(hz, fx, fx + 0.5 * sgn), torch.where(hz, fy + 0.5 * sgn, fy)
    dist, end = [], []
    for way in (-1.0, 1.0):
        dd, e, live = torch.zeros_like(fx), torch.zeros_like(fx), torch.ones_like(hz)
        for step in (1, 1, 1, 1, 1, 1.5, 2, 2, 2, 2, 4, 8):
            dd = torch.where(live, dd + step, dd)
            q = bilinear(lum, torch.where(hz, sy, sy + way * dd), torch.where(hz, sx + way * dd, sx)) - edge
            e = torch.where(live, q, e)
            live = live & (q.abs() < gs)
        dist.append(dd)
        end.append(e)
    near = dist[0] < dist[1]
    dmin, e = torch.where(near, dist[0], dist[1]), torch.where(near, end[0], end[1])
    off = torch.where((M < edge) != (e < 0), 0.5 - dmin / (dist[0] + dist[1]), 0.0)
    avg = (2 * (N + S + W + E) + L[-1, -1] + L[-1, 1] + L[1, -1] + L[1, 1]) / 12
    sp = ((avg - M).abs() / rng_).clamp(max=1)
    sp = (3 - 2 * sp) * sp * sp
    f = torch.maximum(off, 0.75 * sp * sp) * sgn
    out = c.clone()
    out[y, x, :3] = bilinear(c, torch.where(hz, fy + f, fy), torch.where(hz, fx, fx + f))[:, :3]
    return out


def exact(case, seed):
    """What run() returns, in 64 bits: the filter, the room's frame, and the
    closest-hit records of the queries small enough to test every triangle
    (bounded by MOST_TESTS); None for the others."""
    kind = case["kind"]
    if kind == "fxaa":
        return _exact_fxaa(_picture(case["width"], case["height"], seed))
    if kind in ("serve", "sort") or (kind == "frame" and not (case["instances"] == 3 and case["tris"] <= 26)):
        return None
    st = prepare(case, seed)
    if kind == "frame":
        return _exact_room_frame(st["scene"], case["width"], case["height"]) if case["depth"] >= 1 else None
    if "rays" not in st or case["rays"] > 1 << 18:
        return None
    if kind == "build":
        got = _brute(_soup(st["meshes"], st["M"], range(case["meshes"])), st["rays"])
    else:
        s = st["scene"]
        got = _brute(_soup(s.meshes, s.M if case["update"] == "none" else s.moved, s.mesh_id), st["rays"])
    if got is None:
        return None
    out = dict(ids=None, tuv=got[0])
    if "short" in st:
        out["occluded"] = None
    return out
