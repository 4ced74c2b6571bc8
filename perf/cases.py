"""The work this package does for its users, as cases that can be timed.

Four entry points carry it: closest-hit queries on a resident scene (``Scene.trace`` and the
allocation-free ``cr_trace_rays_static``), single renders (``Scene.render``), batches of
render jobs (``cr_batch_*``) and the server (``cr_server_*``).  ``listed()`` names twelve
points of their ranges, ``draw()`` gives others, ``prepare()`` builds what a program holds
before the call (a resident scene, rays or a camera, output buffers, a batch or a server),
and ``run()`` makes the call.

Scene geometry is fixed per size, like an asset that a program loads (kept as host arrays
between preparations); the seed moves the camera, draws the rays and keys the random numbers.

Any-hit queries are timed as the shadow rays of next-event estimation: the occluder that
``CR_OPT_ANY_HIT`` returns to a caller is any one in front of tmax, so its index is no result
to hold a kernel to.
"""
import functools
import math

import numpy as np
import torch

from paper_2310_07182_gb300 import binding as cr
from paper_2310_07182_gb300 import scenes

BVH = {"bvh2": cr.CR_BVH2, "bvh8q": cr.CR_BVH8Q, "bvh4": cr.CR_BVH4}


def listed():
    return [
        # -- closest-hit queries of a caller's rays --------------------------------------
        # a picking / probing query of a few rays on a small scene: the call's latency
        dict(name="trace_1k", op="trace", scene="tiny", size=1024, rays="random", n=1000, bvh="bvh2"),
        # an odd number of coherent camera rays of a viewport on the terrain, no skip ids
        dict(name="trace_camera", op="trace", scene="landscape", size=512, rays="camera", n=300007, bvh="bvh2"),
        # light baking over a dense room: a million incoherent surface rays with skip ids
        dict(name="trace_surface_1m", op="trace", scene="interior", size=2000, rays="surface", n=1000003, bvh="bvh2"),
        # the same kind of query from a loop that must not allocate, at that call's limit
        dict(name="trace_static_64k", op="static", scene="interior", size=200, rays="surface", n=65536, bvh="bvh2"),
        # -- single renders ---------------------------------------------------------------
        # a thumbnail or a test: 64 x 64, one sample, one bounce, 4x4 tiles: launches count
        dict(name="render_tiny", op="render", scene="tiny", size=1024, width=64, height=64, spp=1, bounces=1,
             mode="direction_reuse", tile=4, k=16, nee=False, hybrid_donor=False, bvh="bvh2"),
        # the interactive frame of the headline benchmark: full HD terrain, 1 spp, 2 bounces
        dict(name="render_landscape", op="render", scene="landscape", size=1024, width=1920, height=1080, spp=1,
             bounces=2, mode="direction_reuse", tile=8, k=8, nee=False, hybrid_donor=False, bvh="bvh2"),
        # the same frame by the sorting comparator (key, radix sort, trace)
        dict(name="render_landscape_sort", op="render", scene="landscape", size=1024, width=1920, height=1080, spp=1,
             bounces=2, mode="morton_sort", tile=8, k=8, nee=False, hybrid_donor=False, bvh="bvh2"),
        # a final-quality interior with light samples: 16 spp, 4 bounces, shadow rays
        dict(name="render_interior_nee", op="render", scene="interior", size=2000, width=1280, height=720, spp=16,
             bounces=4, mode="direction_reuse", tile=8, k=8, nee=True, hybrid_donor=True, bvh="bvh2"),
        # the precision variant's layout at a ragged size
        dict(name="render_bvh8q", op="render", scene="interior", size=2000, width=853, height=479, spp=4, bounces=4,
             mode="direction_reuse", tile=8, k=8, nee=False, hybrid_donor=False, bvh="bvh8q"),
        # glass and translucent materials, groups larger than a warp, ragged tiles
        dict(name="render_glass_k64", op="render", scene="glass", size=4096, width=500, height=333, spp=4, bounces=8,
             mode="direction_reuse", tile=16, k=64, nee=False, hybrid_donor=False, bvh="bvh2"),
        # -- many jobs ----------------------------------------------------------------------
        # a planned batch replayed from its graph: mixed sizes over several scenes
        dict(name="batch_16", op="batch", jobs=16, spp=4, bounces=3, side=512, size=256, tile=8, k=8, bvh="bvh2"),
        # requests of mixed size given to a running server at once, until the last is done
        dict(name="serve_24", op="serve", jobs=24, spp=4, bounces=3, side=320, size=256, tile=8, k=8, bvh="bvh2"),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def scene():
        s = rng.choice(["tiny", "landscape", "interior", "glass"])
        return s, {"tiny": lambda: log(256, 16384), "landscape": lambda: log(64, 768),
                   "interior": lambda: log(50, 2000), "glass": lambda: log(256, 16384)}[s]()

    op = rng.choice(["trace", "trace", "static", "render", "render", "render", "batch", "serve"])
    if op in ("trace", "static"):
        s, size = scene()
        return dict(op=op, scene=s, size=size, rays=rng.choice(["random", "camera", "surface"]),
                    n=log(500, 1000000) if op == "trace" else log(500, 65536),
                    bvh=rng.choice(["bvh2", "bvh2", "bvh8q", "bvh4"]) if op == "trace" else "bvh2")
    if op == "render":
        s, size = scene()
        tile, k = rng.choice([(4, 4), (4, 16), (8, 4), (8, 8), (8, 64), (16, 8), (16, 32), (16, 256)])
        mode = rng.choice(["direction_reuse", "direction_reuse", "independent", "morton_sort", "world_reuse"])
        w = log(48, 1600)
        h = max(32, int(w * rng.uniform(0.5, 1.1)))
        spp = rng.choice([1, 1, 2, 4, 8])
        while w * h * spp > 3000000:
            spp = max(1, spp // 2)
            w, h = (w, h) if w * h * spp <= 3000000 else (int(w * 0.8), int(h * 0.8))
        return dict(op="render", scene=s, size=size, width=w, height=h, spp=spp, bounces=rng.randint(1, 5), mode=mode,
                    tile=tile, k=k, nee=s == "interior" and rng.random() < 0.5, hybrid_donor=rng.random() < 0.3,
                    bvh=rng.choice(["bvh2", "bvh2", "bvh2", "bvh8q", "bvh4"]))
    return dict(op=op, jobs=rng.randint(4, 24), spp=rng.choice([1, 2, 4]), bounces=rng.randint(1, 4),
                side=log(96, 512), size=rng.randint(96, 256), tile=8, k=rng.choice([4, 8, 16]),
                bvh=rng.choice(["bvh2", "bvh8q"]))


# ---------------------------------------------------------------------------------------
# Scenes
@functools.lru_cache(maxsize=24)
def _scene(kind, size):
    """The host arrays of an asset: `size` soup triangles, vertices along a side of the terrain's
    grid, or spheres of the room."""
    if kind == "tiny":
        return scenes.tiny(seed=1, n_soup=size, material_mix="mixed")
    if kind == "glass":
        return scenes.tiny(seed=2, n_soup=size, material_mix="transmissive")
    if kind == "landscape":
        return scenes.landscape(seed=7, n_grid=size)
    return _interior(size)


def _interior(n_spheres, seed=11):
    """scenes.interior's room for a number of spheres, put together without a loop over triangles."""
    base = scenes.interior(seed=seed, n_spheres=1)
    rng = np.random.default_rng(seed)
    unit = scenes.uv_sphere((0.0, 0.0, 0.0), 1.0).reshape(-1, 3)
    r = rng.uniform(0.05, 0.3, n_spheres)
    c = np.stack([rng.uniform(-4 + r, 4 - r), rng.uniform(r, 4 - r), rng.uniform(-4 + r, 4 - r)], axis=1)
    near = np.linalg.norm(c - np.array([0.0, 2.0, -3.8]), axis=1) < r + 0.6  # clear of the camera
    c[near, 2] = 4 - r[near]
    sph = (c[:, None, :] + r[:, None, None] * unit[None]).reshape(-1, 9)
    n_wall, per = 12, unit.shape[0] // 3
    cls = rng.choice([scenes.MAT_LAMBERT, scenes.MAT_GGX, scenes.MAT_MIRROR], size=n_spheres, p=[0.6, 0.3, 0.1])
    pal = {t: np.flatnonzero(base.mat_type == t) for t in (scenes.MAT_LAMBERT, scenes.MAT_GGX, scenes.MAT_MIRROR)}
    mat = np.array([rng.choice(pal[int(t)]) for t in cls])
    tris = np.concatenate([base.tri_xyz[:n_wall], sph.astype(np.float32), base.tri_xyz[-2:]])
    tri_mat = np.concatenate([base.tri_mat[:n_wall], np.repeat(mat, per).astype(np.uint32), base.tri_mat[-2:]])
    return scenes.Scene("room%d" % n_spheres, np.ascontiguousarray(tris), tri_mat.astype(np.uint32), base.mat_type,
                        base.mat_params, base.env, base.camera)


def _camera(sc, seed, width, height):
    """The asset's camera, moved a little by the seed."""
    c = sc.camera
    step = 0.01 * float(np.linalg.norm(np.array(c.pos) - np.array(c.look_at)))
    d = np.random.default_rng(seed).uniform(-step, step, 3)
    return scenes.Camera(tuple(float(v) for v in np.array(c.pos) + d), c.look_at, c.up, c.vfov_deg, width, height)


def _unit(v):
    return v / v.norm(dim=1, keepdim=True)


def _rays(sc, kind, n, seed):
    """(n, 8) rays on the GPU and the skip ids (or None)."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    out = torch.zeros((n, 8), dtype=torch.float32, device="cuda")
    out[:, 7] = math.inf
    tri = torch.from_numpy(sc.tri_xyz).cuda().double().reshape(-1, 3, 3)
    lo, hi = tri.amin(dim=(0, 1)), tri.amax(dim=(0, 1))
    if kind == "camera":  # one jittered ray for each pixel of an image of about n pixels, row by row
        cam = _camera(sc, seed, 16, 9)
        w = max(1, int(math.sqrt(n * 16.0 / 9.0)))
        i = torch.arange(n, device="cuda")
        h = (n + w - 1) // w
        f = torch.tensor(np.array(cam.look_at) - np.array(cam.pos), device="cuda", dtype=torch.float64)
        f = f / f.norm()
        r = torch.linalg.cross(f, torch.tensor(cam.up, device="cuda", dtype=torch.float64))
        r = r / r.norm()
        u = torch.linalg.cross(r, f)
        t = math.tan(math.radians(cam.vfov_deg) / 2)
        x = ((i % w) + rand(n)) / w * 2 - 1
        y = 1 - ((i // w) + rand(n)) / h * 2
        d = _unit(f + x[:, None] * (t * w / h) * r + y[:, None] * t * u)
        out[:, 0:3] = torch.tensor(cam.pos, device="cuda", dtype=torch.float32)
        out[:, 4:7] = d.float()
        return out, None
    if kind == "surface":  # cosine-distributed directions from random points of random triangles
        pick = torch.randint(tri.shape[0], (n,), generator=g, device="cuda")
        v = tri[pick]
        s, b = rand(n).sqrt(), rand(n)
        p = (1 - s)[:, None] * v[:, 0] + (s * (1 - b))[:, None] * v[:, 1] + (s * b)[:, None] * v[:, 2]
        nrm = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
        nrm = nrm / nrm.norm(dim=1, keepdim=True).clamp_min(1e-30)
        nrm = torch.where(nrm[:, 1:2] < 0, -nrm, nrm) if sc.name.startswith("landscape") else nrm
        d = _unit(nrm + _unit(torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)) * 0.999)
        out[:, 0:3] = (p + nrm * 1e-5 * p.abs().amax(dim=1, keepdim=True).clamp_min(1.0)).float()
        out[:, 4:7] = d.float()
        return out, pick.to(torch.int32)
    out[:, 0:3] = (lo + rand(n, 3) * (hi - lo)).float()
    out[:, 4:7] = _unit(torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)).float()
    return out, None


class _Handle:
    """A batch or server handle and the scenes it reads, given back in that order."""

    def __init__(self, handle, destroy, keep):
        self.handle, self.destroy, self.keep = handle, destroy, keep

    def __del__(self):
        self.destroy(self.handle)
        for s in self.keep:
            s.close()


# ---------------------------------------------------------------------------------------
def _jobs(case, seed):
    """Scenes and jobs of a batch or of the server's requests: sizes from a quarter of the side to
    the side, odd ones among them, over four assets."""
    rng = np.random.default_rng(seed)
    flags = cr.CR_BVH2 | BVH[case["bvh"]]
    src = [_scene("landscape", case["size"]), _scene("interior", case["size"]), _scene("tiny", 64 * case["size"]),
           _scene("glass", 16 * case["size"])]
    held = [cr.Scene(s, bvh_flags=flags) for s in src]
    shape = np.random.default_rng(case["jobs"])  # the sizes belong to the case, not to the seed
    jobs, outs = [], []
    for i in range(case["jobs"]):
        k = i % len(held)
        w, h = (int(v) for v in shape.integers(max(16, case["side"] // 4), case["side"] + 1, 2))
        out = torch.empty((h, w, 3), dtype=torch.float32, device="cuda")
        mode = ("direction_reuse", "direction_reuse", "independent", "direction_reuse")[i % 4]
        jobs.append(cr.make_job(held[k].handle, _camera(src[k], seed + i, w, h), out, spp=case["spp"],
                                max_bounces=case["bounces"], mode=mode, seed=int(rng.integers(1 << 31)),
                                nee=src[k].env.max() == 0))
        outs.append(out)
    return held, jobs, outs


def prepare(case, seed):
    op = case["op"]
    if op in ("trace", "static"):
        sc = _scene(case["scene"], case["size"])
        S = cr.Scene(sc, bvh_flags=cr.CR_BVH2 | BVH[case["bvh"]])
        rays, skip = _rays(sc, case["rays"], case["n"], seed)
        st = dict(op=op, scene=S, rays=rays, skip=skip, bvh=BVH[case["bvh"]])
        if op == "static":
            st["prim"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
            st["t"] = torch.empty(case["n"], dtype=torch.float32, device="cuda")
        return st
    if op == "render":
        sc = _scene(case["scene"], case["size"])
        S = cr.Scene(sc, bvh_flags=cr.CR_BVH2 | BVH[case["bvh"]])
        kw = dict(spp=case["spp"], max_bounces=case["bounces"], mode=case["mode"], tile=(case["tile"], case["tile"]),
                  k=case["k"], seed=int(seed), nee=case["nee"], hybrid_donor=case["hybrid_donor"],
                  bvh=BVH[case["bvh"]])
        return dict(op=op, scene=S, cam=_camera(sc, seed, case["width"], case["height"]), kw=kw)
    held, jobs, outs = _jobs(case, seed)
    tile = (case["tile"], case["tile"])
    if op == "batch":
        b = cr.cr_batch_create(jobs, cr.make_batch_opts(tile=tile, k=case["k"], bvh=BVH[case["bvh"]],
                                                        flags=cr.CR_BATCH_GRAPH))
        return dict(op=op, batch=_Handle(b, cr.cr_batch_destroy, held), outs=outs)
    s = cr.cr_server_create(1 << 30, tile=tile, k=case["k"], bvh=BVH[case["bvh"]], express_rays=1 << 18)
    return dict(op=op, server=_Handle(s, cr.cr_server_destroy, held), jobs=jobs, outs=outs)


def run(state):
    op = state["op"]
    if op == "trace":
        return state["scene"].trace(state["rays"], state["skip"], bvh=state["bvh"])
    if op == "static":
        cr.cr_trace_rays_static(state["scene"].handle, state["rays"], state["skip"], state["prim"], state["t"])
        return state["prim"], state["t"]
    if op == "render":
        return state["scene"].render(state["cam"], **state["kw"])[0]
    if op == "batch":
        cr.cr_batch_run(state["batch"].handle, stats=False)
        return state["outs"]
    server = state["server"].handle
    for jid in [cr.cr_server_submit(server, j) for j in state["jobs"]]:
        cr.cr_server_wait(server, jid)
    return state["outs"]


# ---------------------------------------------------------------------------------------
# A ray cannot do with less than one path down a balanced binary tree (two boxes of 24
# operations at each level, a 64-byte node read) and one triangle test (40 operations, 48
# bytes); its own record is 32 bytes in and 8 bytes out (4 more with a skip id).  Nodes and
# triangles are shared between rays, so they count once, up to the whole scene.
def _n_tri(case):
    n = case["size"]
    return {"tiny": n + 2, "glass": n + 2, "landscape": 2 * (n - 1) ** 2, "interior": 256 * n + 14}[case["scene"]]


def work(case):
    op = case["op"]
    if op in ("trace", "static"):
        n, tri = case["n"], _n_tri(case)
        return {"bytes": n * (40 + (4 if case["rays"] == "surface" else 0)) + min(tri, n) * 112,
                "flops": n * (48 * math.log2(tri) + 40)}
    if op == "render":
        n, tri, spp, b = case["width"] * case["height"], _n_tri(case), case["spp"], case["bounces"]
        # each path is traced and shaded at most bounces + 1 times; half of them is taken as typical
        rays = n * spp * (1 + b / 2) * (1.5 if case["nee"] else 1)
        return {"bytes": 12 * n + min(tri, rays) * 112, "flops": rays * (48 * math.log2(tri) + 40 + 150)}
    s = case["size"]
    px = case["jobs"] * (0.625 * case["side"]) ** 2
    rays, tri = px * case["spp"] * (1 + case["bounces"] / 2), 2 * s * s + 336 * s
    return {"bytes": 12 * px + tri * 112, "flops": rays * (48 * math.log2(tri / 4) + 40 + 150)}


def exact(case, seed):
    """Closest-hit distances by brute force over all triangles in 64 bits, where that is cheap
    enough.  The hit triangle is a whole number and has no such value.  Images have none: every
    sample is a discrete path whose choices (the hit triangle, the material's lobe, the group's
    donor) follow from the 32-bit arithmetic that defines them, so 64 bits would give the mean of
    other paths."""
    if case["op"] not in ("trace", "static") or case["n"] * _n_tri(case) > 4e9:
        return None
    sc = _scene(case["scene"], case["size"])
    rays, skip = _rays(sc, case["rays"], case["n"], seed)
    tri = torch.from_numpy(sc.tri_xyz).cuda().double().reshape(-1, 3, 3)
    a, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    ids = torch.arange(tri.shape[0], device="cuda")
    best = []
    step = max(1, int(2e7) // tri.shape[0])
    for i in range(0, case["n"], step):
        o, d = rays[i:i + step, None, 0:3].double(), rays[i:i + step, None, 4:7].double()
        p = torch.linalg.cross(d.expand(-1, len(a), -1), e2.expand(d.shape[0], -1, -1))
        det = (e1 * p).sum(-1)
        s = o - a
        u = (s * p).sum(-1) / det
        q = torch.linalg.cross(s, e1.expand(s.shape[0], -1, -1))
        v = (d * q).sum(-1) / det
        t = (e2 * q).sum(-1) / det
        ok = (det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0)
        if skip is not None:
            ok &= ids != skip[i:i + step, None]
        best.append(torch.where(ok, t, math.inf).amin(dim=1))
    return None, torch.cat(best)
