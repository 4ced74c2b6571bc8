"""Scenes whose detail is small against their extent (BVH2 subtrees on grids of their own, one within another):
every path through the BVH2 gives the hits and images of the other layouts, whose boxes are local or exact."""
import numpy as np
import pytest
import torch

from paper_2310_07182_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cr():
    from paper_2310_07182_gb300 import binding
    binding.lib()
    return binding


def _nested(n_soup=2000, smallest=1e-3, levels=4):
    """Soups of triangles, each a fraction of the size of the one around it and inside it, under a light."""
    base = scenes.tiny(seed=8, n_soup=n_soup, material_mix="mixed")
    rng = np.random.default_rng(3)
    tris, mats, centre = [base.tri_xyz], [base.tri_mat], np.zeros(3)
    for size in np.geomspace(1.0, smallest, levels)[1:]:
        centre = centre + rng.uniform(-0.1, 0.1, 3) * size
        c = centre + rng.normal(size=(n_soup, 1, 3)) * size * 0.3
        tris.append((c + rng.normal(size=(n_soup, 3, 3)) * size * 0.02).reshape(-1, 9).astype(np.float32))
        mats.append(rng.integers(0, 2, n_soup).astype(np.uint32))
    wide = np.array([[-4e3, -2, -4e3, 4e3, -2, -4e3, 4e3, -2, 4e3], [-4e3, -2, -4e3, 4e3, -2, 4e3, -4e3, -2, 4e3]], np.float32)
    tri = np.concatenate(tris + [wide])
    mat = np.concatenate(mats + [np.zeros(2, np.uint32)])
    return scenes.Scene("nested", np.ascontiguousarray(tri), mat, base.mat_type, base.mat_params, base.env, base.camera), centre


def _rays(centre, n, seed, near):
    """Rays from several distances at points around the innermost soup, some along an axis."""
    rng = np.random.default_rng(seed)
    rays = np.zeros((n, 8), np.float32)
    d = rng.normal(size=(n, 3))
    far = 10.0 ** rng.uniform(np.log10(near), 2, (n, 1))
    o = centre + far * d / np.linalg.norm(d, axis=1, keepdims=True)
    rays[:, 0:3] = o
    rays[:, 4:7] = (centre + rng.normal(size=(n, 3)) * near - o) * 10.0 ** rng.uniform(-3, 3, (n, 1))
    rays[::5, 4] = 0.0
    rays[1::7, 5:7] = 0.0
    rays[2::7, 4:6] = -0.0
    rays[:, 7] = np.where(rng.random(n) < 0.3, rng.uniform(0, 2, n), np.inf)
    rays[3::11, 7] = -1.0
    return rays


@pytest.mark.parametrize("smallest,levels", [(1e-2, 2), (1e-3, 4), (1e-6, 5)])
@pytest.mark.parametrize("n_rays", [1, 40, 3000, 300007])
def test_hits_agree_with_the_other_layouts(cr, smallest, levels, n_rays):
    sc, centre = _nested(2000, smallest, levels)
    S = cr.Scene(sc, bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q | cr.CR_BVH4)
    rays = torch.from_numpy(_rays(centre, n_rays, n_rays, 3 * smallest)).cuda()
    p8, t8 = S.trace(rays, bvh=cr.CR_BVH8Q)
    p4, t4 = S.trace(rays, bvh=cr.CR_BVH4)
    assert torch.equal(p8, p4) and torch.equal(t8, t4) and (n_rays < 3000 or (p8 >= 0).float().mean() > 0.2)
    for flags in (0, cr.CR_OPT_PERSISTENT, cr.CR_OPT_COUNT, cr.CR_OPT_SPECULATIVE, cr.CR_OPT_PACKET_PRIMARY):
        p, t = S.trace(rays, flags=flags)
        assert torch.equal(p, p8) and torch.equal(t, t8)
    any_p, _ = S.trace(rays, any_hit=True)
    assert torch.equal(any_p >= 0, p8 >= 0)
    n = min(n_rays, cr.CR_TRACE_STATIC_MAX_RAYS)
    p, t = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, device="cuda")
    cr.cr_trace_rays_static(S.handle, rays[:n], None, p, t)
    assert torch.equal(p, p8[:n]) and torch.equal(t, t8[:n])


@pytest.mark.parametrize("stack", [8, 16, 32])
@pytest.mark.parametrize("mode,flags", [("direction_reuse", 0), ("direction_reuse", 8), ("independent", 128), ("independent", 16),
                                        ("direction_reuse", 32 | 64), ("morton_sort", 0)])
def test_images_agree_with_the_other_layouts(cr, stack, mode, flags):
    sc, centre = _nested()
    S = cr.Scene(sc, bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q)
    pos = tuple(float(v) for v in centre + np.array([0.001, 0.002, -0.01]))
    cam = scenes.Camera(pos, tuple(float(v) for v in centre), (0.0, 1.0, 0.0), 50.0, 300, 170)
    kw = dict(spp=2, max_bounces=3, mode=mode, tile=(8, 8), k=8, seed=2)
    want, _ = S.render(cam, bvh=cr.CR_BVH8Q, **kw)
    assert float(want.std()) > 0
    for key in (0, 5) if mode == "morton_sort" else (0,):
        got, _ = S.render(cam, stack=stack, flags=flags, sort_key=key, **kw)
        assert torch.equal(want, got)


@pytest.mark.parametrize("flags", [0, 1])
def test_batches_with_even_scenes_agree(cr, flags):
    """A batch over a scene with several grids and scenes with one, light samples among them."""
    sc, centre = _nested()
    even = scenes.interior(n_spheres=40, width=96, height=64)
    S, T = cr.Scene(sc), cr.Scene(even)
    pos = tuple(float(v) for v in centre + np.array([0.001, 0.002, -0.01]))
    cam = scenes.Camera(pos, tuple(float(v) for v in centre), (0.0, 1.0, 0.0), 50.0, 200, 120)
    kw = dict(spp=3, max_bounces=3, mode="direction_reuse", seed=2)
    want = [S.render(cam, tile=(8, 8), k=8, nee=True, **kw)[0], T.render(even.camera, tile=(8, 8), k=8, nee=True, **kw)[0]]
    outs = [torch.empty_like(w) for w in want]
    jobs = [cr.make_job(s.handle, c, o, nee=True, **kw) for s, c, o in zip((S, T), (cam, even.camera), outs)]
    b = cr.cr_batch_create(jobs, cr.make_batch_opts(tile=(8, 8), k=8, flags=flags))
    try:
        cr.cr_batch_run(b)
        assert all(torch.equal(w, o) for w, o in zip(want, outs))
    finally:
        cr.cr_batch_destroy(b)
    srv = cr.cr_server_create(256 << 20, tile=(8, 8), k=8)
    try:
        for o in outs:
            o.fill_(-1.0)
        for j in [cr.cr_server_submit(srv, j) for j in jobs]:
            cr.cr_server_wait(srv, j, 60000)
        assert all(torch.equal(w, o) for w, o in zip(want, outs))
    finally:
        cr.cr_server_destroy(srv)
