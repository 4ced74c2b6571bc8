"""Triangles that are large against where rays start: a ray that leaves a surface for the side it is on meets
neither that surface's triangle nor the coplanar one beside it, whatever rounding makes of the distance, in
every layout (their boxes are enlarged by different amounts)."""
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


def _scene(half, fine):
    """A soup of the size 1 over a ground of two triangles; `fine`: small enough for a grid of its own."""
    base = scenes.tiny(seed=8, n_soup=3000 if fine else 300, material_mix="mixed")
    soup = base.tri_xyz[:-2] * np.float32(0.5)
    y, h = -1.0, half
    ground = np.array([[-h, y, -h, h, y, -h, h, y, h], [-h, y, -h, h, y, h, -h, y, h]], np.float32)
    tri = np.concatenate([soup, ground])
    mat = np.concatenate([base.tri_mat[:-2], np.zeros(2, np.uint32)])
    return scenes.Scene("wide", np.ascontiguousarray(tri), mat, base.mat_type, base.mat_params, base.env, base.camera)


@pytest.mark.parametrize("half", [100.0, 1000.0, 1e5, 3e6])
@pytest.mark.parametrize("fine", [False, True])
def test_rays_that_leave_the_ground_do_not_meet_it(cr, half, fine):
    sc = _scene(half, fine)
    S = cr.Scene(sc, bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q | cr.CR_BVH4)
    rng = np.random.default_rng(1)
    n = 400000
    rays = np.zeros((n, 8), np.float32)
    x = rng.uniform(-3, 3, n)
    rays[:, 0] = x
    rays[:, 1] = np.float32(-1.0) + np.float32(2.0 ** -18) * rng.integers(1, 4, n)
    rays[:, 2] = x + rng.uniform(-1, 1, n) * 10.0 ** rng.uniform(-6, 0, n)  # near the edge that the two share
    d = rng.normal(size=(n, 3))
    d[:, 1] = np.abs(d[:, 1]) + 1e-3
    rays[:, 4:7] = d / np.linalg.norm(d, axis=1, keepdims=True)
    rays[:, 7] = np.inf
    ground = torch.tensor([sc.n_tri - 2, sc.n_tri - 1], device="cuda")
    skip = torch.from_numpy((sc.n_tri - 2 + (rays[:, 0] < rays[:, 2])).astype(np.int32)).cuda()
    r = torch.from_numpy(rays).cuda()
    first = None
    for bvh in (cr.CR_BVH2, cr.CR_BVH8Q, cr.CR_BVH4):
        for s in (None, skip):
            p, t = S.trace(r, s, bvh=bvh)
            assert not torch.isin(p, ground).any()
            if s is None:
                first = (p, t) if first is None else first
                assert torch.equal(p, first[0]) and torch.equal(t, first[1])
        if bvh != cr.CR_BVH4:
            assert torch.equal(S.trace(r, bvh=bvh, any_hit=True)[0] >= 0, first[0] >= 0)
    m = cr.CR_TRACE_STATIC_MAX_RAYS
    p, t = torch.empty(m, dtype=torch.int32, device="cuda"), torch.empty(m, device="cuda")
    cr.cr_trace_rays_static(S.handle, r[:m], None, p, t)
    assert torch.equal(p, first[0][:m]) and torch.equal(t, first[1][:m])


@pytest.mark.parametrize("half", [300.0, 3e4])
@pytest.mark.parametrize("fine", [False, True])
@pytest.mark.parametrize("nee", [False, True])
def test_images_of_wide_scenes_agree(cr, half, fine, nee):
    sc = _scene(half, fine)
    S = cr.Scene(sc, bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q | cr.CR_BVH4)
    cam = scenes.Camera((0.0, 1.0, 3.0), (0.0, -0.5, 0.0), (0.0, 1.0, 0.0), 60.0, 640, 360)
    kw = dict(spp=2, max_bounces=4, tile=(8, 8), k=8, seed=3, nee=nee)
    want, _ = S.render(cam, bvh=cr.CR_BVH4, **kw)
    for bvh in (cr.CR_BVH2, cr.CR_BVH8Q):
        got, _ = S.render(cam, bvh=bvh, **kw)
        assert torch.equal(want, got)
