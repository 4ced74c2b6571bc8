"""The BVH2 traversal where its stack and its rays leave the ordinary range: stacks that overflow
into local memory (large triangles that all overlap, so both children are hit all the way
down), and ray origins far outside the scene's grid."""
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


def _overlapping(n, seed):
    """n triangles of random shape around the origin, each about as large as the whole scene."""
    rng = np.random.default_rng(seed)
    sc = scenes.tiny(seed=seed, n_soup=n, material_mix="mixed")
    sc.tri_xyz[:n] = rng.normal(size=(n, 9)).astype(np.float32)
    return sc


@pytest.mark.parametrize("n", [3, 40, 3000])
@pytest.mark.parametrize("stack", [8, 16, 32])
def test_full_stacks_render_the_same(cr, n, stack):
    S = cr.Scene(_overlapping(n, 4), bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q)
    kw = dict(spp=1, max_bounces=3, mode="direction_reuse", tile=(8, 8), k=8, seed=2)
    cam = scenes.Camera((0.3, 0.2, -4.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), 50.0, 75, 41)
    want, _ = S.render(cam, bvh=cr.CR_BVH8Q, **kw)
    got, _ = S.render(cam, stack=stack, **kw)
    assert torch.equal(want, got)


@pytest.mark.parametrize("far", [1.0, 30.0, 1e4])
@pytest.mark.parametrize("n_rays", [1, 33, 1999])
def test_far_origins_and_every_layout_agree(cr, far, n_rays):
    S = cr.Scene(_overlapping(500, 9), bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q | cr.CR_BVH4)
    rng = np.random.default_rng(n_rays)
    rays = scenes.random_rays(3, n_rays, target_box=(-2.0, 2.0))
    d = rng.normal(size=(n_rays, 3))
    rays[:, 0:3] = far * d / np.linalg.norm(d, axis=1, keepdims=True)
    rays[:, 4:7] = (rng.uniform(-2, 2, (n_rays, 3)) - rays[:, 0:3]) / far
    rays[::7, 4] = 0.0  # parallel to a pair of planes
    r = torch.from_numpy(rays).cuda()
    p2, t2 = S.trace(r)
    p8, t8 = S.trace(r, bvh=cr.CR_BVH8Q)
    p4, t4 = S.trace(r, bvh=cr.CR_BVH4)
    assert torch.equal(p2, p8) and torch.equal(t2, t8)
    assert torch.equal(p2, p4) and torch.equal(t2, t4)
    assert n_rays == 1 or (p2 >= 0).any()


@pytest.mark.parametrize("n_rays", [1, 31, 33, 4097, 400003])
@pytest.mark.parametrize("dead", ["none", "some", "runs", "all"])
def test_lanes_that_take_new_rays(cr, n_rays, dead):
    """Rays handed out lane by lane (more of them than lanes resident at once, chunks without any
    ray, single dead rays), read from aligned and unaligned lists, give the hits of one ray per
    lane through the BVH8-Q; so do hits that are written over the rays."""
    S = cr.Scene(scenes.tiny(seed=5, n_soup=700, material_mix="mixed"), bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q)
    rays = torch.from_numpy(scenes.random_rays(7, n_rays)).cuda()
    i = torch.arange(n_rays, device="cuda")
    off = {"none": i < 0, "some": i % 5 == 2, "runs": (i // 96) % 3 != 0, "all": i >= 0}[dead]
    rays[off, 7] = -1.0
    want_p, want_t = S.trace(rays, bvh=cr.CR_BVH8Q)
    moved = torch.empty(8 * n_rays + 1, device="cuda")[1:].view(n_rays, 8)
    moved.copy_(rays)
    for r in (rays, moved):
        for flags in (0, cr.CR_OPT_PERSISTENT):
            got_p, got_t = S.trace(r, flags=flags)
            assert torch.equal(want_p, got_p) and torch.equal(want_t, got_t)
    assert (want_p[off] == -1).all() and (n_rays < 100 or dead == "all" or (want_p >= 0).any())
    over = rays.clone().view(-1)
    cr.cr_trace_rays(S.handle, over.view(n_rays, 8), None, over[:n_rays].view(torch.int32), over[n_rays:2 * n_rays],
                     cr.make_opts())
    assert torch.equal(want_p, over[:n_rays].view(torch.int32)) and torch.equal(want_t, over[n_rays:2 * n_rays])
    assert bool(((want_p >= 0) == (S.trace(rays, any_hit=True)[0] >= 0)).all())


@pytest.mark.parametrize("copies,n_rays", [(2, 500), (9, 70), (9, 200000)])
def test_ties_between_lanes_that_share_a_ray(cr, copies, n_rays):
    """Every triangle several times over: lanes that trace parts of one ray find the same distance
    on different copies, and the smallest index wins."""
    base = _overlapping(300, 12)
    order = np.random.default_rng(copies).permutation(copies * base.n_tri)
    sc = scenes.Scene("copies", np.tile(base.tri_xyz, (copies, 1))[order], np.tile(base.tri_mat, copies)[order],
                      base.mat_type, base.mat_params, base.env, base.camera)
    S = cr.Scene(sc, bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q)
    rays = torch.from_numpy(scenes.random_rays(2, n_rays)).cuda()
    p, t = S.trace(rays)
    p8, t8 = S.trace(rays, bvh=cr.CR_BVH8Q)
    assert torch.equal(p, p8) and torch.equal(t, t8) and (p >= 0).any()


@pytest.mark.parametrize("mode", ["direction_reuse", "morton_sort"])
@pytest.mark.parametrize("size,spp", [((1, 1), 2), ((33, 17), 3), ((1500, 1100), 4)])
def test_samples_that_share_a_pass_sum_in_order(cr, mode, size, spp):
    """Samples rendered side by side in a pass (all of them, or fewer than the image has: the largest
    size) give the float sums of one sample after another, and the same ray counts."""
    S = cr.Scene(scenes.tiny(seed=6, n_soup=300, material_mix="transmissive"))
    cam = scenes.Camera((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), 60.0, *size)
    kw = dict(max_bounces=2, mode=mode, tile=(8, 8), k=8, seed=9)
    img, st = S.render(cam, spp=spp, stats=True, **kw)
    total, rays = torch.zeros_like(img), 0
    for s in range(spp):
        one, st1 = S.render(cam, spp=1, frame_base=s, stats=True, **kw)
        total += one
        rays += st1["secondary_rays"]
    assert torch.equal(img, total * torch.tensor(1.0 / spp, dtype=torch.float32, device="cuda"))
    assert st["secondary_rays"] == rays


@pytest.mark.parametrize("spp", [1, 11, 22, 23, 24, 25, 40])
def test_small_and_large_job_tables(cr, spp):
    """A render's job table (an entry per sample side by side, one more for the sums) comes from launch
    arguments where it is small and is copied where it is not; a batch of the same job copies it."""
    S = cr.Scene(scenes.tiny(seed=6, n_soup=300, material_mix="mixed"))
    cam = scenes.Camera((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), 60.0, 40, 24)
    kw = dict(spp=spp, max_bounces=3, mode="direction_reuse", seed=9)
    img, _ = S.render(cam, tile=(8, 8), **kw)
    out = torch.full_like(img, -1.0)
    b = cr.cr_batch_create([cr.make_job(S.handle, cam, out, **kw)], cr.make_batch_opts(tile=(8, 8)))
    try:
        cr.cr_batch_run(b)
        assert torch.equal(img, out)
    finally:
        cr.cr_batch_destroy(b)


@pytest.mark.parametrize("bvh", ["CR_BVH2", "CR_BVH8Q"])
@pytest.mark.parametrize("k,size,spp", [(8, (8, 8), 1), (8, (200, 120), 3), (64, (200, 120), 2)])
def test_chained_launches_and_a_graph_agree(cr, bvh, k, size, spp):
    """Launches set up while the one before ends (render, direct batch; many calls back to back) and the
    ordinary ones of a captured graph give the same image."""
    S = cr.Scene(scenes.tiny(seed=6, n_soup=300, material_mix="mixed"), bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q)
    cam = scenes.Camera((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), 60.0, *size)
    kw = dict(spp=spp, max_bounces=4, mode="direction_reuse", seed=9)
    out = torch.empty((size[1], size[0], 3), device="cuda")
    jobs = [cr.make_job(S.handle, cam, out, **kw)]
    images = []
    for flags in (cr.CR_BATCH_GRAPH, 0):
        b = cr.cr_batch_create(jobs, cr.make_batch_opts(tile=(8, 8), k=k, bvh=getattr(cr, bvh), flags=flags))
        try:
            for _ in range(3):
                out.fill_(-1.0)
                cr.cr_batch_run(b)
                images.append(out.clone())
        finally:
            cr.cr_batch_destroy(b)
    for _ in range(20):
        images.append(S.render(cam, tile=(8, 8), k=k, bvh=getattr(cr, bvh), **kw)[0])
    assert all(torch.equal(images[0], i) for i in images[1:])


@pytest.mark.parametrize("bvh", ["CR_BVH2", "CR_BVH8Q"])
@pytest.mark.parametrize("size,spp", [((8, 8), 1), ((200, 120), 3), ((1500, 1000), 2)])
def test_light_samples_beside_the_next_trace(cr, bvh, size, spp):
    """The trace that runs beside the light samples' (below and above its size rule, one and two scenes, captured
    and not) gives the images of the launches one after the other (a counting pass)."""
    S = cr.Scene(scenes.interior(n_spheres=60, width=96, height=64), bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q)
    T = cr.Scene(scenes.tiny(seed=6, n_soup=300, material_mix="mixed"), bvh_flags=cr.CR_BVH2 | cr.CR_BVH8Q)
    c = scenes.interior(n_spheres=60, width=96, height=64).camera
    cam = scenes.Camera(c.pos, c.look_at, c.up, c.vfov_deg, *size)
    b = getattr(cr, bvh)
    kw = dict(spp=spp, max_bounces=3, mode="direction_reuse", seed=9, nee=True)
    want = S.render(cam, tile=(8, 8), k=8, bvh=b, flags=cr.CR_OPT_COUNT, stats=True, **kw)[0]
    for _ in range(5):
        assert torch.equal(want, S.render(cam, tile=(8, 8), k=8, bvh=b, **kw)[0])
    out, other = torch.empty_like(want), torch.empty_like(want)
    jobs = [cr.make_job(S.handle, cam, out, **kw), cr.make_job(T.handle, cam, other, **kw)]
    for n in (1, 2):
        for flags in (0, cr.CR_BATCH_GRAPH):
            h = cr.cr_batch_create(jobs[:n], cr.make_batch_opts(tile=(8, 8), k=8, bvh=b, flags=flags))
            try:
                for _ in range(3):
                    out.fill_(-1.0)
                    cr.cr_batch_run(h)
                    assert torch.equal(want, out)
            finally:
                cr.cr_batch_destroy(h)
