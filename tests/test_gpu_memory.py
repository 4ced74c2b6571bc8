"""Device memory of renders of several samples: bounded over all scenes and batches, and when little is free fewer
samples share a pass; the images stay."""
import pytest
import torch

from paper_2310_07182_gb300 import scenes

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def cr():
    from paper_2310_07182_gb300 import binding
    binding.lib()
    return binding


@pytest.fixture
def leave():
    """leave(n): take device memory until n bytes are free."""
    held = []

    def take(n):
        torch.cuda.synchronize()
        held.append(torch.empty(max(0, torch.cuda.mem_get_info()[0] - n), dtype=torch.uint8, device="cuda"))
    yield take
    held.clear()
    torch.cuda.empty_cache()


def _cam(w, h):
    return scenes.Camera((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), 60.0, w, h)


def _scene(cr):
    return cr.Scene(scenes.tiny(seed=6, n_soup=300, material_mix="mixed"))


# 16 samples of 640 x 360 in a pass: 524 MB of path state, 177 more with light samples, 490 more for the two
# phases.  At 900 MB the first fit and the last do not, at 300 MB none does; a sample per pass takes 33.
@pytest.mark.parametrize("free", [900 * MB, 300 * MB])
@pytest.mark.parametrize("flags,nee", [(0, False), (0, True), (128, False), (128, True)])
def test_renders_when_memory_is_short(cr, leave, free, flags, nee):
    kw = dict(spp=16, max_bounces=2, tile=(8, 8), k=8, seed=9, flags=flags, nee=nee)
    S = _scene(cr)
    want, _ = S.render(_cam(640, 360), **kw)
    S.close()
    S = _scene(cr)
    out = torch.empty_like(want)
    leave(free)
    S.render(_cam(640, 360), out=out, **kw)
    assert torch.equal(want, out)
    out.fill_(-1.0)
    S.render(_cam(640, 360), out=out, **kw)  # in the workspace that was found
    assert torch.equal(want, out)
    S.close()


@pytest.mark.parametrize("free", [900 * MB, 300 * MB])
def test_batches_when_memory_is_short(cr, leave, free):
    S = _scene(cr)
    kw = dict(max_bounces=2, seed=9)
    sizes = [(640, 360, 16), (320, 200, 5), (64, 64, 1)]
    want = [S.render(_cam(w, h), spp=n, tile=(8, 8), k=8, **kw)[0] for w, h, n in sizes]
    S.close()
    S = _scene(cr)
    outs = [torch.empty_like(w) for w in want]
    jobs = [cr.make_job(S.handle, _cam(w, h), o, spp=n, **kw) for (w, h, n), o in zip(sizes, outs)]
    leave(free)
    for flags in (0, cr.CR_BATCH_GRAPH):
        b = cr.cr_batch_create(jobs, cr.make_batch_opts(tile=(8, 8), k=8, flags=flags))
        try:
            cr.cr_batch_run(b)
            assert all(torch.equal(w, o) for w, o in zip(want, outs))
        finally:
            cr.cr_batch_destroy(b)
    S.close()


def _held(f):
    """Device bytes that f() leaves allocated."""
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    f()
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0]


def test_scenes_that_have_rendered_hold_a_bounded_share(cr):
    """64 samples of 640 x 360 take 1.2 GB in passes of 36: not of every scene that has rendered once."""
    kw = dict(spp=64, max_bounces=1, tile=(8, 8), k=8, seed=9)
    out = torch.empty((360, 640, 3), device="cuda")
    S = _scene(cr)
    first = _held(lambda: S.render(_cam(640, 360), out=out, **kw))
    assert first > 600 * MB
    want = out.clone()
    many = [_scene(cr) for _ in range(40)]
    held = _held(lambda: [s.render(_cam(640, 360), out=out, **kw) for s in many])
    total = torch.cuda.mem_get_info()[1]
    assert first + held < total // 16 + 41 * 64 * MB  # a sample per pass takes 33 MB
    assert torch.equal(out, want)
    for s in many + [S]:
        s.close()
    S = _scene(cr)  # what they held has been given back
    assert _held(lambda: S.render(_cam(640, 360), out=out, **kw)) > 600 * MB
    S.close()


def test_renders_leave_most_of_the_free_memory(cr, leave):
    kw = dict(spp=64, max_bounces=1, tile=(8, 8), k=8, seed=9)
    out = torch.empty((360, 640, 3), device="cuda")
    S = _scene(cr)
    S.render(_cam(640, 360), out=out, **kw)
    want = out.clone()
    S.close()
    S = _scene(cr)
    leave(3000 * MB)
    launches = []
    for _ in range(3):
        held = _held(lambda: launches.append(S.render(_cam(640, 360), out=out, stats=True, **kw)[1]["kernel_launches"]))
        assert held < 3000 * MB // 8 + 64 * MB and torch.equal(out, want)
    assert held == 0 and launches[0] == launches[1] == launches[2]  # the workspace that was found is kept
    S.close()


def test_device_bytes_are_what_a_batch_needs(cr, leave):
    S = _scene(cr)
    out = torch.empty((360, 640, 3), device="cuda")
    opts = cr.make_batch_opts(tile=(8, 8), k=8)
    def job(n):
        return [cr.make_job(S.handle, _cam(640, 360), out, spp=n, max_bounces=1)]
    one, many = (cr.cr_batch_device_bytes(job(n), opts) for n in (1, 64))
    assert one <= many < one + 64 * 1024  # the tables of 64 passes
    leave(many + 64 * MB)
    b = cr.cr_batch_create(job(64), opts)
    cr.cr_batch_run(b)
    cr.cr_batch_destroy(b)
    S.close()
