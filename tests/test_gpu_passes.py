"""Samples that share passes where they do not all fit one: sums that go on from pass to pass, and jobs of a batch
that are done in an earlier pass than others."""
import pytest
import torch

from paper_2310_07182_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cr():
    from paper_2310_07182_gb300 import binding
    binding.lib()
    return binding


def _cam(w, h):
    return scenes.Camera((0.0, 0.0, -3.0), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), 60.0, w, h)


def _in_order(S, cam, spp, **kw):
    """The mean of single samples added one after another."""
    total = torch.zeros((cam.height, cam.width, 3), device="cuda")
    for s in range(spp):
        total += S.render(cam, spp=1, frame_base=s, **kw)[0]
    return total * torch.tensor(1.0 / spp, dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("spp", [6, 10, 11])
def test_sums_over_several_passes(cr, spp):
    """1500 x 1100 pixels are 1,660,416 slots in 8x8 tiles: five samples of 2^23 slots share a pass."""
    S = cr.Scene(scenes.tiny(seed=6, n_soup=300, material_mix="transmissive"))
    cam = _cam(1500, 1100)
    kw = dict(max_bounces=2, tile=(8, 8), k=8, seed=9)
    img, st = S.render(cam, spp=spp, stats=True, **kw)
    one_pass = S.render(cam, spp=5, stats=True, **kw)[1]["kernel_launches"] - 1  # the job table's launch comes once
    assert st["kernel_launches"] - 1 == -(-spp // 5) * one_pass
    assert torch.equal(img, _in_order(S, cam, spp, **kw))


@pytest.mark.parametrize("flags", [0, 1])
def test_batches_whose_jobs_end_in_different_passes(cr, flags):
    """Three jobs of about 2^20 slots: two samples of each share a pass; of 1, 3, 7 and 2 samples."""
    S = cr.Scene(scenes.tiny(seed=6, n_soup=300, material_mix="mixed"))
    T = cr.Scene(scenes.tiny(seed=7, n_soup=500, material_mix="transmissive"))
    specs = [(S, 1024, 1000, 1), (T, 1000, 1024, 3), (S, 960, 1023, 7), (T, 33, 17, 2)]
    kw = dict(max_bounces=2, seed=4)
    want = [_in_order(s, _cam(w, h), n, tile=(8, 8), k=8, **kw) for s, w, h, n in specs]
    outs = [torch.full_like(w, -1.0) for w in want]
    jobs = [cr.make_job(s.handle, _cam(w, h), o, spp=n, **kw) for (s, w, h, n), o in zip(specs, outs)]
    b = cr.cr_batch_create(jobs, cr.make_batch_opts(tile=(8, 8), k=8, flags=flags))
    try:
        for _ in range(2):
            for o in outs:
                o.fill_(-1.0)
            cr.cr_batch_run(b)
            assert all(torch.equal(w, o) for w, o in zip(want, outs))
    finally:
        cr.cr_batch_destroy(b)
