"""The one-launch plan of small batches (plan_and_records) against the counting
sort that larger ones take: the same bits for every galaxy, at counts around a
warp, a CTA and the line between the two, with mixed sides and PSFs and with
galaxies that are rejected; forward, adjoint and composite."""

import numpy as np
import pytest

from workloads import composite_galaxies, mixed_galaxies

pytestmark = pytest.mark.gpu

LINE = 2048   # galaxies of the largest small plan


def _status(r, fails):
    from paper_2012_15797_gb300 import capi
    if fails:
        with pytest.raises(capi.MogError):
            r.sync_status()
    else:
        r.sync_status()


@pytest.mark.parametrize("count", [1, 2, 7, 8, 9, 33, 255, 257, 1023, LINE])
def test_same_bits_as_the_counting_sort(gpu_renderer, count):
    import torch
    from paper_2012_15797_gb300.renderer import to_device
    r = gpu_renderer
    # a batch above the line whose first `count` galaxies are the small batch
    gals = mixed_galaxies(LINE + 300, seed=700 + count, n_psf=5)
    gals.size = np.minimum(gals.size, 128).astype(np.int32)
    if count > 8:   # an unknown side, an unknown PSF, a parameter that is not finite
        gals.size[3] = 48
        gals.psf[5] = 5000
        gals.flux[7] = np.nan
    big, small = to_device(gals), to_device(gals.subset(np.arange(count)))
    a = torch.full((big.total,), 3.0, device="cuda")
    b = torch.full((small.total,), 3.0, device="cuda")
    r.render(big, a)
    _status(r, count > 8)
    r.render(small, b)
    _status(r, count > 8)
    assert torch.equal(a[:small.total], b)
    go = torch.randn(big.total, device="cuda")
    ga = torch.full((big.count, 7), 3.0, device="cuda")
    gb = torch.full((count, 7), 3.0, device="cuda")
    r.render_backward(big, go, ga, sersic=True)
    _status(r, count > 8)
    r.render_backward(small, go[:small.total].contiguous(), gb, sersic=True)
    _status(r, count > 8)
    assert torch.equal(ga[:count], gb)


@pytest.mark.parametrize("count", [1, 40, LINE])
def test_composites(gpu_renderer, count):
    import torch
    from paper_2012_15797_gb300.renderer import to_device
    disk, bulge = composite_galaxies(LINE + 64, seed=71, sizes=(32, 64, 128))
    sub = np.arange(count)
    for shift in ("phase", "lanczos"):
        big = gpu_renderer.render_composite(to_device(disk), to_device(bulge), shift=shift)
        small = gpu_renderer.render_composite(to_device(disk.subset(sub)), to_device(bulge.subset(sub)), shift=shift)
        gpu_renderer.sync_status()
        assert torch.equal(big[:small.numel()], small)
