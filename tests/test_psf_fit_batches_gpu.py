"""PSF-mixture fits of large batches take smaller CTAs than those of a few images
(more than three images per SM of at most 24 chunks of 256 pixels; with two
components twelve, of five chunks; with one any size from twelve per SM): every image has the
same rows and chi^2, bit for bit, in both, at sizes around whole chunks."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _image(rng, h, w):
    y, x = np.mgrid[0:h, 0:w].astype(np.float64)
    s = rng.uniform(1.2, 2.2)
    img = np.zeros((h, w))
    for wt, var in ((0.75, s * s), (0.2, 4 * s * s), (0.05, 9 * s * s)):
        img += wt * np.exp(-0.5 * ((x - w // 2) ** 2 + (y - h // 2) ** 2) / var) / (2 * np.pi * var)
    return (img + 1e-5 * rng.standard_normal((h, w))).astype(np.float32)


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("h,w", [(16, 16), (17, 15), (16, 17), (25, 25), (32, 40), (35, 37)])
def test_a_large_batch_has_the_bits_of_a_small_one(gpu_renderer, k, h, w):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(1000 * k + h)
    few = torch.from_numpy(np.stack([_image(rng, h, w) for _ in range(24)])).cuda()
    line = (12 if k == 2 else 3) * sms
    many = few.repeat(line // 24 + 1, 1, 1)
    assert many.shape[0] > line
    rows, chi2 = gpu_renderer.fit_psf_mixtures(few, k=k, iters=40)
    more_rows, more_chi2 = gpu_renderer.fit_psf_mixtures(many, k=k, iters=40)
    gpu_renderer.sync_status()
    assert bool(torch.isfinite(rows).all()) and bool(torch.isfinite(chi2).all())
    n = many.shape[0] // 24
    assert torch.equal(more_rows, rows.repeat(n, 1, 1)[:many.shape[0]])
    assert torch.equal(more_chi2, chi2.repeat(n)[:many.shape[0]])


def test_one_component_and_large_images(gpu_renderer):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(7)
    few = torch.from_numpy(np.stack([_image(rng, 81, 83) for _ in range(8)])).cuda()   # 27 chunks
    many = few.repeat((12 * sms) // 8 + 1, 1, 1)
    rows, chi2 = gpu_renderer.fit_psf_mixtures(few, k=1, iters=25)
    more_rows, more_chi2 = gpu_renderer.fit_psf_mixtures(many, k=1, iters=25)
    gpu_renderer.sync_status()
    n = many.shape[0] // 8
    assert torch.equal(more_rows, rows.repeat(n, 1, 1)) and torch.equal(more_chi2, chi2.repeat(n))
