"""The kernels with 16 values per thread (256 x 256, 128 x 128, 64 x 64) against the FP64
oracle, with a galaxy that is skipped in the middle.  Forward, every mode: batch
sizes around the pipeline depth (tables one galaxy ahead, records three ahead),
for 256 x 256 below and above the line from which a CTA and no longer a cluster
renders a galaxy: max |d pixel| <= 2e-6 flux (the render tolerance); adding to
an image gives the image plus the model.  Adjoint: every kernel agrees with the
oracle's gradients within the adjoint tolerance; at integer offsets the Lanczos
shift does the same operations as the phase shift, so that every gradient but x
and y is the same."""

import numpy as np
import pytest

from oracle import lanczos as L
from oracle import render as R
from test_render_gpu import EDGE, _gals, _row

pytestmark = pytest.mark.gpu

TOL = 2e-6


def _batch(count, bad, size=256):
    rows = [_row(**{"size": size, "x": 0.37 - 0.1 * (i % 7), "y": -0.21 + 0.05 * (i % 7), **EDGE[(i % 7) % len(EDGE)]})
            for i in range(count)]
    gals = _gals(rows)
    if bad is not None:
        gals.flux[bad] = np.nan
    return gals


@pytest.mark.parametrize("mode", ["phase", "lanczos", "loss", "composite"])
@pytest.mark.parametrize("size,count,bad", [(256, 1, None), (256, 2, 0), (256, 3, 1), (256, 7, 3), (256, 640, 637),
                                            (128, 1, None), (128, 2, 0), (128, 3, 1), (128, 640, 637),
                                            (64, 1, None), (64, 2, 0), (64, 3, 1), (64, 640, 637)])
def test_parity_with_skipped_galaxies(gpu_renderer, tables, mode, size, count, bad):
    import torch
    from paper_2012_15797_gb300 import capi
    from paper_2012_15797_gb300.renderer import patches, to_device
    gals = _batch(count, bad, size)
    # one CTA per SM and long queue chunks: a CTA takes several galaxies in turn
    capi.mog_set_launch_shape(gpu_renderer.ctx, 0, size, 1, 8, 0)
    try:
        b = to_device(gals)
        out = torch.full((b.total,), 7.0, device="cuda")
        data = torch.zeros_like(out)
        chi2 = None
        if mode == "loss":
            ivar = torch.full((count,), 0.5, device="cuda")
            _, chi2 = gpu_renderer.render_chi2(b, data, ivar, out)   # grad = 2 ivar (model - 0) = model
        elif mode == "composite":
            gpu_renderer.render_composite(b, b, out)
        else:
            gpu_renderer.render(b, out, shift=mode)
        if bad is None:
            gpu_renderer.sync_status()
        else:
            with pytest.raises(capi.MogError):
                gpu_renderer.sync_status()
    finally:
        capi.mog_set_launch_shape(gpu_renderer.ctx, 0, size, 0, 1, 0)
    got = patches(out, b)
    for i in range(max(0, count - 7), count):
        if i == bad:
            assert bool((got[i] == 7.0).all())
            assert chi2 is None or bool(torch.isnan(chi2[i]))
            continue
        g = gals.row(i)
        psf = gpu_renderer.psfs[g["psf"]]
        ref = (L.render_lanczos if mode == "lanczos" else R.render)(g, psf.image, psf.mog, tables)
        flux = g["flux"] * (2.0 if mode == "composite" else 1.0)
        ref = ref * (2.0 if mode == "composite" else 1.0)
        img = got[i].double().cpu().numpy()
        assert np.max(np.abs(img - ref)) <= TOL * flux, i
        if chi2 is not None:
            want = 0.5 * np.sum(ref * ref)
            assert abs(float(chi2[i]) - want) <= 1e-5 * want, i


@pytest.mark.parametrize("sersic", [False, True])
@pytest.mark.parametrize("size,count,bad", [(256, 1, None), (256, 3, 1), (256, 41, 38), (256, 300, 297),
                                            (128, 1, None), (128, 3, 1), (128, 400, 397)])
def test_adjoint_parity_with_skipped_galaxies(gpu_renderer, tables, sersic, size, count, bad):
    import torch
    from paper_2012_15797_gb300 import capi
    from paper_2012_15797_gb300.renderer import to_device
    from oracle import adjoint as A
    gals = _batch(count, bad, size)
    b = to_device(gals)
    go = torch.randn(b.total, generator=torch.Generator(device="cuda").manual_seed(count), device="cuda")
    gp = torch.full((count, 7 if sersic else 6), 7.0, device="cuda")
    gpu_renderer.render_backward(b, go, gp, sersic=sersic)
    if bad is None:
        gpu_renderer.sync_status()
    else:
        with pytest.raises(capi.MogError):
            gpu_renderer.sync_status()
    got = gp.double().cpu().numpy()
    for i in range(max(0, count - 4), count):
        if i == bad:
            assert np.all(got[i] == 7.0)
            continue
        g = gals.row(i)
        psf = gpu_renderer.psfs[g["psf"]]
        pix = go[int(b.offsets[i]):int(b.offsets[i]) + size * size].double().cpu().numpy().reshape(size, size)
        hat = R.psf_spectrum(psf.image, size)
        want = A.vjp(g, hat, psf.mog, tables, pix)
        norm = np.abs(pix).sum()
        scale = np.array([1.0] + [abs(g["flux"])] * 5)
        assert np.all(np.abs(got[i, :6] - want) <= 1e-4 * np.abs(want) + 1e-5 * norm * scale), i
        if sersic:
            dn = float(np.sum(A.sersic_derivative(g, hat, psf.mog, tables) * pix))
            assert abs(got[i, 6] - dn) <= 1e-4 * abs(dn) + 1e-5 * norm * abs(g["flux"]), i


@pytest.mark.parametrize("size,count", [(256, 1), (256, 41), (256, 300), (128, 1), (128, 400)])
def test_lanczos_adjoint_small_and_large_batches(gpu_renderer, tables, size, count):
    import torch
    from paper_2012_15797_gb300.renderer import to_device
    from test_lanczos_adjoint_gpu import check, oracle_grads_lanczos
    gals = _batch(count, None, size)
    b = to_device(gals)
    go = torch.randn(b.total, generator=torch.Generator(device="cuda").manual_seed(count), device="cuda")
    got = gpu_renderer.render_backward(b, go, shift="lanczos")
    last = [go[int(b.offsets[-1]):].double().cpu().numpy().reshape(size, size)]
    one = gals.subset(np.array([count - 1]))
    check(got[-1:].double().cpu().numpy(), oracle_grads_lanczos(one, gpu_renderer.psfs, tables, last), one, last)
    gals.x[:] = np.round(gals.x * 4)
    gals.y[:] = np.round(gals.y * 4)
    b = to_device(gals)
    lz = gpu_renderer.render_backward(b, go, shift="lanczos")
    phase = gpu_renderer.render_backward(b, go)
    gpu_renderer.sync_status()
    cols = [0, 3, 4, 5]
    assert torch.equal(lz[:, cols], phase[:, cols])


@pytest.mark.parametrize("mode", ["phase", "lanczos"])
@pytest.mark.parametrize("size", [64, 128, 256])
def test_adding_to_an_image_is_the_image_plus_the_model(gpu_renderer, mode, size):
    import torch
    from paper_2012_15797_gb300.renderer import to_device
    b = to_device(_batch(9, None, size))
    base = torch.randn(b.total, device="cuda")
    out = base.clone()
    gpu_renderer.render(b, out, shift=mode, add=True)
    assert torch.equal(out, base + gpu_renderer.render(b, shift=mode))
    gpu_renderer.sync_status()


@pytest.mark.parametrize("chunk", [1, 3])
@pytest.mark.parametrize("mode", ["phase", "lanczos"])
def test_psfs_that_change_from_galaxy_to_galaxy(gpu_renderer, mode, chunk):
    """64 x 64, few galaxies of each of five PSFs per CTA (one CTA per SM), the
    first of a PSF skipped now and then: the bits of every galaxy by itself."""
    import torch
    from paper_2012_15797_gb300 import capi
    from paper_2012_15797_gb300.renderer import patches, to_device
    count = 1500
    gals = _batch(count, None, 64)
    gals.psf[:] = np.arange(count) % 5
    gals.flux[::211] = np.nan
    capi.mog_set_launch_shape(gpu_renderer.ctx, 0, 64, 1, chunk, 0)
    try:
        b = to_device(gals)
        out = gpu_renderer.render(b, torch.zeros(b.total, device="cuda"), shift=mode)
        with pytest.raises(capi.MogError):
            gpu_renderer.sync_status()
    finally:
        capi.mog_set_launch_shape(gpu_renderer.ctx, 0, 64, 0, 1, 0)
    got = patches(out, b)
    for i in range(1, count, 37):
        if np.isnan(gals.flux[i]):
            continue
        one = to_device(gals.subset(np.array([i])))
        alone = patches(gpu_renderer.render(one, shift=mode), one)[0]
        assert torch.equal(got[i], alone), i
    gpu_renderer.sync_status()
