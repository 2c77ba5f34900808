"""The 256 x 256 forward kernel (16 values per thread, per-galaxy tables one
galaxy ahead, records three ahead) against the FP64 oracle at batch sizes
around its pipeline depth, with a galaxy that is skipped in the middle, in
every mode: max |d pixel| <= 2e-6 flux (the render tolerance)."""

import numpy as np
import pytest

from oracle import lanczos as L
from oracle import render as R
from test_render_gpu import EDGE, _gals, _row

pytestmark = pytest.mark.gpu

TOL = 2e-6


def _batch(count, bad):
    rows = [_row(**{"size": 256, "x": 0.37 - 0.1 * i, "y": -0.21 + 0.05 * i, **EDGE[i % len(EDGE)]})
            for i in range(count)]
    gals = _gals(rows)
    if bad is not None:
        gals.flux[bad] = np.nan
    return gals


@pytest.mark.parametrize("mode", ["phase", "lanczos", "loss", "composite"])
@pytest.mark.parametrize("count,bad", [(1, None), (2, 0), (3, 1), (5, 4), (7, 3)])
def test_parity_with_skipped_galaxies(gpu_renderer, tables, mode, count, bad):
    import torch
    from paper_2012_15797_gb300 import capi
    from paper_2012_15797_gb300.renderer import patches, to_device
    gals = _batch(count, bad)
    # one CTA per SM and long queue chunks: a CTA takes several galaxies in turn
    capi.mog_set_launch_shape(gpu_renderer.ctx, 0, 256, 1, 8, 0)
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
        capi.mog_set_launch_shape(gpu_renderer.ctx, 0, 256, 0, 1, 0)
    got = patches(out, b)
    for i in range(count):
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
