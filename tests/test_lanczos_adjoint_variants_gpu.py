"""The Lanczos adjoint's kernel variants that the plain ones do not reach: with the
Sersic-index gradient and with an eigen-PSF, at the sides whose kernels have one
form (256 x 256: test_routes256_gpu.py), against the FP64 oracle with the
adjoint's tolerance; constant-PSF and eigen-PSF galaxies in one batch, and one
that is skipped."""

import numpy as np
import pytest

from oracle import eigenpsf as E
from oracle import lanczos as L
from oracle import render as R
from test_adjoint_gpu import _gals, _row
from test_eigenpsf_gpu import eig, eig_renderer   # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu

ROWS = [
    dict(e1=0.3, e2=-0.2, x=0.31, y=-0.44), dict(profile=2, sersic_n=2.6, e1=-0.25, e2=0.1, x=-0.12, y=0.27),
    dict(profile=2, sersic_n=5.1, log_re=np.log(7.0), x=1.4, y=0.05),
    dict(log_re=np.log(12.0), profile=1, sersic_n=4.0, e1=0.1, e2=0.2, x=-0.5, y=0.49),
    dict(profile=2, sersic_n=0.7, log_re=np.log(0.4), x=0.0, y=0.25),
]


def _want(gals, i, pos, eig, psf0, tables, pix, sersic):   # noqa: F811
    g = gals.row(i)
    if g["psf"] == 1:
        img, mog = E.psf_at(eig, float(pos[0][i]), float(pos[1][i]))
    else:
        img, mog = psf0.image, psf0.mog
    hat = R.psf_spectrum(img, g["size"])
    out = L.vjp_lanczos(g, hat, mog, tables, pix)
    if sersic:
        out = np.append(out, np.sum(L.sersic_derivative_lanczos(g, hat, mog, tables) * pix))
    return out


@pytest.mark.parametrize("size", [32, 64, 128])
@pytest.mark.parametrize("sersic", [False, True])
@pytest.mark.parametrize("eigen", [False, True])
def test_against_the_oracle(gpu_renderer, eig_renderer, eig, psf0, tables, size, sersic, eigen):   # noqa: F811
    import torch
    from paper_2012_15797_gb300 import capi
    from paper_2012_15797_gb300.renderer import to_device
    r = eig_renderer if eigen else gpu_renderer
    gals = _gals([_row(size=size, psf=p, **e) for p in ((1, 0) if eigen else (0,)) for e in ROWS])
    skipped = 2
    gals.flux[skipped] = np.nan
    rng = np.random.default_rng(500 + size)
    pos = (rng.uniform(0, 4096, len(gals)).astype(np.float32), rng.uniform(0, 4096, len(gals)).astype(np.float32))
    pix = [rng.normal(size=(size, size)).astype(np.float32).astype(np.float64) + 0.25 for _ in range(len(gals))]
    b = to_device(gals, positions=pos if eigen else None)
    go = torch.from_numpy(np.concatenate([g.ravel() for g in pix]).astype(np.float32)).cuda()
    gp = torch.full((len(gals), 7 if sersic else 6), 7.0, device="cuda")
    r.render_backward(b, go, gp, sersic=sersic, shift="lanczos")
    with pytest.raises(capi.MogError):
        r.sync_status()
    got = gp.double().cpu().numpy()
    for i in range(len(gals)):
        if i == skipped:
            assert np.all(got[i] == 7.0)
            continue
        want = _want(gals, i, pos, eig, psf0, tables, pix[i], sersic)
        scale = np.array([1.0] + [float(gals.flux[i])] * (len(want) - 1)) * np.abs(pix[i]).sum()
        assert np.all(np.abs(got[i] - want) <= 1e-4 * np.abs(want) + 1e-5 * scale), (i, got[i], want)
