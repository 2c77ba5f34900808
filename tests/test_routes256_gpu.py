"""256 x 256 galaxies: the kernel of a few (a cluster of CTAs per galaxy) and the
one of many (a CTA per galaxy) are chosen by how many there are, so a galaxy has
to have the same bits from both, in every mode.  Batches above the lines between
them (8 galaxies per SM; 0.75 for the adjoint, 1.5 with the Lanczos shift), with
galaxies that are skipped, against the batch of their first galaxies, and against
the FP64 oracle with the tolerances of the parity tests (render: max |d pixel| <=
2e-6 flux; gradients: 1e-4 |g| + 1e-5 ||dL/dpix||_1 s)."""

import numpy as np
import pytest

from oracle import eigenpsf as E
from oracle import lanczos as L
from oracle import render as R
from workloads import eigen_positions
from test_eigenpsf_gpu import eig, eig_renderer   # noqa: F401  (fixtures)
from test_values16_gpu import _batch

pytestmark = pytest.mark.gpu

FEW = 24          # galaxies of the small batch
SKIPPED = (3, 20)  # galaxies with a parameter that is not finite
MANY = 3200
N = 256


@pytest.fixture
def renderer(request, gpu_renderer, eig_renderer):   # noqa: F811
    return {"constant": gpu_renderer, "eigen": eig_renderer}[request.param]


def _galaxies(count, eigen):
    gals = _batch(count, None, N)
    gals.log_re[::3] = np.log(40.0)   # some with real-space terms
    gals.profile[::6] = 1
    gals.sersic_n[::6] = 4.0
    gals.flux[list(SKIPPED)] = np.nan
    gals.flux[count - 2] = np.nan
    if eigen:
        gals.psf[:] = 1
    return gals, (eigen_positions(count, seed=91) if eigen else None)


def _reference(gals, pos, i, shift, renderer, eig, tables):   # noqa: F811
    g = gals.row(i)
    if pos is not None:
        img, mog = E.psf_at(eig, float(pos[0][i]), float(pos[1][i]))
    else:
        img, mog = renderer.psfs[g["psf"]].image, renderer.psfs[g["psf"]].mog
    return (L.render_lanczos if shift == "lanczos" else R.render)(g, img, mog, tables)


def _sub(gals, pos):
    few = np.arange(FEW)
    return gals.subset(few), (None if pos is None else (pos[0][:FEW], pos[1][:FEW]))


def _status(r):
    from paper_2012_15797_gb300 import capi
    with pytest.raises(capi.MogError):
        r.sync_status()


@pytest.mark.parametrize("shift", ["phase", "lanczos"])
@pytest.mark.parametrize("renderer,eigen,mode", [   # (composites take constant PSFs)
    ("constant", False, "render"), ("constant", False, "add"), ("constant", False, "composite"),
    ("eigen", True, "render"), ("eigen", True, "add")], indirect=["renderer"])
def test_renders(renderer, eig, tables, eigen, mode, shift):   # noqa: F811
    import torch
    from paper_2012_15797_gb300.renderer import patches, to_device
    count = MANY
    gals, pos = _galaxies(count, eigen)
    base = torch.randn(count * N * N, generator=torch.Generator(device="cuda").manual_seed(7), device="cuda")

    def run(g, q):
        b = to_device(g, positions=q)
        out = base[:b.total].clone()
        if mode == "composite":
            renderer.render_composite(b, b, out, shift=shift)
        else:
            renderer.render(b, out, shift=shift, add=mode == "add")
        _status(renderer)
        return out, b

    many, b = run(gals, pos)
    few, bf = run(*_sub(gals, pos))
    assert torch.equal(many[:few.numel()], few)
    skipped = [*SKIPPED, count - 2]
    got, before = patches(many, b), patches(base, b)
    if mode == "add":
        plain = torch.zeros_like(base)
        renderer.render(b, plain, shift=shift)
        _status(renderer)
        assert torch.equal(many, base + plain)
    for i in skipped:
        assert torch.equal(got[i], before[i])
    for i in [*range(7), *range(count - 4, count)]:
        if i in skipped:
            continue
        flux = float(gals.flux[i]) * (2.0 if mode == "composite" else 1.0)
        ref = _reference(gals, pos, i, shift, renderer, eig, tables) * (2.0 if mode == "composite" else 1.0)
        img = got[i].double().cpu().numpy()
        if mode == "add":   # (the sum is rounded to the pixel that was there)
            img, tol = img - before[i].double().cpu().numpy(), 2e-6 * flux + 3e-7 * float(before[i].abs().max())
        else:
            tol = 2e-6 * flux
        assert np.max(np.abs(img - ref)) <= tol, i


def test_lanczos_batches_in_host_memory(gpu_renderer):
    """Chunks below the line between the kernels, the same bits as one call above it."""
    import torch
    from paper_2012_15797_gb300.renderer import host_batch, to_device
    gals = _batch(MANY, None, N)
    gals.log_re[::3] = np.log(40.0)
    want = gpu_renderer.render(to_device(gals), shift="lanczos")
    got = gpu_renderer.render_host(host_batch(gals), torch.empty(want.numel()), shift="lanczos")
    gpu_renderer.sync_status()
    assert torch.equal(want.cpu(), got)


@pytest.mark.parametrize("renderer,eigen", [("constant", False), ("eigen", True)], indirect=["renderer"])
def test_loss(renderer, eig, tables, eigen):   # noqa: F811
    """Pixels, gradient patches and chi^2, whose sum has one order in both kernels."""
    import torch
    from paper_2012_15797_gb300.renderer import patches, to_device
    count = MANY
    gals, pos = _galaxies(count, eigen)
    data = torch.randn(count * N * N, generator=torch.Generator(device="cuda").manual_seed(8), device="cuda")
    ivar = torch.rand(count, generator=torch.Generator(device="cuda").manual_seed(9), device="cuda") + 0.5

    def run(g, q):
        b = to_device(g, positions=q)
        grad = torch.full((b.total,), 7.0, device="cuda")
        model = torch.full((b.total,), 7.0, device="cuda")
        _, chi2 = renderer.render_chi2(b, data[:b.total], ivar[:b.count], grad, model=model)
        _status(renderer)
        return b, grad, model, chi2

    b, grad, model, chi2 = run(gals, pos)
    _, fgrad, fmodel, fchi2 = run(*_sub(gals, pos))
    assert torch.equal(grad[:fgrad.numel()], fgrad) and torch.equal(model[:fmodel.numel()], fmodel)
    assert torch.equal(chi2[:FEW].nan_to_num(-1.0), fchi2.nan_to_num(-1.0))
    skipped = [*SKIPPED, count - 2]
    assert sorted(torch.nonzero(torch.isnan(chi2))[:, 0].tolist()) == skipped
    pg, pm, pd = patches(grad, b), patches(model, b), patches(data, b)
    for i in [*range(7), *range(count - 4, count)]:
        if i in skipped:
            assert bool((pg[i] == 7.0).all()) and bool((pm[i] == 7.0).all())
            continue
        ref = _reference(gals, pos, i, "phase", renderer, eig, tables)
        assert np.max(np.abs(pm[i].double().cpu().numpy() - ref)) <= 2e-6 * float(gals.flux[i]), i
        assert torch.equal(pg[i], 2.0 * ivar[i] * (pm[i] - pd[i]))
        want = float(ivar[i]) * np.sum((ref - pd[i].double().cpu().numpy()) ** 2)
        assert abs(float(chi2[i]) - want) <= 1e-5 * want, i


@pytest.mark.parametrize("shift", ["phase", "lanczos"])
@pytest.mark.parametrize("sersic", [False, True])
@pytest.mark.parametrize("renderer,eigen", [("constant", False), ("eigen", True)], indirect=["renderer"])
def test_adjoint(renderer, eig, tables, eigen, sersic, shift):   # noqa: F811
    import torch
    from oracle import adjoint as A
    from paper_2012_15797_gb300.renderer import to_device
    count = 400   # more than there are CTAs, so that some take two galaxies
    gals, pos = _galaxies(count, eigen)
    go = torch.randn(count * N * N, generator=torch.Generator(device="cuda").manual_seed(10), device="cuda") + 0.25

    def run(g, q):
        b = to_device(g, positions=q)
        gp = torch.full((b.count, 7 if sersic else 6), 7.0, device="cuda")
        renderer.render_backward(b, go[:b.total].contiguous(), gp, sersic=sersic, shift=shift)
        _status(renderer)
        return gp

    many, few = run(gals, pos), run(*_sub(gals, pos))
    assert torch.equal(many[:FEW], few)
    skipped = [*SKIPPED, count - 2]
    for i in [*range(7), *range(count - 4, count)]:
        if i in skipped:
            assert bool((many[i] == 7.0).all())
            continue
        g = gals.row(i)
        if g["e1"] == 0.0 and g["e2"] == 0.0:   # not differentiable by e1, e2
            continue
        if eigen:
            img, mog = E.psf_at(eig, float(pos[0][i]), float(pos[1][i]))
        else:
            img, mog = renderer.psfs[g["psf"]].image, renderer.psfs[g["psf"]].mog
        pix = go[i * N * N:(i + 1) * N * N].double().cpu().numpy().reshape(N, N)
        hat = R.psf_spectrum(img, N)
        want = (L.vjp_lanczos if shift == "lanczos" else A.vjp)(g, hat, mog, tables, pix)
        if sersic:
            dn = (L.sersic_derivative_lanczos if shift == "lanczos" else A.sersic_derivative)(g, hat, mog, tables)
            want = np.append(want, np.sum(dn * pix))
        scale = np.array([1.0] + [abs(g["flux"])] * (len(want) - 1)) * np.abs(pix).sum()
        got = many[i].double().cpu().numpy()
        assert np.all(np.abs(got - want) <= 1e-4 * np.abs(want) + 1e-5 * scale), (i, got, want)


def test_served_alone_and_in_a_micro_batch(gpu_renderer):
    """Requests of a few 256 x 256 galaxies among others, one micro-batch each
    and in micro-batches of hundreds: the same gradients and chi^2."""
    from paper_2012_15797_gb300.serving import Server, make_fits
    from workloads import mixed_galaxies
    gals = _batch(400, None, N)
    gals.size[::5] = mixed_galaxies(80, seed=92, n_psf=1).size
    gals.log_re[:] = np.minimum(gals.log_re, np.log(gals.size / 8.0)).astype(np.float32)
    state = make_fits(gpu_renderer, [gals])
    rng = np.random.default_rng(93)
    reqs = []
    for _ in range(12):
        c = int(rng.integers(1, 60))
        first = int(rng.integers(0, len(gals) - c + 1))
        p = gals.params6()[first:first + c].copy()
        p[:, 0] *= 1.0 + 0.05 * rng.standard_normal(c)
        reqs.append((0, first, p.astype(np.float32)))
    got = []
    for most in (0, 4096):
        srv = Server(gpu_renderer, budget_bytes=1 << 30, lanes=1, max_batch_galaxies=most)
        srv.add_fit(**state[0])
        tickets, keeps = srv.replay(reqs, np.zeros(len(reqs)))
        srv.wait_replayed(tickets, keeps)
        stats = srv.stats()
        assert (stats["batches"] == len(reqs)) == (most == 0)
        srv.close()
        got.append([(k[1].copy(), k[2].copy()) for k in keeps])
    for (g0, c0), (g1, c1) in zip(*got):
        assert np.all(np.isfinite(g0)) and np.all(np.isfinite(c0))
        np.testing.assert_array_equal(g0, g1)
        np.testing.assert_array_equal(c0, c1)


def test_autotuning_few_galaxies_leaves_the_kernel_of_many_at_its_full_size(tables, psf0):
    """Where the cluster kernel renders, CTAs per SM change nothing: no choice of
    them is kept from its times, for the larger batches of the same context."""
    import torch
    from paper_2012_15797_gb300.renderer import Renderer, to_device
    from workloads import mixed_galaxies
    r = Renderer(tables, [psf0])
    try:
        gals = mixed_galaxies(1300, seed=94, n_psf=1)   # above the line of renders in all, 256 x 256 galaxies below both
        assert np.count_nonzero(gals.size == 256) < 100
        b = to_device(gals)
        out, go = torch.empty(b.total, device="cuda"), torch.randn(b.total, device="cuda")
        shapes = r.autotune(b, out, go, torch.empty(b.count, 6, device="cuda"), reps=1)
        r.sync_status()
        assert shapes[("fwd", 256)][0] == 2 and shapes[("fwd", 256)][2] == 0
        assert shapes[("bwd", 256)][:2] == (1, 1)
    finally:
        r.close()
