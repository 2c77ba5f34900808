"""What users of the renderer have it do, as cases that can be timed.

Each case is one call (or one fit step) through ``renderer.Renderer`` on a
population with the distributions of ``workloads/galaxies.py``: r_e
log-uniform from 0.3 px, |e| <= 0.6, flux log-uniform 1-1e4, offsets in
[-0.5, 0.5), exp / deV or Sersic profiles, patch sides 32-256.  ``exact`` is
the same model written out in 64 bits with torch alone.
"""

import json
import math
import os
from types import SimpleNamespace

import numpy as np
import torch

from paper_2012_15797_gb300 import renderer as mog

SIDES = (32, 64, 128, 256)
# share of the mixed population per side: r_e log-uniform 0.3-20 px, the side
# the smallest >= 8 r_e
_SPAN = math.log(20.0 / 0.3)
MIXED = {32: math.log(4.0 / 0.3) / _SPAN, 64: math.log(2.0) / _SPAN, 128: math.log(2.0) / _SPAN,
         256: math.log(1.25) / _SPAN}
# most galaxies a drawn case of a kind has: side 64, and the mixed population
MOST = {"render": 100_000, "graph": 200_000, "fit": 50_000, "backward": 30_000, "lanczos": 30_000,
        "lanczos_backward": 10_000, "eigen": 40_000, "composite": 60_000, "host": 5_000, "psf_fit": 64}


def _case(name, kind, count, side, psfs=1, sersic=False, cd=False):
    """side: 32-256, or 0 for the mixed population (Sersic profiles, sides by
    r_e).  psfs: how many PSFs the galaxies are spread over.  sersic: also the
    gradient by the Sersic index.  cd: per-galaxy WCS matrices."""
    c = {"kind": kind, "count": count, "side": side, "psfs": psfs, "sersic": sersic, "cd": cd}
    return dict(c, name=name) if name else c


def listed():
    return [
        # an interactive program or a sampler that renders one source at a time
        _case("one_galaxy_64", "render", 1, 64),
        # one request of a concurrent fit (1-512 galaxies of mixed sides, WCS matrices): render, loss, gradients
        _case("request_mixed_181", "fit", 181, 0, psfs=64, cd=True),
        # a catalogue tile on one patch side, one PSF
        _case("tile_64", "render", 100_000, 64),
        # a survey brick: every side, 64 PSFs, rendered again and again through a captured graph
        _case("brick_mixed_graph", "graph", 200_000, 0, psfs=64),
        # a step of fitting a tile's galaxies to their observed patches
        _case("fit_tile_64", "fit", 50_000, 64),
        # gradients for free Sersic indices over a brick's sides, given the upstream gradient
        _case("backward_mixed_sersic", "backward", 30_000, 0, psfs=64, sersic=True),
        # the Lanczos sub-pixel shift that pipelines comparing with the Tractor ask for
        _case("lanczos_mixed", "lanczos", 30_001, 0, psfs=16),
        # fitting with that shift
        _case("lanczos_backward_64", "lanczos_backward", 9_999, 64),
        # a tile whose PSF varies over the image
        _case("eigen_tile_64", "eigen", 40_000, 64),
        # bulge + disk galaxies of every side
        _case("composite_mixed", "composite", 60_000, 0),
        # parameters and patches in host memory
        _case("host_mixed", "host", 4_099, 0, psfs=4),
        # the mixtures of an exposure's PSFs, fitted on the device
        _case("psf_mixtures_64", "psf_fit", 64, 64),
    ]


def draw(rng):
    kind = rng.choice(sorted(MOST))
    side = rng.choice((0, 0, 32, 64, 64, 128, 256))
    if kind == "psf_fit":   # images from 24 x 24 to 72 x 72, odd sides among them
        return _case(None, kind, _log_int(rng, 1, 64), rng.randint(24, 72))
    # galaxies of the larger sides cost more: the same pixels at most
    area = 4096 if kind in ("render", "fit", "lanczos_backward", "eigen") else _mean_area(0)
    most = max(1, min(MOST[kind], int(MOST[kind] * area / _mean_area(side))))
    psfs = 1 if kind in ("eigen", "composite") else rng.choice((1, 3, 16, 64))
    grads = kind in ("backward", "lanczos_backward")
    return _case(None, kind, _log_int(rng, 1, most), side, psfs=psfs, sersic=grads and rng.random() < 0.5,
                 cd=kind in ("render", "fit", "backward") and rng.random() < 0.3)


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _mean_area(side):
    return float(side * side) if side else sum(s * n * n for n, s in MIXED.items())


def work(case):
    """Parameters and patches once; per pixel the inverse (or forward) real
    transform, 5 N^2 log2 N, and the mixture on the N (N / 2 + 1) bins with
    eight components (the share in real space costs less)."""
    g, kind, side = case["count"], case["kind"], case["side"]
    if kind == "psf_fit":   # the images once, the rows; one Jacobian pass of 18 parameters and its products
        return {"bytes": g * (4.0 * side * side + 76.0), "flops": g * side * side * (3 * 60.0 + 18 * 19.0 + 36.0)}
    sides = {side: 1.0} if side else MIXED
    pix = g * _mean_area(side)
    fft = g * sum(s * 5.0 * n * n * math.log2(n) for n, s in sides.items())
    bins = g * sum(s * n * (n / 2 + 1) for n, s in sides.items())
    profiles = 2 if kind == "composite" else 1
    fwd = fft + bins * (14.0 + 2.0 * 8 * profiles)
    bwd = fft + bins * (32.0 + 7.0 * 8)
    par = (64.0 if case["cd"] else 48.0) * g * profiles
    if kind == "fit":       # data in, the gradient patch out (the gradients' input is this call's own)
        return {"bytes": 8.0 * pix + 2 * par + 28.0 * g, "flops": fwd + bwd}
    if kind in ("backward", "lanczos_backward"):
        return {"bytes": 4.0 * pix + par + (28.0 if case["sersic"] else 24.0) * g, "flops": bwd}
    return {"bytes": 4.0 * pix + par + (8.0 * g if kind == "eigen" else 0.0), "flops": fwd}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
class _Galaxies(SimpleNamespace):
    def __len__(self):
        return len(self.flux)


_TABLES = None


def _tables():
    global _TABLES
    if _TABLES is None:
        path = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "workloads",
                            "mog_profiles.json")
        with open(path) as f:
            doc = json.load(f)
        _TABLES = {int(t["id"]): SimpleNamespace(nodes=np.array(t["nodes"], dtype=np.float64),
                                                 amp=np.array(t["amp"], dtype=np.float64).reshape(-1, 12),
                                                 var=np.array(t["var"], dtype=np.float64).reshape(-1, 12))
                   for t in doc["tables"]}
    return _TABLES


def _pixel_gauss(size, var):
    c = size // 2
    y, x = np.mgrid[0:size, 0:size].astype(np.float64)
    return np.exp(-0.5 * ((x - c) ** 2 + (y - c) ** 2) / var) / (2 * np.pi * var)


def _psf_image(s, size=64):
    """Core 0.8 N(s) + 0.2 N(2 s), Moffat (beta = 3) wings at weight 0.05."""
    c = size // 2
    y, x = np.mgrid[0:size, 0:size].astype(np.float64)
    wings = (1.0 + ((x - c) ** 2 + (y - c) ** 2) / (4.62 * s) ** 2) ** -3.0
    core = 0.8 * _pixel_gauss(size, s * s) + 0.2 * _pixel_gauss(size, 4 * s * s)
    img = 0.95 * core / core.sum() + 0.05 * wings / wings.sum()
    return (img / img.sum()).astype(np.float32)


def _psfs(rng, n):
    out = []
    for _ in range(n):
        s = rng.uniform(1.2, 2.5)
        mix = [[0.76, 0.0, 0.0, s * s, 0.0, s * s], [0.19, 0.0, 0.0, 4 * s * s, 0.0, 4 * s * s],
               [0.05, 0.02, -0.01, 12 * s * s, 0.3, 11 * s * s]]
        out.append(SimpleNamespace(image=_psf_image(s), mog=np.array(mix)))
    return out


def _eigen_psf():
    """Six components (degree 2) sharing three Gaussian shapes: the width
    drifts over a 4096-pixel image."""
    var = np.array([1.6, 3.4, 13.0])
    shapes = np.array([[0.0, 0.0, v, 0.0, v] for v in var])
    amp = np.array([[0.50, 0.38, 0.12], [0.06, -0.05, -0.01], [-0.04, 0.03, 0.01], [0.01, -0.02, 0.01],
                    [0.02, -0.01, -0.01], [-0.01, 0.02, -0.01]])
    g = np.stack([_pixel_gauss(64, v) for v in var])
    return SimpleNamespace(components=np.tensordot(amp, g, axes=1).astype(np.float32), degree=2,
                           norm=(2048.0, 2048.0, 2048.0, 2048.0), mog_shape=shapes, mog_amp=amp)


def _shape(rng, g, emax):
    m, phi = rng.uniform(0.0, emax, g), rng.uniform(0.0, np.pi, g)
    return m * np.cos(2 * phi), m * np.sin(2 * phi)


def _f32(**kw):
    f = {k: np.ascontiguousarray(v, dtype=np.int32 if k in ("profile", "psf", "size") else np.float32)
         for k, v in kw.items()}
    return _Galaxies(**f)


def _per_side(g):
    ends = np.floor(np.cumsum([MIXED[n] for n in SIDES]) * g + 0.5).astype(int)
    ends[-1] = g
    return np.diff(ends, prepend=0)


def _galaxies(case, rng):
    g, side = case["count"], case["side"]
    if side:
        size = np.full(g, side)
        log_re = rng.uniform(math.log(0.3), math.log(0.3125 * side), g)
    else:   # as many galaxies of each side for every seed, in the seed's order
        size = np.repeat(SIDES, _per_side(g))
        lo, hi = np.log(np.where(size == 32, 0.3, size / 16)), np.log(np.minimum(20.0, size / 8))
        order = rng.permutation(g)
        size, log_re = size[order], rng.uniform(lo, hi)[order]
    e1, e2 = _shape(rng, g, 0.6)
    flux = np.exp(rng.uniform(0.0, math.log(1e4), g))
    x, y = rng.uniform(-0.5, 0.5, g), rng.uniform(-0.5, 0.5, g)
    psf = rng.integers(0, case["psfs"], g)
    if not side or case["sersic"]:
        n, profile = rng.uniform(0.5, 6.0, g), np.full(g, 2)
    else:
        profile = rng.integers(0, 2, g)
        n = np.where(profile == 0, 1.0, 4.0)
    return _f32(flux=flux, x=x, y=y, log_re=log_re, e1=e1, e2=e2, sersic_n=n, profile=profile, psf=psf, size=size)


def _bulges(disk, rng):
    g = len(disk)
    e1, e2 = _shape(rng, g, 0.3)
    return _f32(flux=disk.flux * rng.uniform(0.1, 2.0, g), x=disk.x, y=disk.y,
                log_re=disk.log_re + np.log(rng.uniform(0.2, 0.6, g)), e1=e1, e2=e2, sersic_n=np.full(g, 4.0),
                profile=np.full(g, 1), psf=disk.psf, size=disk.size)


def _wcs(rng, g):
    """Rotations and small shears and scales about the pixel grid."""
    t, s = rng.uniform(0.0, 2 * np.pi, g), rng.uniform(0.9, 1.1, g)
    cd = np.stack([s * np.cos(t), s * np.sin(t), -np.sin(t) + rng.uniform(-0.05, 0.05, g), np.cos(t)], axis=1)
    return cd.astype(np.float32).reshape(g, 2, 2)


def _inputs(case, seed):
    """The host arrays of a case, from the seed alone."""
    rng = np.random.default_rng([seed, 15797])
    if case["kind"] == "psf_fit":
        images = np.stack([_psf_image(rng.uniform(1.2, 2.5), case["side"]) for _ in range(case["count"])])
        return SimpleNamespace(images=images)
    psfs = [_eigen_psf()] if case["kind"] == "eigen" else _psfs(rng, case["psfs"])
    gals = _galaxies(case, rng)
    g = len(gals)
    if case["kind"] == "composite":   # exponential disks
        gals.profile[:] = 0
        gals.sersic_n[:] = 1.0
    return SimpleNamespace(
        psfs=psfs, gals=gals, bulges=_bulges(gals, rng) if case["kind"] == "composite" else None,
        positions=(rng.uniform(0, 4096, g).astype(np.float32), rng.uniform(0, 4096, g).astype(np.float32))
        if case["kind"] == "eigen" else None,
        cd=_wcs(rng, g) if case["cd"] else None)


def _observed(gals, total, offsets, seed):
    """Observed patches and inverse variances: elliptical Gaussians of about
    each galaxy's size with noise of 1% of the peak."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    data = torch.randn(total, generator=gen, device="cuda")
    ivar = torch.empty(len(gals), device="cuda")
    for n in np.unique(gals.size):
        idx = np.nonzero(gals.size == n)[0]
        for part in np.array_split(idx, max(1, len(idx) * int(n) ** 2 // (1 << 26))):
            p = {k: torch.from_numpy(getattr(gals, k)[part]).cuda()[:, None, None]
                 for k in ("flux", "x", "y", "log_re", "e1", "e2")}
            r2 = torch.exp(2 * p["log_re"])
            a, d, b = 0.6 * r2 * (1 - p["e1"]) + 4.0, 0.6 * r2 * (1 + p["e1"]) + 4.0, -0.6 * r2 * p["e2"]
            det = a * d - b * b
            c = torch.arange(int(n), device="cuda", dtype=torch.float32) - int(n) / 2
            dx, dy = c[None, None, :] - p["x"] - 0.1, c[None, :, None] - p["y"] + 0.1
            peak = p["flux"] / (2 * math.pi * torch.sqrt(det))
            model = peak * torch.exp(-0.5 * (d * dx * dx - 2 * b * dx * dy + a * dy * dy) / det)
            at = torch.from_numpy(offsets[part]).cuda()[:, None] + torch.arange(int(n) ** 2, device="cuda")
            data[at] = model.reshape(len(part), -1) + 0.01 * peak[:, :, 0] * data[at]
            ivar[torch.from_numpy(part).cuda()] = (1.0 / (0.01 * peak) ** 2)[:, 0, 0]
    return data, ivar


def _upstream(total, seed):
    """A residual-like upstream gradient."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(total, generator=gen, device="cuda") + 0.25


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    d = _inputs(case, seed)
    s = SimpleNamespace(kind=case["kind"], sersic=case["sersic"])
    if s.kind == "psf_fit":
        s.r = mog.Renderer(_tables(), [])
        s.images = torch.from_numpy(d.images).cuda()
        return s
    s.r = mog.Renderer(_tables(), d.psfs)
    if s.kind == "host":
        s.host = mog.host_batch(d.gals, pin=True)
        s.out = torch.empty(s.host[1], dtype=torch.float32).pin_memory()
        return s
    s.batch = mog.to_device(d.gals, positions=d.positions, cd=d.cd)
    total = s.batch.total
    if s.kind == "composite":
        s.bulges = mog.to_device(d.bulges)
    if s.kind == "fit":
        s.data, s.ivar = _observed(d.gals, total, s.batch.offsets, seed)
        s.grad_pix = torch.empty(total, device="cuda")
        s.chi2 = torch.empty(s.batch.count, device="cuda")
    elif s.kind in ("backward", "lanczos_backward"):
        s.upstream = _upstream(total, seed)
    else:
        s.out = torch.empty(total, device="cuda")
    if s.kind == "graph":
        s.graph = s.r.graph(s.batch, s.out)
    return s


def run(s):
    r = s.r
    if s.kind == "render":
        return r.render(s.batch, s.out)
    if s.kind == "graph":
        return s.graph.launch()
    if s.kind == "fit":
        grad_pix, chi2 = r.render_chi2(s.batch, s.data, s.ivar, s.grad_pix, s.chi2)
        return {"grad_pix": grad_pix, "chi2": chi2, "grads": r.render_backward(s.batch, grad_pix)}
    if s.kind == "backward":
        return r.render_backward(s.batch, s.upstream, sersic=s.sersic)
    if s.kind == "lanczos":
        return r.render(s.batch, s.out, shift="lanczos")
    if s.kind == "lanczos_backward":
        return r.render_backward(s.batch, s.upstream, sersic=s.sersic, shift="lanczos")
    if s.kind == "eigen":
        return r.render(s.batch, s.out)
    if s.kind == "composite":
        return r.render_composite(s.batch, s.bulges, s.out)
    if s.kind == "host":
        return r.render_host(s.host, s.out)
    rows, chi2 = r.fit_psf_mixtures(s.images)
    return {"rows": rows, "chi2": chi2}


# ---------------------------------------------------------------------------
# The model in 64 bits
# ---------------------------------------------------------------------------
NAMES = ("flux", "x", "y", "log_re", "e1", "e2", "sersic_n")


def _mixture(gals, part, n_idx):
    """(a, v), (G, 12) each, at Sersic indices n_idx: linear in a and log v."""
    prof = gals.profile[part]
    a = torch.zeros(len(part), 12, dtype=torch.float64, device="cuda")
    v = torch.ones_like(a)
    for pid, t in _tables().items():
        sel = torch.from_numpy(np.nonzero(prof == pid)[0]).cuda()
        if not len(sel):
            continue
        amp, logv = (torch.from_numpy(q.astype(np.float32)).cuda().double() for q in (t.amp, t.var))
        logv = torch.log(logv)
        if len(t.nodes) == 1:
            aa, vv = amp[0].expand(len(sel), 12), torch.exp(logv[0]).expand(len(sel), 12)
        else:
            u = (n_idx[sel] - t.nodes[0]) * ((len(t.nodes) - 1) / (t.nodes[-1] - t.nodes[0]))
            u = u.clamp(0.0, len(t.nodes) - 1.0)
            j = u.detach().long().clamp(max=len(t.nodes) - 2)
            w = (u - j)[:, None]
            aa = (1 - w) * amp[j] + w * amp[j + 1]
            vv = torch.exp((1 - w) * logv[j] + w * logv[j + 1])
        a, v = a.index_copy(0, sel, aa), v.index_copy(0, sel, vv)
    return a, v


def _covariance(p, cd):
    """Pixel covariance per unit profile variance: (s11, s12, s22)."""
    r2, e = torch.exp(2 * p["log_re"]), torch.sqrt(p["e1"] ** 2 + p["e2"] ** 2)
    beta = (1 - e) / (1 + e)
    h, gq = 0.5 * (1 + beta ** 2), 0.5 * (beta ** 2 - 1)
    s11, s12, s22 = r2 * (h + gq * p["e1"] / e), -r2 * gq * p["e2"] / e, r2 * (h - gq * p["e1"] / e)
    if cd is not None:
        m = torch.linalg.inv(cd.double())
        s = torch.stack([torch.stack([s11, s12], -1), torch.stack([s12, s22], -1)], -2)
        s = m @ s @ m.transpose(1, 2)
        s11, s12, s22 = s[:, 0, 0], s[:, 0, 1], s[:, 1, 1]
    return s11, s12, s22


def _spectra(psf_images, n):
    """Half spectra of PSF images (K, h, w) centred at index 0 of n x n."""
    k, h, w = psf_images.shape
    full = torch.zeros(k, n, n, dtype=torch.float64, device="cuda")
    img = torch.from_numpy(np.ascontiguousarray(psf_images)).cuda().double()
    y0, x0 = n // 2 - h // 2, n // 2 - w // 2
    ys, xs = max(0, y0), max(0, x0)
    ye, xe = min(n, y0 + h), min(n, x0 + w)
    full[:, ys:ye, xs:xe] = img[:, ys - y0:ye - y0, xs - x0:xe - x0]
    return torch.fft.rfft2(torch.roll(full, (-(n // 2), -(n // 2)), (1, 2)))


def _lanczos_weights(d):
    t = torch.arange(-3, 4, device="cuda", dtype=torch.float64) - d[:, None]
    w = torch.where(t.abs() < 3, torch.sinc(t) * torch.sinc(t / 3), torch.zeros_like(t))
    return w / w.sum(1, keepdim=True)


def _model(p, gals, part, n, psf_hat, psf_mog, cd, lanczos):
    """(G, n, n) patches.  psf_hat (G, n, n / 2 + 1); psf_mog (G, k, 6)."""
    x, y = p["x"], p["y"]
    if lanczos:
        ix, iy = torch.floor(x.detach() + 0.5), torch.floor(y.detach() + 0.5)
        fx, fy, x, y = x - ix, y - iy, ix, iy
    a, v = _mixture(gals, part, p["sersic_n"])
    s11, s12, s22 = _covariance(p, cd)
    tr = s11 + s22
    nu = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)[None, None, :] / n
    om = torch.fft.fftfreq(n, dtype=torch.float64, device="cuda")[None, :, None]
    q = s11[:, None, None] * nu * nu + 2 * s12[:, None, None] * nu * om + s22[:, None, None] * om * om
    c = torch.arange(n, device="cuda", dtype=torch.float64)
    mix, real = 0.0, 0.0
    for i in range(12):
        ns = 0.5 * n / torch.sqrt(v[:, i] * tr)
        t = (ns - 3).clamp(0, 1)
        wf = t * t * (3 - 2 * t)
        amp = p["flux"] * a[:, i]
        live = a[:, i].detach() != 0
        if live.any():
            mix = mix + (amp * wf)[:, None, None] * torch.exp(-2 * math.pi ** 2 * v[:, i, None, None] * q)
        sel = torch.nonzero(live & (wf.detach() < 1))[:, 0]
        if not len(sel):
            continue
        add = 0.0
        for k in range(psf_mog.shape[1]):
            w, mx, my, pxx, pxy, pyy = (psf_mog[sel, k, u] for u in range(6))
            cxx, cxy, cyy = v[sel, i] * s11[sel] + pxx, v[sel, i] * s12[sel] + pxy, v[sel, i] * s22[sel] + pyy
            det = cxx * cyy - cxy * cxy
            dx = c[None, None, :] - (n / 2 + x[sel] + mx)[:, None, None]
            dy = c[None, :, None] - (n / 2 + y[sel] + my)[:, None, None]
            e = (cyy / det)[:, None, None] * dx * dx - 2 * (cxy / det)[:, None, None] * dx * dy
            e = e + (cxx / det)[:, None, None] * dy * dy
            g = (amp * (1 - wf))[sel] * w / (2 * math.pi * torch.sqrt(det))
            add = add + g[:, None, None] * torch.exp(-0.5 * e)
        zero = torch.zeros(len(part), n, n, dtype=torch.float64, device="cuda")
        real = real + zero.index_add(0, sel, add)
    ph = -2 * math.pi * ((n / 2 + x)[:, None, None] * nu + (n / 2 + y)[:, None, None] * om)
    spec = mix * psf_hat * torch.complex(torch.cos(ph), torch.sin(ph))
    rows = torch.fft.ifft(spec, dim=1)
    # the self-conjugate columns contribute their real part
    edge = torch.zeros(n // 2 + 1, device="cuda", dtype=torch.float64)
    edge[0] = edge[-1] = 1.0
    rows = torch.complex(rows.real, rows.imag * (1 - edge))
    out = torch.fft.irfft(rows, n=n, dim=2) + real
    if lanczos:
        wx, wy = _lanczos_weights(fx), _lanczos_weights(fy)
        out = sum(wx[:, u, None, None] * torch.roll(out, u - 3, 2) for u in range(7))
        out = sum(wy[:, u, None, None] * torch.roll(out, u - 3, 1) for u in range(7))
    return out


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "psf_fit":
        return _fit_mixtures(torch.from_numpy(d.images).cuda().double())
    gals = d.gals
    g = len(gals)
    off, total = _offsets(gals.size)
    lanczos = kind.startswith("lanczos")
    grads = kind in ("fit", "backward", "lanczos_backward")
    names = NAMES if case["sersic"] else NAMES[:6]
    pix = torch.empty(total, dtype=torch.float64, device="cuda") if kind not in ("backward", "lanczos_backward") else None
    gout = torch.empty(g, len(names), dtype=torch.float64, device="cuda") if grads else None
    chi2 = torch.empty(g, dtype=torch.float64, device="cuda")
    if kind == "fit":
        data, ivar = _observed(gals, total, off, seed)
    elif grads:
        up = _upstream(total, seed)
    if kind == "eigen":
        m = _eigen_terms(d)
        shape, amp = d.psfs[0].mog_shape.astype(np.float32), d.psfs[0].mog_amp.astype(np.float32)
        eig_mog = torch.cat([(m @ torch.from_numpy(amp).cuda().double())[:, :, None],
                             torch.from_numpy(shape).cuda().double()[None].expand(g, -1, -1)], 2)
    else:
        mogs = torch.from_numpy(np.stack([q.mog.astype(np.float32) for q in d.psfs])).cuda().double()
    for n in (int(q) for q in np.unique(gals.size)):
        if kind == "eigen":
            hats = _spectra(d.psfs[0].components, n)
        else:
            hats = _spectra(np.stack([q.image for q in d.psfs]), n)
        idx = np.nonzero(gals.size == n)[0]
        step = max(1, (1 << 23 if grads else 1 << 25) // (n * n))
        for lo in range(0, len(idx), step):
            part = idx[lo:lo + step]
            tp = torch.from_numpy(part).cuda()
            at = torch.from_numpy(off[part]).cuda()[:, None] + torch.arange(n * n, device="cuda")
            if kind == "eigen":
                hat, pm = torch.einsum("gc,clk->glk", m[tp].to(hats.dtype), hats), eig_mog[tp]
            else:
                which = torch.from_numpy(gals.psf[part].astype(np.int64)).cuda()
                hat, pm = hats[which], mogs[which]
            cd = torch.from_numpy(d.cd[part]).cuda() if d.cd is not None else None
            p = {k: torch.from_numpy(getattr(gals, k)[part]).cuda().double().requires_grad_(grads) for k in NAMES}
            img = _model(p, gals, part, n, hat, pm, cd, lanczos)
            if kind == "composite":
                b = {k: torch.from_numpy(getattr(d.bulges, k)[part]).cuda().double() for k in NAMES}
                img = img + _model(b, d.bulges, part, n, hat, pm, cd, lanczos)
            img = img.reshape(len(part), -1)
            if kind == "fit":
                r = img - data[at].double()
                iv = ivar[tp].double()
                c2 = iv * (r * r).sum(1)
                chi2[tp] = c2.detach()
                pix[at] = (2 * iv[:, None] * r).detach()
                loss = c2.sum()
            elif grads:
                loss = (img * up[at].double()).sum()
            else:
                pix[at] = img
            if grads:
                got = torch.autograd.grad(loss, [p[k] for k in names], allow_unused=True)
                gout[tp] = torch.stack([torch.zeros(len(part), dtype=torch.float64, device="cuda") if q is None else q
                                        for q in got], 1)
    if kind == "fit":
        return {"grad_pix": pix, "chi2": chi2, "grads": gout}
    if grads:
        return gout
    return pix.cpu() if kind == "host" else pix


def _offsets(sizes):
    area = sizes.astype(np.int64) ** 2
    return np.concatenate([[0], np.cumsum(area)[:-1]]).astype(np.int64), int(area.sum())


def _eigen_terms(d):
    u0, v0, su, sv = d.psfs[0].norm
    u, v = ((torch.from_numpy(q).cuda().double() - c) / s for q, c, s in zip(d.positions, (u0, v0), (su, sv)))
    return torch.stack([torch.ones_like(u), u, v, u * u, u * v, v * v], 1)


def _fit_mixtures(img, k=3, iters=300):
    """Damped Gauss-Newton fits of k-component mixtures to a batch of images,
    from the documented start (image sum and second moment)."""
    b, h, w = img.shape
    yy, xx = torch.meshgrid(torch.arange(h, device="cuda", dtype=torch.float64) - h // 2,
                            torch.arange(w, device="cuda", dtype=torch.float64) - w // 2, indexing="ij")
    dx, dy, data = xx.reshape(1, -1), yy.reshape(1, -1), img.reshape(b, -1)
    tot = data.sum(1)
    s = torch.sqrt(((data * (dx * dx + dy * dy)).sum(1) / (2 * tot)).clamp(min=0.25))
    w0 = torch.tensor([0.55, 0.35, 0.08, 0.015], dtype=torch.float64, device="cuda")[:k]
    th = torch.zeros(b, k, 6, dtype=torch.float64, device="cuda")
    for c, sc in enumerate((0.6, 1.1, 2.2, 4.0)[:k]):
        th[:, c, 0] = torch.log(w0[c] / w0.sum() * tot)
        th[:, c, 3] = th[:, c, 5] = torch.log(s * sc)

    def parts(th, jac):
        model, cols = 0.0, []
        for c in range(k):
            lw, mx, my, la, bb, lc = (th[:, c, u, None] for u in range(6))
            a, cc = torch.exp(la), torch.exp(lc)
            det = (a * cc) ** 2
            ixx, ixy, iyy = (bb * bb + cc * cc) / det, -a * bb / det, a * a / det
            ex, ey = dx - mx, dy - my
            ux, uy = ixx * ex + ixy * ey, ixy * ex + iyy * ey
            g = torch.exp(lw - 0.5 * (ex * ux + ey * uy)) / (2 * math.pi * a * cc)
            model = model + g
            if jac:
                qxx, qxy, qyy = 0.5 * (ux * ux - ixx), 0.5 * (ux * uy - ixy), 0.5 * (uy * uy - iyy)
                cols += [g, g * ux, g * uy, g * (2 * a * a * qxx + 2 * a * bb * qxy), g * (2 * a * qxy + 2 * bb * qyy),
                         g * 2 * cc * cc * qyy]
        return (model - data, torch.stack(cols, 2)) if jac else model - data

    lam = torch.full((b,), 1e-3, dtype=torch.float64, device="cuda")
    eye = torch.eye(6 * k, dtype=torch.float64, device="cuda")
    for _ in range(iters):
        r, j = parts(th, True)
        a = j.transpose(1, 2) @ j
        gr = (j * r[:, :, None]).sum(1)
        sc = torch.sqrt(torch.diagonal(a, dim1=1, dim2=2))
        m = a / (sc[:, :, None] * sc[:, None, :]) + lam[:, None, None] * eye
        step = torch.linalg.solve(m, -(gr / sc)[:, :, None])[:, :, 0] / sc
        new = th + step.reshape(b, k, 6)
        better = (parts(new, False) ** 2).sum(1) < (r * r).sum(1)
        th = torch.where(better[:, None, None], new, th)
        lam = torch.where(better, (lam / 3).clamp(min=1e-10), (lam * 4).clamp(max=1e6))
    chi2 = (parts(th, False) ** 2).sum(1)
    th = torch.gather(th, 1, torch.argsort(-th[:, :, 0], 1)[:, :, None].expand(-1, -1, 6))
    a, bb, cc = torch.exp(th[:, :, 3]), th[:, :, 4], torch.exp(th[:, :, 5])
    rows = torch.stack([torch.exp(th[:, :, 0]), th[:, :, 1], th[:, :, 2], a * a, a * bb, bb * bb + cc * cc], 2)
    return {"rows": rows, "chi2": chi2}
