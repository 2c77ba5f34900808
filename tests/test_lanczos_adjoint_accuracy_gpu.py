"""Rounding of the Lanczos adjoint's d/dx and d/dy where it shows: wide galaxies
and an upstream gradient with a mean.  The slopes of the shift's weights add up
to zero, so the mean contributes nothing; a remainder r of their FP32 sum would
contribute r flux sum(g) / N^2, and FP32 sums of seven taps of up to 1.4 leave r
of about 1e-7 (unit in the last place 2^-23).

Tolerance, upstream of N(1, 1): 3e-8 flux + 1e-6 |value|.  What is left to
rounding: each pixel's convolved gradient, to about 2e-7 with random sign, which
the model's N^2 / 10 or more pixels average to below 1e-8 flux; the products of
the transform and the weights' own rounding, relative to the value, 3e-7."""

import numpy as np
import pytest

from test_adjoint_gpu import _gals, _row
from test_lanczos_adjoint_gpu import gpu_grads_lanczos, oracle_grads_lanczos

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [32, 64, 128, 256])
def test_a_mean_of_the_upstream_gradient_leaves_x_and_y_alone(gpu_renderer, tables, size):
    rng = np.random.default_rng(900 + size)
    rows = [_row(size=size, flux=100.0, x=float(rng.uniform(-0.5, 0.5)), y=float(rng.uniform(-0.5, 0.5)),
                 e1=float(rng.uniform(-0.3, 0.3)), e2=float(rng.uniform(-0.3, 0.3)),
                 log_re=float(np.log(size * rng.uniform(0.25, 0.3125)))) for _ in range(20)]
    gals = _gals(rows)
    gp = [rng.normal(size=(size, size)) + 1.0 for _ in rows]
    gp = [g.astype(np.float32).astype(np.float64) for g in gp]
    got = gpu_grads_lanczos(gpu_renderer, gals, gp)
    want = oracle_grads_lanczos(gals, gpu_renderer.psfs, tables, gp)
    for k in (1, 2):
        err = np.abs(got[:, k] - want[:, k])
        assert np.all(err <= 3e-8 * gals.flux + 1e-6 * np.abs(want[:, k])), (k, err / gals.flux)
