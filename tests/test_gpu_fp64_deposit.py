"""FP64 deposit at the edges of its forms (grid points listed per trajectory, or steps walked in
order; steps divided over CTAs), against the oracle: few and many grid points per step, one
step, block edges, one pixel and tile remainders, electrons partly and wholly off the grid."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from gpu_cases import gpu_bounds, gpu_run, oracle_run  # noqa: E402
from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu


def _n_hat(n_pix, seed=3):
    rng = np.random.Generator(np.random.PCG64(seed))
    tx, ty = rng.uniform(-0.03, 0.03, n_pix), rng.uniform(-0.03, 0.03, n_pix)
    return np.stack([np.sin(tx), np.cos(tx) * np.sin(ty), np.cos(tx) * np.cos(ty)], -1)


def _compare(tr, n_hat, grid, **kw):
    got = gpu_run(tr, n_hat, grid, lw.LW_FP64, spectrum=False, **kw)
    want = oracle_run(tr, n_hat, grid, spectrum=False, **kw)
    scale = np.abs(want["rec"]).max()
    # the same contributions (bit-identical), added in another order: a few ulps of the largest
    assert np.abs(got["rec"] - want["rec"]).max() <= 1e-14 * scale
    assert got["status"] == want["status"]


@pytest.mark.parametrize("n_s", [1, 2, 255, 256, 257, 1000])
@pytest.mark.parametrize("bins_per_step", [0.02, 0.4, 0.6, 5.0])
def test_steps_and_density(n_s, bins_per_step):
    tr = simple.transverse_oscillation(3, n_s, 1e-17, 0.999, 0.01, 37.0)
    n_hat = _n_hat(130)
    lo, hi = gpu_bounds(tr, n_hat)
    n_bins = max(3, int(n_s * bins_per_step))
    _compare(tr, n_hat, lw.grid_from_bounds(lo - 0.01 * (hi - lo), hi + 0.01 * (hi - lo), n_bins))


@pytest.mark.parametrize("n_pix", [1, 31, 127, 128, 129])
@pytest.mark.parametrize("bins_per_step", [0.1, 3.0])
def test_pixel_tiles_velocity_field(n_pix, bins_per_step):
    tr = simple.transverse_oscillation(2, 600, 1e-17, 0.9995, 0.005, 51.0, seed=4)
    n_hat = _n_hat(n_pix, seed=n_pix)
    lo, hi = gpu_bounds(tr, n_hat)
    grid = lw.grid_from_bounds(lo, hi, int(600 * bins_per_step))
    _compare(tr, n_hat, grid, flags=oracle.FLAG_ACCEL | oracle.FLAG_VELOCITY, R=2.0)


@pytest.mark.parametrize("lo_f,hi_f", [(0.3, 0.6), (-2.0, 0.4), (0.7, 3.0), (0.999, 1.5)])
@pytest.mark.parametrize("bins_per_step", [0.1, 3.0])
def test_grid_covers_a_part(lo_f, hi_f, bins_per_step):
    tr = simple.transverse_oscillation(3, 500, 1e-17, 0.998, 0.02, 23.0, seed=9)
    n_hat = _n_hat(40)
    lo, hi = gpu_bounds(tr, n_hat)
    a, b = lo + lo_f * (hi - lo), lo + hi_f * (hi - lo)
    n_bins = max(2, int(500 * bins_per_step * (hi_f - lo_f)))
    _compare(tr, n_hat, lw.grid_from_bounds(a, b, n_bins))
