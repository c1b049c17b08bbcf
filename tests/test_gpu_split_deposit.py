"""Mixed deposit of few electrons and pixels, whose blocks of samples are divided over CTAs: part
boundaries inside and at anchor batches (32 blocks), more parts than blocks, single blocks, pixel
tiles with remainders, against the oracle bin by bin (a grid point dropped or taken twice at a
boundary is an error of order one in its bin)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_cases import gpu_bounds, gpu_run, oracle_run  # noqa: E402
from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu


def _compare(n_e, n_s, n_pix, block, bins_per_step, prec):
    tr = simple.transverse_oscillation(n_e, n_s, 1e-17, 0.999, 0.01, 97.0, seed=n_s)
    rng = np.random.Generator(np.random.PCG64(n_pix))
    tx, ty = rng.uniform(-0.03, 0.03, n_pix), rng.uniform(-0.03, 0.03, n_pix)
    n_hat = np.stack([np.sin(tx), np.cos(tx) * np.sin(ty), np.cos(tx) * np.cos(ty)], -1)
    lo, hi = gpu_bounds(tr, n_hat)
    grid = lw.grid_from_bounds(lo, hi + 0.02 * (hi - lo), max(4, int(n_s * bins_per_step)))
    got = gpu_run(tr, n_hat, grid, prec, spectrum=False, block=block)
    want = oracle_run(tr, n_hat, grid, spectrum=False)
    # the mixed path's bound on this family of trajectories (97 samples per period: the field
    # changes by 7 % of its maximum across a step at most)
    assert np.abs(got["rec"] - want["rec"]).max() <= 1e-4 * np.abs(want["rec"]).max()
    assert got["status"] == want["status"]


@pytest.mark.parametrize("blocks", [1, 2, 31, 32, 33, 64, 70])
@pytest.mark.parametrize("prec", [lw.LW_MIXED, lw.LW_MIXED_KAHAN, lw.LW_MIXED_F32X4])
def test_part_boundaries(blocks, prec):
    _compare(2, 16 * blocks, 5, 16, 0.7, prec)
    _compare(1, 16 * blocks + 1, 3, 16, 3.0, prec)


@pytest.mark.parametrize("n_pix", [1, 255, 256, 257, 513])
@pytest.mark.parametrize("n_e", [1, 3])
def test_tiles(n_pix, n_e):
    _compare(n_e, 300, n_pix, 64, 0.5, lw.LW_MIXED_F32)
