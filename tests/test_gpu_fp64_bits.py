"""FP64 contributions are the oracle's to the bit: one electron has one contribution per bin, so no
order of additions enters.  Fields of ordinary size, of 1e-310 to 1e-270 (where the residual of a
shared reciprocal is no longer exact), and zero."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from gpu_cases import gpu_bounds, gpu_run, oracle_run  # noqa: E402
from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-290, 1e-300, 1e-308, 1e-318, 1e-330, 0.0])
@pytest.mark.parametrize("bins_per_step", [0.05, 2.5])
@pytest.mark.parametrize("flags", [oracle.FLAG_ACCEL, oracle.FLAG_ACCEL | oracle.FLAG_VELOCITY])
def test_contributions(scale, bins_per_step, flags):
    tr = simple.transverse_oscillation(1, 900, 1e-17, 0.999, 0.01, 37.0, seed=7)
    # beta_dot of about 1e15 at scale 1
    tr = simple.Trajectories(tr.t, tr.r, tr.beta, tr.beta_dot * scale)
    rng = np.random.Generator(np.random.PCG64(5))
    tx, ty = rng.uniform(-0.03, 0.03, 200), rng.uniform(-0.03, 0.03, 200)
    n_hat = np.stack([np.sin(tx), np.cos(tx) * np.sin(ty), np.cos(tx) * np.cos(ty)], -1)
    lo, hi = gpu_bounds(tr, n_hat)
    grid = lw.grid_from_bounds(lo, hi + 0.02 * (hi - lo), int(900 * bins_per_step))
    got = gpu_run(tr, n_hat, grid, lw.LW_FP64, spectrum=False, flags=flags)
    want = oracle_run(tr, n_hat, grid, spectrum=False, flags=flags)
    assert np.array_equal(got["rec"], want["rec"])
    assert got["status"] == want["status"]
