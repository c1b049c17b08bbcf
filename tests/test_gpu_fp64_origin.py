"""FP64 deposit of a bunch away from the coordinates' origin: the search's FP32 terms of n . r round
to more than a step there, and a search in FP64 takes over.  Records against the oracle, and the time
beside that at the origin (walking from where the FP32 search landed took hundreds of steps per
grid point)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_cases import gpu_bounds, gpu_run, oracle_run  # noqa: E402
from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu

SHIFTS = [(0.0, 0.0, 10.0), (1.0, 0.0, 0.0), (0.3, -2.0, 30.0)]


def _shifted(tr, d):
    return simple.Trajectories(tr.t, tr.r + np.array(d), tr.beta, tr.beta_dot)


def _n_hat(n_pix):
    """Directions 1e-10 rad apart around 25 mrad, so that a shift moves all arrivals alike."""
    tx = 0.025 + 1e-10 * np.arange(n_pix)
    return np.stack([np.sin(tx), np.zeros(n_pix), np.cos(tx)], -1)


@pytest.mark.parametrize("shift", SHIFTS)
@pytest.mark.parametrize("n_s,n_bins", [(2, 1), (700, 3), (700, 40), (700, 300), (4001, 25)])
def test_record(shift, n_s, n_bins):
    tr = _shifted(simple.transverse_oscillation(3, n_s, 1e-17, 0.999, 0.01, 37.0, seed=2), shift)
    n_hat = _n_hat(131)
    lo, hi = gpu_bounds(tr, n_hat)
    grid = lw.grid_from_bounds(lo, hi, n_bins)
    got = gpu_run(tr, n_hat, grid, lw.LW_FP64, spectrum=False)
    want = oracle_run(tr, n_hat, grid, spectrum=False)
    # the same contributions (bit-identical), added in another order: a few ulps of the largest
    assert np.abs(got["rec"] - want["rec"]).max() <= 1e-14 * np.abs(want["rec"]).max()
    assert got["status"] == want["status"]


@pytest.mark.parametrize("shift", SHIFTS)
def test_time(shift):
    tr = simple.transverse_oscillation(400, 5000, 1e-17, 0.999, 0.002, 97.0, seed=4)
    det = lw.Detector(_n_hat(256))
    best = []
    for case in (tr, _shifted(tr, shift)):
        traj = lw.lw_trajectories_upload(case.t, case.r, case.beta, case.beta_dot,
                                         sections=lw.LW_SECTION_FP64)
        grid = lw.grid_from_bounds(*lw.lw_grid_bounds(traj, det).cpu().tolist(), 25)
        rec = lw.lw_deposit_time_domain(traj, det, grid, lw.LW_FP64)
        times = []
        for _ in range(9):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            lw.lw_deposit_time_domain(traj, det, grid, lw.LW_FP64, record=rec)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        best.append(min(times))
    print(best)
    assert best[1] <= 3.0 * best[0]
