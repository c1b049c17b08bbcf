"""Small deposits of a bunch, far fewer grid points than steps.  Where the grid could hold as many per
step as the walk's lines say, what decides that costs next to nothing; few electrons' blocks are not
divided over CTAs.  Beside the same deposit with a view whose order stands elsewhere, which has no mean
advance and decides nothing."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu


def _times(n_e, n_s, n_pix, n_bins, prec, spread):
    """Shortest times [ms] of the deposit and of the one that decides nothing."""
    tr = simple.transverse_oscillation(n_e, n_s, 1e-17, 0.999, 0.002, 97.0, seed=n_e)
    # arrivals spread over many times an electron's own span
    own = n_s * 1e-17 * 1e-3
    shift = np.linspace(0.0, spread * own * 299792458.0, n_e)
    tr = simple.Trajectories(tr.t, tr.r - shift[:, None, None] * np.array([0.0, 0.0, 1.0]), tr.beta,
                             tr.beta_dot)
    rng = np.random.Generator(np.random.PCG64(1))
    tx, ty = rng.uniform(-0.02, 0.02, (2, n_pix))
    n_hat = np.stack([np.sin(tx), np.cos(tx) * np.sin(ty), np.cos(tx) * np.cos(ty)], -1)
    traj = lw.lw_trajectories_upload(tr.t, tr.r, tr.beta, tr.beta_dot, sections=lw.LW_SECTION_MIXED)
    view = lw.lw_traj.from_buffer_copy(traj.view)
    order = traj.order().clone()
    view.order = order.data_ptr()
    other = lw.Trajectories(traj.ws, view)
    det = lw.Detector(n_hat)
    grid = lw.grid_from_bounds(*lw.lw_grid_bounds(traj, det).cpu().tolist(), n_bins)
    shape, dtype = lw.record_shape(det, grid, prec)
    rec = torch.empty(shape, dtype=dtype, device="cuda")
    best = [float("inf")] * 2
    for rep in range(12):
        for n, view_of in enumerate((traj, other)):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(50):
                lw.lw_deposit_time_domain(view_of, det, grid, prec, record=rec)
            b.record()
            b.synchronize()
            if rep >= 2:
                best[n] = min(best[n], a.elapsed_time(b) / 50)
    print(best)
    return best


@pytest.mark.parametrize("n_e,n_s,n_pix,n_bins", [(226, 1855, 714, 9686), (926, 1523, 984, 7492),
                                                  (2900, 1050, 799, 4100)])
@pytest.mark.parametrize("prec", [lw.LW_MIXED, lw.LW_MIXED_F32, lw.LW_MIXED_F32X4])
def test_sparse_tiles_cost_no_launch(n_e, n_s, n_pix, n_bins, prec):
    chosen, undecided = _times(n_e, n_s, n_pix, n_bins, prec, 500)
    assert chosen <= 1.04 * undecided + 1e-3   # (a row of CTAs that end at once: 5 to 15 us)


def test_sparse_tiles_of_few_electrons():
    """209 electrons, whose blocks a denser tile's would be divided: 0.003 points per step."""
    chosen, divided = _times(209, 3239, 779, 25345, lw.LW_MIXED_F32, 3000)
    assert chosen <= 1.01 * divided + 1e-3
