"""Mixed deposit of dense grids (from about one grid point per step on), whose blocks are walked
sample by sample, at the edges of the walk: densities on both sides of its threshold, segments of
32 samples with remainders, more grid points per segment than its map holds (256), one block and
several, electrons of very different densities in one launch, pixel tiles on both sides of the
threshold, grids that cover a part of the trajectory, every record and both field terms, against
the oracle bin by bin."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from gpu_cases import gpu_bounds, gpu_run, oracle_run, record_value  # noqa: E402
from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu


def _compare(tr, n_pix, grid_of, prec, block=512, **kw):
    rng = np.random.Generator(np.random.PCG64(n_pix))
    tx, ty = rng.uniform(-0.03, 0.03, n_pix), rng.uniform(-0.03, 0.03, n_pix)
    n_hat = np.stack([np.sin(tx), np.cos(tx) * np.sin(ty), np.cos(tx) * np.cos(ty)], -1)
    grid = grid_of(*gpu_bounds(tr, n_hat))
    got = gpu_run(tr, n_hat, grid, prec, spectrum=False, block=block, **kw)
    want = oracle_run(tr, n_hat, grid, spectrum=False, **kw)
    # the mixed path's bound on this family (97 samples per period); a grid point dropped or taken
    # twice is an error of order one in its bin
    assert np.abs(got["rec"] - want["rec"]).max() <= 1e-4 * np.abs(want["rec"]).max()
    assert got["status"] == want["status"]


def _whole(n_bins):
    return lambda lo, hi: lw.grid_from_bounds(lo, hi + 0.02 * (hi - lo), n_bins)


@pytest.mark.parametrize("n_s", [1, 31, 32, 33, 511, 512, 513, 1100])
@pytest.mark.parametrize("per_step", [0.4, 0.5, 0.95, 1.05, 3.3, 12.0])
def test_steps_and_density(n_s, per_step):
    tr = simple.transverse_oscillation(2, n_s, 1e-17, 0.999, 0.01, 97.0, seed=n_s)
    _compare(tr, 3, _whole(max(4, int(n_s * per_step))), lw.LW_MIXED_F32X4)


@pytest.mark.parametrize("block", [16, 32, 64, 1024])
def test_blocks(block):
    tr = simple.transverse_oscillation(1, 1500, 1e-17, 0.999, 0.01, 97.0)
    _compare(tr, 2, _whole(4500), lw.LW_MIXED, block=block)


@pytest.mark.parametrize("prec", [lw.LW_MIXED, lw.LW_MIXED_KAHAN, lw.LW_MIXED_F32,
                                  lw.LW_MIXED_F32X4])
@pytest.mark.parametrize("flags", [oracle.FLAG_ACCEL, oracle.FLAG_VELOCITY,
                                   oracle.FLAG_ACCEL | oracle.FLAG_VELOCITY])
def test_records_and_fields(prec, flags):
    tr = simple.transverse_oscillation(3, 300, 1e-17, 0.999, 0.01, 97.0, seed=3)
    _compare(tr, 259, _whole(700), prec, flags=flags, R=1.5)


@pytest.mark.parametrize("lo_f,hi_f", [(0.3, 0.31), (-1.0, 0.5), (0.6, 2.0)])
def test_grid_covers_a_part(lo_f, hi_f):
    tr = simple.transverse_oscillation(2, 700, 1e-17, 0.999, 0.01, 97.0, seed=5)
    n_bins = max(400, int(2000 * (hi_f - lo_f)))
    _compare(tr, 5, lambda lo, hi: lw.grid_from_bounds(lo + lo_f * (hi - lo),
                                                       lo + hi_f * (hi - lo), n_bins),
             lw.LW_MIXED_F32)


def test_dense_and_sparse_electrons():
    """Electrons of 40 different speeds, whose advanced time's rate differs sixfold."""
    parts = [simple.transverse_oscillation(1, 400, 1e-17, b, 0.003, 97.0, seed=k)
             for k, b in enumerate(np.linspace(0.997, 0.9995, 40))]
    tr = simple.Trajectories(parts[0].t, *[np.concatenate([getattr(p, n) for p in parts])
                                           for n in ("r", "beta", "beta_dot")])
    _compare(tr, 6, _whole(300), lw.LW_MIXED_F32X4, block=64)


def test_tiles_on_both_sides_of_the_threshold():
    """1,100 pixels from the axis outwards: the rate of the advanced time, 1 - n.beta, grows with the
    angle, so that the first tiles of 512 pixels are searched and the last is walked."""
    tr = simple.transverse_oscillation(2, 300, 1e-17, 0.999, 0.002, 97.0, seed=8)
    th = np.linspace(0.0, 0.09, 1100)
    n_hat = np.stack([np.sin(th), np.zeros_like(th), np.cos(th)], -1)
    lo, hi = gpu_bounds(tr, n_hat)
    grid = lw.grid_from_bounds(lo, hi + 0.02 * (hi - lo), 300)
    got = gpu_run(tr, n_hat, grid, lw.LW_MIXED_F32X4, spectrum=False)
    want = oracle_run(tr, n_hat, grid, spectrum=False)
    assert np.abs(got["rec"] - want["rec"]).max() <= 1e-4 * np.abs(want["rec"]).max()
    assert got["status"] == want["status"]


@pytest.mark.parametrize("prec", [lw.LW_MIXED, lw.LW_MIXED_KAHAN, lw.LW_MIXED_F32])
@pytest.mark.parametrize("per_step", [1.35, 1.45, 1.75, 1.85, 3.9, 4.2, 7.0])
def test_density_of_each_record(prec, per_step):
    tr = simple.transverse_oscillation(2, 300, 1e-17, 0.999, 0.01, 97.0, seed=9)
    _compare(tr, 3, _whole(int(300 * per_step * 1.02)), prec)


def test_view_with_another_order():
    """A view whose order was taken out, or stands elsewhere, has no mean advance to decide by: its
    dense tiles are searched and its record is the same."""
    tr = simple.transverse_oscillation(3, 400, 1e-17, 0.999, 0.01, 97.0, seed=4)
    n_hat = np.array([[0.0, 0.0, 1.0], [0.01, 0.0, np.sqrt(1 - 1e-4)]])
    grid = _whole(900)(*gpu_bounds(tr, n_hat))
    want = oracle_run(tr, n_hat, grid, spectrum=False)["rec"]
    traj = lw.lw_trajectories_upload(tr.t, tr.r, tr.beta, tr.beta_dot)
    own = traj.order().clone()
    det = lw.Detector(n_hat)
    for order in (traj.view.order, None, own.data_ptr()):
        traj.view.order = order
        got = record_value(lw.lw_deposit_time_domain(traj, det, grid, lw.LW_MIXED), lw.LW_MIXED)
        assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()
