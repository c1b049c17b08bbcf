"""Which way a tile of the mixed deposit is taken, and that it does not matter: the walk of dense
tiles and the search add the same contributions, to the bit (a record of one electron has one
contribution per bin, so no order of additions enters)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import configs, simple  # noqa: E402

pytestmark = pytest.mark.gpu


def _n_hat(n_pix, lo=-0.03, hi=0.03):
    rng = np.random.Generator(np.random.PCG64(n_pix))
    tx, ty = rng.uniform(lo, hi, n_pix), rng.uniform(lo, hi, n_pix)
    return np.stack([np.sin(tx), np.cos(tx) * np.sin(ty), np.cos(tx) * np.cos(ty)], -1)


def _grid(traj, det, n_bins):
    lo, hi = lw.lw_grid_bounds(traj, det).cpu().tolist()
    return lw.grid_from_bounds(lo, hi + 0.02 * (hi - lo), n_bins)


def _searched(traj):
    """The same trajectories as a view whose order (the same one) stands elsewhere, so that it has no
    mean advance: its tiles are all searched."""
    view = lw.lw_traj.from_buffer_copy(traj.view)
    order = traj.order().clone()
    view.order = order.data_ptr()
    out = lw.Trajectories(traj.ws, view)
    out._keep = order, getattr(traj, "_inputs", None)
    return out


def _deposit(traj, det, grid, prec, flags=lw.LW_FIELD_ACCEL):
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rec = lw.lw_deposit_time_domain(traj, det, grid, prec, flags, status=status)
    return rec, int(status.item())


@pytest.mark.parametrize("prec", [lw.LW_MIXED, lw.LW_MIXED_KAHAN, lw.LW_MIXED_F32,
                                  lw.LW_MIXED_F32X4])
@pytest.mark.parametrize("flags", [1, 2, 3])
@pytest.mark.parametrize("n_s,per_step,block", [(300, 6.0, 64), (1100, 4.5, 512), (37, 9.0, 16)])
def test_walk_and_search_agree_to_the_bit(prec, flags, n_s, per_step, block):
    tr = simple.transverse_oscillation(1, n_s, 1e-17, 0.999, 0.01, 97.0, seed=n_s)
    traj = lw.lw_trajectories_upload(tr.t, tr.r, tr.beta, tr.beta_dot, block=block)
    det = lw.Detector(_n_hat(259), R=1.5)
    grid = _grid(traj, det, int(n_s * per_step))
    walked, st_w = _deposit(traj, det, grid, prec, flags)
    searched, st_s = _deposit(_searched(traj), det, grid, prec, flags)
    assert torch.equal(walked, searched) and st_w == st_s
    assert walked.abs().max() > 0


def _irregular(kind, n_e=1, n_s=600):
    """Trajectories that the upload flags, from sample 250 of electron 0 on: a superluminal step (the
    advanced time goes back by about 20 steps), a step backwards longer than c0 dt (over the rest
    of the grid), a repeated sample, a sample whose time goes back, one
    that is not finite."""
    tr = simple.transverse_oscillation(n_e, n_s, 1e-17, 0.999, 0.01, 97.0, seed=6)
    t, r = np.tile(tr.t, (n_e, 1)), tr.r.copy()
    if kind == "back":
        r[0, 250:, 2] += 9e-11
    elif kind == "ahead":
        r[0, 250:, 2] -= 6.2e-9
    elif kind == "repeat":
        t[0, 250], r[0, 250] = t[0, 249], r[0, 249]
    elif kind == "time":
        t[0, 250] -= 2.5e-17
    else:
        r[0, 250, 0] = np.nan
    return simple.Trajectories(t, r, tr.beta, tr.beta_dot)


@pytest.mark.parametrize("prec", [lw.LW_MIXED, lw.LW_MIXED_F32, lw.LW_MIXED_F32X4])
@pytest.mark.parametrize("kind", ["back", "ahead", "repeat", "time", "nan"])
def test_irregular_inputs_are_searched(prec, kind):
    """Dense tiles of inputs that the upload flags: the record and the status of the search, also
    where the coordinate goes back within a block."""
    clean = simple.transverse_oscillation(1, 600, 1e-17, 0.999, 0.01, 97.0, seed=6)
    det = lw.Detector(_n_hat(70))
    grid = _grid(lw.lw_trajectories_upload(clean.t, clean.r, clean.beta, clean.beta_dot), det, 3000)
    tr = _irregular(kind)
    traj = lw.lw_trajectories_upload(tr.t, tr.r, tr.beta, tr.beta_dot, block=512)
    got, st = _deposit(traj, det, grid, prec)
    want, st_s = _deposit(_searched(traj), det, grid, prec)
    assert st == st_s and st & (lw.LW_ST_STEP | lw.LW_ST_TIME | lw.LW_ST_NONFINITE)
    assert torch.equal(got, want) and bool(torch.isfinite(got).all()) and got.abs().max() > 0


def _span(traj):
    """The mean advance that the upload stores behind the order: after two keys and 4,096 counters."""
    at = traj.view.order + (4 * traj.n_e + 255) // 256 * 256 + 16 + 4 * 4096 - traj.ws.data_ptr()
    return traj.ws[at:at + 32].view(torch.float64)


def _per_step(traj, n_hat, grid):
    """Grid points per step of the mean advance, averaged over the pixels of each tile of 512."""
    span = _span(traj).cpu().numpy()
    adv = span[0] - (n_hat[:, 0] * span[1] + n_hat[:, 1] * span[2]
                     - (1.0 - n_hat[:, 2]) * span[3]) / 299792458.0
    return [float(adv[k:k + 512].mean()) / (grid.dt_u * traj.n_s) for k in range(0, len(adv), 512)]


def _ms(*calls):
    """Shortest of nine runs of each call, in turn, by events on the stream."""
    best = [float("inf")] * len(calls)
    for rep in range(11):
        for n, call in enumerate(calls):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            call()
            b.record()
            b.synchronize()
            if rep >= 2:
                best[n] = min(best[n], a.elapsed_time(b))
    return best


def test_dense_tiles_are_walked():
    """Pixels from the axis outwards: 1 - n.beta grows with the angle, and with it the grid points
    per step of the three tiles (0.9, 1.6 and 3).  The first is searched, the others are walked:
    seen by the time, which is longer when the stored mean advance says that no tile is dense (1.5, 3
    points per step take about 0.6 and 0.5 of the search's time walked), and about the same as
    that when the view's order stands elsewhere."""
    tr = simple.transverse_oscillation(512, 3000, 1e-17, 0.999, 0.002, 97.0, seed=8)
    th = np.linspace(0.0, 0.09, 1536)
    n_hat = np.stack([np.sin(th), np.zeros_like(th), np.cos(th)], -1)
    traj = lw.lw_trajectories_upload(tr.t, tr.r, tr.beta, tr.beta_dot)
    det = lw.Detector(n_hat)
    grid = _grid(traj, det, 12300)
    assert [v > 1.3 for v in _per_step(traj, n_hat, grid)] == [False, True, True]
    first, _ = _deposit(traj, det, grid, lw.LW_MIXED_F32X4)
    other = _searched(traj)
    walked, moved = _ms(lambda: _deposit(traj, det, grid, lw.LW_MIXED_F32X4),
                        lambda: _deposit(other, det, grid, lw.LW_MIXED_F32X4))
    _span(traj).zero_()
    assert _per_step(traj, n_hat, grid) == [0.0, 0.0, 0.0]
    (searched,) = _ms(lambda: _deposit(traj, det, grid, lw.LW_MIXED_F32X4))
    print(walked, moved, searched)
    assert walked < 0.8 * searched and walked < 0.8 * moved
    rec, _ = _deposit(traj, det, grid, lw.LW_MIXED_F32X4)
    # FP32 additions of the same contributions in two orders; a tile deposited twice or not at all
    # is an error of order one
    assert (first - rec).abs().max() <= 1e-3 * rec.abs().max()


@pytest.mark.parametrize("prec,per_step", [(lw.LW_MIXED_F32X4, 1.1), (lw.LW_MIXED_F32, 1.5),
                                           (lw.LW_MIXED, 1.9), (lw.LW_MIXED_KAHAN, 4.3),
                                           (lw.LW_MIXED_KAHAN, 8.0)])
def test_a_bunch_is_not_slower_than_by_search(prec, per_step):
    """Electrons of a bunch, each over its own part of the grid, just above the lines and beyond (grid
    points per step, averaged over the 256 pixels)."""
    w = configs.c2x(n_e=400, n_s=6000, nx=16, n_bins=1 << 12)
    traj = lw.lw_trajectories_upload(w.traj.t, w.traj.r, w.traj.beta, w.traj.beta_dot)
    other = _searched(traj)
    det = lw.Detector(w.n_hat)
    lo, hi = lw.lw_grid_bounds(traj, det).cpu().tolist()
    grid = lw.grid_from_bounds(lo, hi, 1 << 16)
    (had,) = _per_step(traj, w.n_hat, grid)
    grid = lw.grid_from_bounds(lo, hi, int(per_step / had * (1 << 16)))
    chosen, searched = _ms(lambda: lw.lw_deposit_time_domain(traj, det, grid, prec),
                           lambda: lw.lw_deposit_time_domain(other, det, grid, prec))
    print(chosen, searched)
    assert chosen <= 1.04 * searched
