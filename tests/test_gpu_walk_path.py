"""Which launch deposits a tile of the mixed deposit, and that it does not matter: the walk of dense
tiles and the search add the same contributions, to the bit (a record of one electron has one
contribution per bin, so no order of additions enters)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu


def _n_hat(n_pix, lo=-0.03, hi=0.03):
    rng = np.random.Generator(np.random.PCG64(n_pix))
    tx, ty = rng.uniform(lo, hi, n_pix), rng.uniform(lo, hi, n_pix)
    return np.stack([np.sin(tx), np.cos(tx) * np.sin(ty), np.cos(tx) * np.cos(ty)], -1)


def _grid(traj, det, n_bins):
    lo, hi = lw.lw_grid_bounds(traj, det).cpu().tolist()
    return lw.grid_from_bounds(lo, hi + 0.02 * (hi - lo), n_bins)


def _searched(traj):
    """The same trajectories as a view without the upload's order, whose tiles are all searched."""
    view = lw.lw_traj.from_buffer_copy(traj.view)
    view.order = None
    out = lw.Trajectories(traj.ws, view)
    out._inputs = getattr(traj, "_inputs", None)
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


def _span(traj):
    """The mean advance that the upload stores behind the order: after two keys and 4,096 counters."""
    at = traj.view.order + (4 * traj.n_e + 255) // 256 * 256 + 16 + 4 * 4096 - traj.ws.data_ptr()
    return traj.ws[at:at + 32].view(torch.float64).cpu().numpy()


def _dense(traj, n_hat, grid, line):
    """Per tile of 512 pixels: whether its middle pixel's mean advance is above the line."""
    span = _span(traj)
    mid = n_hat[np.minimum(np.arange(0, len(n_hat), 512) + 256, len(n_hat) - 1)]
    adv = span[0] - (mid[:, 0] * span[1] + mid[:, 1] * span[2]
                     - (1.0 - mid[:, 2]) * span[3]) / 299792458.0
    return adv / grid.dt_u > line * traj.n_s


def _kernel_us(call):
    """Device time of the walk's and of the search's launches in one call [us]."""
    from torch.profiler import ProfilerActivity, profile
    call()
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    seen = {e.key: e.self_device_time_total for e in prof.key_averages()}
    if not any("deposit_mixed_kernel" in k for k in seen):
        pytest.skip("no trace of the launches here")
    return [sum(v for k, v in seen.items() if name in k)
            for name in ("deposit_walk_kernel", "deposit_mixed_kernel")]


def test_each_tile_has_one_launch():
    """Pixels from the axis outwards: 1 - n.beta grows with the angle, so that with this grid the
    first tiles are searched, the last is walked, and both launches have work; with eight times
    the bins all are walked and the search's CTAs end at once; without the order there is no walk."""
    tr = simple.transverse_oscillation(256, 3000, 1e-17, 0.999, 0.002, 97.0, seed=8)
    th = np.linspace(0.0, 0.09, 1536)
    n_hat = np.stack([np.sin(th), np.zeros_like(th), np.cos(th)], -1)
    traj = lw.lw_trajectories_upload(tr.t, tr.r, tr.beta, tr.beta_dot)
    det = lw.Detector(n_hat)
    grid = _grid(traj, det, 6120)
    fine = lw.Grid(grid.t_min, grid.dt_u / 8.0, grid.n_bins * 8)
    prec = lw.LW_MIXED_F32X4
    some, all_ = _dense(traj, n_hat, grid, 1.0), _dense(traj, n_hat, fine, 1.0)
    assert not some[0] and some[-1] and all_.all()
    walk_some, search_some = _kernel_us(lambda: _deposit(traj, det, grid, prec))
    walk_all, search_all = _kernel_us(lambda: _deposit(traj, det, fine, prec))
    walk_none, search_none = _kernel_us(lambda: _deposit(_searched(traj), det, grid, prec))
    assert walk_none == 0 and search_none > search_some > 3 * search_all
    assert walk_all > 3 * search_all and walk_some > 3 * search_all
