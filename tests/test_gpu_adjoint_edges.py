"""FP64 adjoint where its work is cut: sample tiles of 64 divided over CTAs, 32-pixel warp sums and
128-pixel tiles with remainders, steps with none, one or many grid points, grids that cover a part
of the trajectory, against the oracle's chain-rule gradient."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from gpu_cases import gpu_bounds  # noqa: E402
from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu


def _case(n_e, n_s, n_pix, bins, lo_f=-0.01, hi_f=1.01):
    tr = simple.transverse_oscillation(n_e, n_s, 1e-17, 0.999, 0.01, 37.0, seed=n_s)
    rng = np.random.Generator(np.random.PCG64(n_pix))
    tx, ty = rng.uniform(-0.03, 0.03, n_pix), rng.uniform(-0.03, 0.03, n_pix)
    n_hat = np.stack([np.sin(tx), np.cos(tx) * np.sin(ty), np.cos(tx) * np.cos(ty)], -1)
    lo, hi = gpu_bounds(tr, n_hat)
    return tr, n_hat, lw.grid_from_bounds(lo + lo_f * (hi - lo), lo + hi_f * (hi - lo), bins)


@pytest.mark.parametrize("n_e,n_s,n_pix,bins,lo_f,hi_f", [
    (1, 1, 1, 2, -0.01, 1.01), (2, 63, 3, 16, -0.01, 1.01), (1, 64, 33, 256, -0.01, 1.01),
    (2, 65, 5, 64, -0.01, 1.01), (1, 128, 129, 32, -0.01, 1.01), (1, 200, 31, 512, 0.4, 0.6),
    (2, 150, 7, 64, -1.0, 0.5)])
def test_fp64_adjoint_against_oracle(n_e, n_s, n_pix, bins, lo_f, hi_f):
    tr, n_hat, grid = _case(n_e, n_s, n_pix, bins, lo_f, hi_f)
    rng = np.random.Generator(np.random.PCG64(1))
    g = rng.standard_normal((n_pix, bins // 2 + 1))
    traj = lw.lw_trajectories_upload(tr.t, tr.r, tr.beta, tr.beta_dot, sections=lw.LW_SECTION_FP64)
    det = lw.Detector(n_hat)
    rec = lw.lw_deposit_time_domain(traj, det, grid, lw.LW_FP64)
    _, X = lw.lw_spectrum(rec, lw.LW_FP64, n_pix, grid, want_X=True)
    got = lw.lw_spectrum_grad(traj, det, grid, X, torch.from_numpy(g).cuda())
    want = oracle.tdm_grad(tr.t, tr.r, tr.beta, tr.beta_dot, n_hat, grid.t_min, grid.dt_u,
                           grid.n_bins, g)
    for a, b in zip(got, want):
        # as the element-wise bound of the other adjoint tests: D = 1 - n.beta carries 1e-16 in
        # 1e-3, the record's transforms and their products a few more
        assert np.abs(a.cpu().numpy() - b).max() <= 1e-9 * np.abs(b).max()


@pytest.mark.parametrize("n_e,n_s,n_pix,bins,lo_f,hi_f", [
    (1, 1, 1, 2, -0.01, 1.01), (2, 63, 3, 16, -0.01, 1.01), (1, 64, 33, 256, -0.01, 1.01),
    (3, 65, 5, 64, -0.01, 1.01), (1, 128, 129, 32, -0.01, 1.01), (1, 200, 31, 512, 0.4, 0.6),
    (2, 150, 7, 64, -1.0, 0.5), (1, 130, 2, 4096, -0.01, 1.01)])
def test_mixed_adjoint_against_fp64(n_e, n_s, n_pix, bins, lo_f, hi_f):
    """The mixed adjoint at its own cuts (tiles of 64 samples with the sample before, groups of four
    bins, the last sample) against the FP64 adjoint of the same X', element by element."""
    tr, n_hat, grid = _case(n_e, n_s, n_pix, bins, lo_f, hi_f)
    g = np.random.Generator(np.random.PCG64(2)).standard_normal((n_pix, bins // 2 + 1))
    g = torch.from_numpy(g).cuda()
    traj = lw.lw_trajectories_upload(tr.t, tr.r, tr.beta, tr.beta_dot)
    det = lw.Detector(n_hat)
    rec = lw.lw_deposit_time_domain(traj, det, grid, lw.LW_FP64)
    _, X = lw.lw_spectrum(rec, lw.LW_FP64, n_pix, grid, want_X=True)
    want = lw.lw_spectrum_grad(traj, det, grid, X, g)
    got = lw.lw_spectrum_grad(traj, det, grid, X.to(torch.complex64), g)
    for a, b in zip(got, want):
        # the bound of the mixed adjoint's comparison with the oracle
        assert float((a - b).abs().max()) <= 1e-4 * float(b.abs().max())
