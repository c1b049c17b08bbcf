"""FP64 adjoint at samples whose |beta|^2 lies within rounding of 1: the forward takes the field of a
sample as zero from the rounded sum (b_x^2 + b_y^2) + b_z^2 on, and the adjoint's gradient is zero
there and only there, whatever a fused sum would say."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from gpu_cases import gpu_bounds  # noqa: E402
from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu

libm = ctypes.CDLL("libm.so.6")
libm.fma.restype = ctypes.c_double
libm.fma.argtypes = [ctypes.c_double] * 3


def _luminal(count):
    """Velocities for which the rounded sum and the fused one fall on different sides of 1."""
    rng = np.random.Generator(np.random.PCG64(9))
    found = {True: [], False: []}
    while min(len(v) for v in found.values()) < count:
        b0, b1 = rng.uniform(-1e-2, 1e-2, 2).tolist()
        b2 = float(np.sqrt(1.0 - b0 * b0 - b1 * b1))
        for _ in range(4):
            plain = (b0 * b0 + b1 * b1) + b2 * b2 < 1.0
            fused = libm.fma(b2, b2, libm.fma(b1, b1, b0 * b0)) < 1.0
            if plain != fused:
                found[plain].append((b0, b1, b2))
            b2 = float(np.nextafter(b2, 0.0))
    return np.array(found[True][:count] + found[False][:count])


def test_gradient_is_zero_where_the_field_is():
    tr = simple.transverse_oscillation(2, 150, 1e-17, 0.999, 0.01, 37.0, seed=3)
    beta = tr.beta.copy()
    at = np.arange(20, 140, 6)
    beta[0, at] = _luminal(10)
    tx = np.linspace(0.02, 0.04, 33)
    n_hat = np.stack([np.sin(tx), np.zeros_like(tx), np.cos(tx)], -1)
    lo, hi = gpu_bounds(tr, n_hat)
    grid = lw.grid_from_bounds(lo, hi + 0.01 * (hi - lo), 256)
    g = np.random.Generator(np.random.PCG64(1)).standard_normal((33, 129))
    traj = lw.lw_trajectories_upload(tr.t, tr.r, beta, tr.beta_dot, sections=lw.LW_SECTION_FP64)
    det = lw.Detector(n_hat)
    rec = lw.lw_deposit_time_domain(traj, det, grid, lw.LW_FP64)
    _, X = lw.lw_spectrum(rec, lw.LW_FP64, 33, grid, want_X=True)
    got = [v.cpu().numpy() for v in lw.lw_spectrum_grad(traj, det, grid, X, torch.from_numpy(g).cuda())]
    want = oracle.tdm_grad(tr.t, tr.r, beta, tr.beta_dot, n_hat, grid.t_min, grid.dt_u,
                           grid.n_bins, g)
    for a, b in zip(got, want):
        # as the other adjoint tests: D = 1 - n.beta carries 1e-16 in 2e-4
        assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()
    assert not got[2][0, at[10:]].any() and got[2][0, at[:10]].all(-1).all()
