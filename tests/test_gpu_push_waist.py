"""GPU Boris push and its gradient in a wave of practically infinite waist, up to waists whose Rayleigh
length overflows, against the pusher written in torch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2206_03015_gb300 import lw  # noqa: E402
from paper_2206_03015_gb300.autograd import boris_push  # noqa: E402
from workloads.boris import gaussian_bunch  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w0", [1.0, 1e60, 1e100, 1e149, 1e151, 1e153, 1e155, 1e200, 1e300])
def test_push(w0):
    n_s, t0, dt = 60, -0.6e-15, 0.02e-15
    r0, u0 = gaussian_bunch(33, 5, 2e-6, 2e-6, 30e-6, 40.0, 1e-2, 0.5e-6, t0)
    r, u = torch.from_numpy(r0), torch.from_numpy(u0)
    a0, w = (torch.tensor(v, dtype=torch.float64) for v in (0.7, w0))
    want = boris_push(r, u, a0, w, 0.8e-6, 20e-15, t0, t0 + n_s * dt, n_s)
    got = [torch.empty(n_s + 1, dtype=torch.float64, device="cuda")]
    got += [torch.empty((33, n_s + 1, 3), dtype=torch.float64, device="cuda") for _ in range(3)]
    lw.lw_boris_push(r.cuda(), u.cuda(), t0, dt, n_s, (0.8e-6, 0.7, w0, 20e-15), *got)
    # a few roundings of 1.1e-16 per step; beta_dot's phase omega xi (at most 2.4e15 x 4e-13 rad)
    # carries its relative rounding as an absolute one, a few 1e-13
    for a, b, tol in zip(got[1:], want[1:], (1e-13, 1e-13, 1e-11)):
        assert float((a.cpu() - b).abs().max()) <= tol * float(b.abs().max())


@pytest.mark.parametrize("w0", [1.0, 1e60, 1e100, 1e149, 1e151, 1e155, 1e200])
def test_gradient_is_that_of_a_plane_wave(w0):
    """dL/du0 and dL/da0 as with a waist of 100 m, and no dependence on the waist."""
    n_s, t0, dt = 40, -0.4e-15, 0.02e-15
    r0, u0 = gaussian_bunch(33, 6, 2e-6, 2e-6, 30e-6, 40.0, 1e-2, 0.5e-6, t0)
    r, u = torch.from_numpy(r0).cuda(), torch.from_numpy(u0).cuda()
    g = torch.Generator().manual_seed(3)
    W = [torch.randn((33, n_s + 1, 3), dtype=torch.float64, generator=g).cuda() for _ in range(3)]
    du, dl = lw.lw_boris_push_grad(r, u, t0, dt, n_s, (0.8e-6, 0.7, w0, 20e-15), *W)
    dv, dm = lw.lw_boris_push_grad(r, u, t0, dt, n_s, (0.8e-6, 0.7, 100.0, 20e-15), *W)
    # rho^2/w0^2 is 1e-11 at 1 m; the phase z/zR = 1e-11 rad turns at most as much
    assert float((du - dv).norm()) <= 1e-9 * float(dv.norm())
    assert abs(float(dl[0] - dm[0])) <= 1e-9 * abs(float(dm[0]))
    assert np.isfinite(float(dl[1])) and abs(float(dl[1])) <= 1e-9 * abs(float(dm[0])) / w0
