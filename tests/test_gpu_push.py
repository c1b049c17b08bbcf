"""GPU Boris push and its gradient at the edges of their electron groups (32 per CTA) and step
counts: the push against the numpy pusher of the workloads, and split into blocks against one
call; the gradient against torch autograd through the torch-written pusher."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads.boris import GaussianLaser, boris_trajectories, gaussian_bunch  # noqa: E402

pytestmark = pytest.mark.gpu

LASER = GaussianLaser(lam=0.8e-6, a0=0.7, w0=6e-6, fwhm=20e-15)
L = (LASER.lam, LASER.a0, LASER.w0, LASER.fwhm)


def _start(n_e, n_s):
    # steps of 0.02 fs around the pulse's peak; a waist of a few bunch radii and z of a sizeable
    # part of the Rayleigh length, so that every factor of the beam matters
    t0 = -0.01e-15 * n_s
    r0, u0 = gaussian_bunch(n_e, 11 + n_e, 2e-6, 2e-6, 30e-6, 40.0, 1e-2, 0.5e-6, t0)
    return r0, u0, t0, 0.02e-15


def _push(r0, u0, t0, dt, n_s, step0=0):
    n_e = r0.shape[0]
    t = torch.empty(n_s + 1, dtype=torch.float64, device="cuda")
    out = [torch.empty((n_e, n_s + 1, 3), dtype=torch.float64, device="cuda") for _ in range(3)]
    lw.lw_boris_push(r0, u0, t0, dt, n_s, L, t, *out, step0=step0)
    return [t] + out


@pytest.mark.parametrize("n_e", [1, 31, 32, 33, 65])
@pytest.mark.parametrize("n_s", [1, 2, 41])
def test_push_matches_numpy(n_e, n_s):
    r0, u0, t0, dt = _start(n_e, n_s)
    ref = boris_trajectories(r0, u0, LASER, t0, t0 + n_s * dt, n_s)
    r, u = torch.from_numpy(r0).cuda(), torch.from_numpy(u0).cuda()
    t, R, B, A = (x.cpu().numpy() for x in _push(r, u, t0, dt, n_s))
    # a few roundings of 1.1e-16 per step on r and beta; beta_dot's phase omega xi (at most
    # 2.4e15 x 4e-13 rad) carries its relative rounding as an absolute one, a few 1e-13
    assert np.abs(t - ref.t).max() <= 1e-30
    assert np.abs(R - ref.r).max() <= 1e-13 * np.abs(ref.r).max()
    assert np.abs(B - ref.beta).max() <= 1e-13
    assert np.abs(A - ref.beta_dot).max() <= 1e-11 * np.abs(ref.beta_dot).max()
    assert np.abs(r.cpu().numpy() - R[:, -1]).max() == 0.0
    # u = gamma beta: beta carries 1e-16, times gamma^2 through 1/sqrt(1 - beta^2)
    g = 1.0 / np.sqrt(1.0 - (B[:, -1] ** 2).sum(-1, keepdims=True))
    assert np.abs(u.cpu().numpy() - g * B[:, -1]).max() <= 1e-11 * np.abs(u0).max()


@pytest.mark.parametrize("n_e,cuts", [(33, (1, 7, 40)), (5, (39, 40))])
def test_push_in_blocks_is_bit_identical(n_e, cuts):
    n_s = 40
    r0, u0, t0, dt = _start(n_e, n_s)
    whole = _push(torch.from_numpy(r0).cuda(), torch.from_numpy(u0).cuda(), t0, dt, n_s)
    r, u = torch.from_numpy(r0).cuda(), torch.from_numpy(u0).cuda()
    lo = 0
    for hi in cuts:
        t, R, B, A = _push(r, u, t0, dt, hi - lo, step0=lo)
        assert torch.equal(t, whole[0][lo:hi + 1])
        for a, b in zip((R, B, A), whole[1:]):
            assert torch.equal(a, b[:, lo:hi + 1])
        lo = hi


@pytest.mark.parametrize("n_e", [1, 32, 33])
@pytest.mark.parametrize("n_s", [1, 2, 3, 40])
def test_push_gradient_matches_autograd(n_e, n_s):
    from paper_2206_03015_gb300.autograd import boris_push
    r0, u0, t0, dt = _start(n_e, n_s)
    g = torch.Generator().manual_seed(n_e * 100 + n_s)
    r = torch.from_numpy(r0)
    u = torch.from_numpy(u0).requires_grad_(True)
    a0 = torch.tensor(LASER.a0, dtype=torch.float64, requires_grad=True)
    w0 = torch.tensor(LASER.w0, dtype=torch.float64, requires_grad=True)
    t, R, B, A = boris_push(r, u, a0, w0, LASER.lam, LASER.fwhm, t0, t0 + n_s * dt, n_s)
    # every sample's position, velocity and acceleration weighted alike
    W = [torch.randn(x.shape, dtype=torch.float64, generator=g) / float(x.detach().abs().max())
         for x in (R, B, A)]
    sum((w * x).sum() for w, x in zip(W, (R, B, A))).backward()
    du, dl = lw.lw_boris_push_grad(r.cuda(), u.detach().cuda(), t0, dt, n_s, L,
                                   *[w.cuda() for w in W])
    # both are FP64 chains of n_s steps; the laser phase (1e3 rad) carries 1e-13 of rounding
    # into terms that are summed with either sign
    for got, ref in ((du.cpu(), u.grad), (dl.cpu(), torch.stack([a0.grad, w0.grad]))):
        for c in range(got.shape[-1]):
            a, b = got[..., c], ref[..., c]
            assert float((a - b).norm()) <= 1e-10 * float(b.norm()), (c, a, b)
