"""Electron order, ends and input status of the upload on both sides of its one-CTA form (2,048
electrons) and of its 1,024 threads, with shared and per-electron time axes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2206_03015_gb300 import lw  # noqa: E402

pytestmark = pytest.mark.gpu

C0 = 299792458.0


@pytest.mark.parametrize("n_e", [1, 2, 31, 33, 1023, 1024, 1025, 2048, 2049])
@pytest.mark.parametrize("t_per_electron", [False, True])
@pytest.mark.parametrize("sections", [lw.LW_SECTION_FP64, lw.LW_SECTION_MIXED])
def test_order_and_bounds(n_e, t_per_electron, sections):
    rng = np.random.Generator(np.random.PCG64(n_e))
    t = 1e-15 * np.arange(4.0)
    r = np.zeros((n_e, 4, 3))
    r[..., 2] = rng.normal(scale=1e-5, size=(n_e, 1)) + 0.9 * C0 * t
    r[..., 0] = rng.normal(scale=1e-6, size=(n_e, 1))
    b = np.zeros((n_e, 4, 3))
    b[..., 2] = 0.9
    tt = t if not t_per_electron else t + rng.uniform(0, 1e-14, (n_e, 1))
    traj = lw.lw_trajectories_upload(tt, r, b, np.zeros_like(b), sections=sections, block=16)
    order = traj.order().cpu().numpy()
    assert np.array_equal(np.sort(order), np.arange(n_e))
    tau = (tt if t_per_electron else np.broadcast_to(t, (n_e, 4)))[:, 0] - r[:, 0, 2] / C0
    # sorted by buckets of 1/4096 of the range (a bucket's width of disorder, and its rounding)
    step = (tau.max() - tau.min()) / 4096
    assert np.all(np.diff(tau[order]) >= -1.001 * step)
    det = lw.Detector(np.array([[0.0, 0.0, 1.0], [0.01, 0.0, np.sqrt(1 - 1e-4)]]))
    lo, hi = lw.lw_grid_bounds(traj, det).cpu().tolist()
    n = det.n_hat.cpu().numpy()
    T = np.broadcast_to(tt, (n_e, 4))
    ta = [T[:, i, None] - (r[:, i] @ n.T) / C0 for i in (0, 3)]
    assert lo == pytest.approx(ta[0].min(), abs=1e-27) and hi == pytest.approx(ta[1].max(), abs=1e-27)


def test_reused_workspace_keeps_its_order_between_uploads():
    """Two uploads into one workspace without a wait between them, each followed by a deposit."""
    rng = np.random.Generator(np.random.PCG64(7))
    t = torch.from_numpy(1e-17 * np.arange(400.0)).cuda()
    det = lw.Detector(np.array([[0.0, 0.0, 1.0], [0.02, 0.0, np.sqrt(1 - 4e-4)]]))
    cases, ws = [], None
    for k in range(2):
        r = np.zeros((300, 400, 3))
        r[..., 2] = rng.normal(scale=1e-7, size=(300, 1)) + 0.99 * C0 * 1e-17 * np.arange(400.0)
        b = np.zeros_like(r)
        b[..., 2] = 0.99
        a = np.zeros_like(r)
        a[..., 0] = rng.normal(scale=1e14, size=(300, 1))
        cases.append([torch.from_numpy(x).cuda() for x in (r, b, a)])
    alone = []
    for c in cases:
        traj = lw.lw_trajectories_upload(t, *c, sections=lw.LW_SECTION_MIXED)
        if not alone:
            grid = lw.grid_from_bounds(-2e-15, 2e-15, 4096)
        alone.append(lw.lw_deposit_time_domain(traj, det, grid, lw.LW_MIXED))
        torch.cuda.synchronize()
    for c, want in zip(cases, alone):
        traj = lw.lw_trajectories_upload(t, *c, sections=lw.LW_SECTION_MIXED, ws=ws)
        ws = traj.ws
        got = lw.lw_deposit_time_domain(traj, det, grid, lw.LW_MIXED)
        # the same FP32 contributions added in FP64 in another order
        assert float((got - want).abs().max()) <= 1e-13 * float(want.abs().max())
