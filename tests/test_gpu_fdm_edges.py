"""GPU frequency-domain method where its work is cut: blocks of 1,024 frequencies (odd and even
counts, remainders), groups of 32 samples with remainders, fewer samples than ring slots, samples
divided over a cluster or not, per-electron time axes, against the oracle's direct sum."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from gpu_cases import rel_l2  # noqa: E402
from paper_2206_03015_gb300 import lw  # noqa: E402
from workloads import simple  # noqa: E402

pytestmark = pytest.mark.gpu


def _compare(n_e, n_s, n_pix, n_omega, t_per_electron=False):
    tr = simple.random_smooth(n_e, n_s, 2e-17, n_s + n_e, gamma=5.0, amp=0.3,
                              t_per_electron=t_per_electron)
    rng = np.random.Generator(np.random.PCG64(n_pix))
    tx, ty = rng.uniform(-0.1, 0.1, n_pix), rng.uniform(-0.1, 0.1, n_pix)
    n_hat = np.stack([np.sin(tx), np.cos(tx) * np.sin(ty), np.cos(tx) * np.cos(ty)], -1)
    traj = lw.lw_trajectories_upload(tr.t, tr.r, tr.beta, tr.beta_dot, sections=lw.LW_SECTION_FP64)
    d_omega = 4e15 / n_omega
    S = lw.lw_spectrum_fdm(traj, lw.Detector(n_hat), 1e14, d_omega, n_omega, 2e-17).cpu().numpy()
    ref, _ = oracle.fdm(tr.t, tr.r, tr.beta, tr.beta_dot, n_hat,
                        1e14 + d_omega * np.arange(n_omega), 2e-17)
    # FP32 twiddles and fields of 1e-7 per term, as in the other comparison with the oracle
    for m in range(n_pix):
        assert rel_l2(S[m], ref[m]) <= 1e-5, m


@pytest.mark.parametrize("n_omega", [1, 31, 129, 1023, 1024, 1025, 2048, 2049, 3072, 4096])
def test_frequency_blocks(n_omega):
    _compare(2, 120, 2, n_omega)


@pytest.mark.parametrize("n_e,n_s", [(1, 1), (1, 14), (1, 15), (1, 31), (3, 42), (1, 127), (2, 80),
                                     (16, 127), (17, 130), (5, 2047)])
@pytest.mark.parametrize("t_per_electron", [False, True])
def test_sample_groups(n_e, n_s, t_per_electron):
    _compare(n_e, n_s, 3, 200, t_per_electron)


def test_many_pixels():
    _compare(1, 70, 1300, 64)
