"""Spectra at the edges of the transform dispatch (one CTA per pixel pair below, four-step above):
lengths 2^9 .. 2^15, odd and single pixels, and pixel counts on both sides of the rule, against
torch's FP64 transform."""
import math

import pytest

torch = pytest.importorskip("torch")

from paper_2206_03015_gb300 import lw  # noqa: E402

pytestmark = pytest.mark.gpu

EPS0, C0 = 8.8541878128e-12, 299792458.0


def _record(prec, n_pix, n_bins, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(n_pix, 3, n_bins, dtype=torch.float64, device="cuda", generator=g) * 1e17
    x[:, 2] *= 0.01
    if prec in (lw.LW_FP64, lw.LW_MIXED):
        return x
    if prec == lw.LW_MIXED_F32:
        return x.float()
    if prec == lw.LW_MIXED_F32X4:
        out = torch.zeros(n_pix, n_bins, 4, device="cuda")
        out[..., :3] = x.permute(0, 2, 1)
        return out
    hi = x.float()
    return torch.stack([hi, (x - hi.double()).float()], -1).contiguous()


def _check(prec, n_pix, log2):
    n_bins = 1 << log2
    rec = _record(prec, n_pix, n_bins, 7 * log2 + n_pix)
    grid = lw.Grid(0.0, 3.0e-18, n_bins)
    S, X = lw.lw_spectrum(rec, prec, n_pix, grid, want_X=True)
    S2 = lw.lw_spectrum(rec, prec, n_pix, grid)
    K = lw.Q_E ** 2 / (16.0 * math.pi ** 3 * EPS0 * C0)
    ref = torch.conj_physical(torch.fft.rfft(lw.record_value(rec, prec), dim=-1))
    ref = ref * (math.sqrt(K) * grid.dt_u)
    # log2(N) roundings of the unit roundoff each (and a few of scale and split), in the 2-norm;
    # relative to each pixel's own spectrum, so that no pixel hides behind another
    eps = (2.0 ** -53 if prec == lw.LW_FP64 else 2.0 ** -24) * (log2 + 4)
    want_S = (ref.abs() ** 2).sum(1)
    for got, want in ((X, ref), (S, want_S), (S2, want_S)):   # X' kept or not
        d = (got.to(want.dtype) - want).flatten(1).norm(dim=1) / want.flatten(1).norm(dim=1)
        assert float(d.max()) <= eps, (prec, n_pix, log2, float(d.max()), eps)


@pytest.mark.parametrize("log2", [9, 10, 11, 12, 13, 14, 15])
@pytest.mark.parametrize("prec", [lw.LW_FP64, lw.LW_MIXED, lw.LW_MIXED_KAHAN, lw.LW_MIXED_F32,
                                  lw.LW_MIXED_F32X4])
def test_lengths_and_layouts(prec, log2):
    for n_pix in (1, 5):
        _check(prec, n_pix, log2)


@pytest.mark.parametrize("log2", [13, 14])
@pytest.mark.parametrize("n_pix", [150, 151, 153])
def test_both_sides_of_the_pixel_rule(log2, n_pix):
    _check(lw.LW_MIXED_F32X4, n_pix, log2)
    _check(lw.LW_MIXED_F32, n_pix, log2)
