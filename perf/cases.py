"""Timed work of the framework: the calls a user makes, through the public entry points.

A case is a dict of plain values; its "kind" names the call:

  step      stored trajectories -> spectra: upload, deposit, spectrum (device-resident inputs,
            buffers kept between steps)
  deposit   one time-domain deposit of uploaded trajectories; returns the record
  spectrum  spectra of a record in hand, with or without X'
  grad      FP64 spectrum of trajectory samples and its gradient (LWSpectrum)
  chain     gradient step through the GPU pusher (PushSpectrum): u0, a0, w0
  in_situ   push and deposit block by block, grid from a trial push
  batch     a planned batch of variants: one persistent deposit and the variants' spectra
  fdm       the frequency-domain method

Stored trajectories are electrons of a Gaussian bunch meeting a linearly polarised pulse
head-on, from the light-front solution of a plane wave (each electron sees the amplitude of
the Gaussian beam at its own radius), evaluated in FP64 at uniform lab times: seeded,
smooth and subluminal like a Boris-pushed bunch, made on the GPU in one go.
"""
from __future__ import annotations

import math

import torch

from paper_2206_03015_gb300 import insitu, lw
from paper_2206_03015_gb300.autograd import LWSpectrum, PushSpectrum, band_mask

C0 = 299792458.0
Q_E = 1.602176634e-19
EPS0 = 8.8541878128e-12
M_E = 9.1093837015e-31

PREC = {"fp64": lw.LW_FP64, "mixed": lw.LW_MIXED, "kahan": lw.LW_MIXED_KAHAN,
        "f32": lw.LW_MIXED_F32, "f32x4": lw.LW_MIXED_F32X4}

# beams: bunch sizes [m], mean gamma, relative spread, normalised emittance [m], laser
# (wavelength, a0, waist, intensity FWHM duration), detector half angle times gamma
BEAMS = {
    # electrons of one energy a few nm apart in a 10 fs pulse (plane wave), detector +-1/gamma
    "tiny": dict(s=(0.0, 0.0, 5e-9), gamma=50.0, spread=0.0, eps=0.0,
                 laser=(1.0e-6, 0.1, math.inf, 10e-15), half=1.0),
    # the paper's inverse Compton bunch: 5 x 5 x 10 um, gamma 60, 0.8 um laser
    "bunch": dict(s=(5e-6, 5e-6, 10e-6), gamma=60.0, spread=1e-3, eps=0.5e-6,
                  laser=(0.8e-6, 0.5, 20e-6, 30e-15), half=1.5),
    # a short bunch whose emitted line the observer grid resolves
    "short": dict(s=(0.5e-6, 0.5e-6, 0.1e-6), gamma=60.0, spread=1e-3, eps=0.5e-6,
                  laser=(0.8e-6, 0.5, 20e-6, 30e-15), half=1.5),
    # co-located electrons on axis in a 10 fs, a0 = 1 pulse
    "point": dict(s=(0.0, 0.0, 0.0), gamma=60.0, spread=1e-3, eps=0.0,
                  laser=(1.0e-6, 1.0, 20e-6, 10e-15), half=1.0),
}


def listed():
    return [
        # the smallest call: 16 electrons in a plane wave, 32 x 32 pixels; latency and launches
        dict(name="step_tiny", kind="step", beam="tiny", n_e=16, n_s=2000, nx=32, ny=32,
             n_bins=4096, prec="mixed"),
        # an ordinary simulation with ragged sizes and the planar FP32 record
        dict(name="step_medium", kind="step", beam="bunch", n_e=1001, n_s=4000, nx=50, ny=45,
             n_bins=16384, prec="f32"),
        # the paper's case at full size: the benchmark's step, the largest one
        dict(name="step_paper", kind="step", beam="bunch", n_e=10000, n_s=10000, nx=64, ny=64,
             n_bins=65536, prec="f32x4"),
        # compensated record, both field terms, odd sizes, a grid that is no power of two
        dict(name="deposit_kahan", kind="deposit", beam="short", n_e=999, n_s=3001, nx=37, ny=41,
             n_bins=20000, prec="kahan", velocity=True),
        # the FP64 path, which users check the mixed one against
        dict(name="deposit_fp64", kind="deposit", beam="bunch", n_e=1000, n_s=5000, nx=32, ny=32,
             n_bins=16384, prec="fp64", velocity=False),
        # spectra of a short grid (one CTA per pixel pair)
        dict(name="spectrum_4096", kind="spectrum", nx=64, ny=64, n_bins=4096, prec="mixed",
             want_X=False),
        # FP64 spectra with X' kept for a gradient, odd pixel count, four-step transform
        dict(name="spectrum_fp64", kind="spectrum", nx=33, ny=31, n_bins=16384, prec="fp64",
             want_X=True),
        # gradient of FP64 spectra with respect to given trajectories
        dict(name="grad_fp64", kind="grad", beam="point", n_e=64, n_s=1200, nx=20, ny=20,
             n_bins=4096),
        # the gradient step of the mixed chain at the size of the framework's own benchmark
        dict(name="chain_mixed", kind="chain", beam="point", n_e=2048, n_s=4096, nx=32, ny=32,
             n_bins=16384, prec="f32x4"),
        # trajectories never stored: push and deposit in blocks of 1,024 steps
        dict(name="in_situ", kind="in_situ", beam="bunch", n_e=1500, n_s=5000, nx=32, ny=32,
             n_bins=16384, prec="f32x4"),
        # a design sweep: eight variants of different sizes in one launch
        dict(name="batch", kind="batch", beam="bunch", variants=8, n_e_lo=256, n_e_hi=2048,
             n_s_lo=1000, n_s_hi=6000, side_lo=16, side_hi=48, log2_lo=12, log2_hi=15,
             prec="f32x4"),
        # the comparison method on a resolved bunch
        dict(name="fdm", kind="fdm", beam="short", n_e=64, n_s=1000, nx=12, ny=12, n_omega=2048),
    ]


def _fewer_points(c, most):
    """The case with as many electrons as keep its grid points reached at `most`."""
    one = _points(c["beam"], 1, c["n_s"], c["nx"] * c["ny"], c["n_bins"])
    c["n_e"] = max(16, min(c["n_e"], int(most / one)))
    return c


def draw(rng):
    def logi(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "step", "deposit", "deposit", "spectrum", "grad", "chain",
                       "in_situ", "batch", "fdm"])
    if kind == "step":
        beam = rng.choice(["tiny", "bunch", "bunch", "short"])
        c = dict(kind=kind, beam=beam, n_e=logi(16, 6000), n_s=logi(500, 10000), nx=logi(16, 64),
                 ny=logi(16, 64), n_bins=1 << rng.randint(12, 16),
                 prec=rng.choice(["mixed", "f32", "f32x4", "kahan", "fp64"]))
        cap = 2.0e9 if c["prec"] == "fp64" else 4.0e10 if beam == "bunch" else 8.0e9
        while c["n_e"] * c["n_s"] * c["nx"] * c["ny"] > cap:
            c["n_e"] = max(16, c["n_e"] * 2 // 3)
            c["nx"] = max(16, c["nx"] * 3 // 4)
            c["n_s"] = max(500, c["n_s"] * 3 // 4)
        return _fewer_points(c, 1.0e8 if c["prec"] == "fp64" else 1.0e9)
    if kind == "deposit":
        c = dict(kind=kind, beam=rng.choice(["bunch", "short"]), n_e=logi(200, 3000),
                 n_s=logi(1000, 6000), nx=logi(16, 48), ny=logi(16, 48),
                 n_bins=logi(4000, 40000), prec=rng.choice(["kahan", "f32", "f32x4", "fp64"]),
                 velocity=rng.random() < 0.3)
        cap = 4.0e9 if c["prec"] == "fp64" else 1.0e10
        while c["n_e"] * c["n_s"] * c["nx"] * c["ny"] > cap:
            c["n_e"] = max(200, c["n_e"] * 2 // 3)
            c["nx"] = max(16, c["nx"] * 3 // 4)
            c["n_s"] = max(1000, c["n_s"] * 3 // 4)
        return _fewer_points(c, 1.0e8 if c["prec"] == "fp64" else 1.0e9)
    if kind == "spectrum":
        log2 = rng.randint(10, 16)
        prec = rng.choice(["mixed", "f32", "f32x4", "kahan", "fp64"])
        side = min(64, int(math.sqrt((1 << 27) >> log2)))
        return dict(kind=kind, nx=logi(9, side), ny=logi(9, side), n_bins=1 << log2, prec=prec,
                    want_X=rng.random() < 0.5)
    if kind == "grad":
        return dict(kind=kind, beam="point", n_e=logi(16, 96), n_s=logi(300, 1500),
                    nx=logi(8, 24), ny=logi(8, 24), n_bins=1 << rng.randint(11, 13))
    if kind == "chain":
        return dict(kind=kind, beam="point", n_e=logi(64, 2048), n_s=logi(500, 4096),
                    nx=logi(8, 32), ny=logi(8, 32), n_bins=1 << rng.randint(12, 14),
                    prec="f32x4")
    if kind == "in_situ":
        return dict(kind=kind, beam=rng.choice(["bunch", "short"]), n_e=logi(100, 3000),
                    n_s=logi(1000, 6000), nx=logi(16, 40), ny=logi(16, 40),
                    n_bins=1 << rng.randint(12, 15), prec=rng.choice(["f32", "f32x4"]))
    if kind == "batch":
        return dict(kind=kind, beam="bunch", variants=rng.randint(3, 12), n_e_lo=128,
                    n_e_hi=logi(512, 2048), n_s_lo=800, n_s_hi=logi(2000, 6000), side_lo=16,
                    side_hi=rng.randint(20, 48), log2_lo=12, log2_hi=15,
                    prec=rng.choice(["f32", "f32x4", "mixed"]))
    return dict(kind="fdm", beam="short", n_e=logi(16, 100), n_s=logi(300, 1500), nx=logi(4, 14),
                ny=logi(4, 14), n_omega=logi(256, 3000))


# ------------------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _detector(nx, ny, half):
    """Cell-centred directions over +-half in both angles (far field, around +z)."""
    ax = (2.0 * (torch.arange(nx, dtype=torch.float64) + 0.5) / nx - 1.0) * half
    ay = (2.0 * (torch.arange(ny, dtype=torch.float64) + 0.5) / ny - 1.0) * half
    tx, ty = torch.meshgrid(ax, ay, indexing="ij")
    n = torch.stack([torch.sin(tx), torch.cos(tx) * torch.sin(ty),
                     torch.cos(tx) * torch.cos(ty)], -1)
    return n.reshape(-1, 3).contiguous().cuda()


def _pulse_half(laser):
    """Half length in phase time of the cos^2 pulse whose intensity FWHM is the laser's."""
    return laser[3] / (4.0 / math.pi * math.acos(0.5 ** 0.25))


def _window(b):
    return 0.5 * (_pulse_half(b["laser"]) + 4.0 * b["s"][2] / C0) * 1.05


def _bunch(b, n_e, g):
    """(r, u) at t = 0: positions, u = gamma beta, truncated at 4 sigma."""
    z = torch.randn(n_e, 6, dtype=torch.float64, device="cuda", generator=g).clamp_(-4.0, 4.0)
    sx, sy, sz = b["s"]
    gam = b["gamma"] * (1.0 + b["spread"] * z[:, 3])
    xp = z[:, 4] * (b["eps"] / (b["gamma"] * sx) if sx > 0 else 0.0)
    yp = z[:, 5] * (b["eps"] / (b["gamma"] * sy) if sy > 0 else 0.0)
    uz = torch.sqrt((gam * gam - 1.0) / (1.0 + xp * xp + yp * yp))
    r = torch.stack([sx * z[:, 0], sy * z[:, 1], sz * z[:, 2]], -1)
    return r, torch.stack([uz * xp, uz * yp, uz], -1)


def _trajectories(b, n_e, n_s, seed):
    """(t [n_s+1], r, beta, beta_dot [n_e][n_s+1][3]) of the bunch in the pulse
    a(xi) = a0 cos^2(pi xi / 2T) cos(omega xi): with h = gamma + u_z and u_y conserved and
    u_x = u_x0 + a, the lab time and x are integrals of a and a^2 (sums of sines), and the
    phase time xi at a lab time follows by a fixed-point iteration (contraction a^2/h^2)."""
    lam, a0, w0, _ = b["laser"]
    T, om = _pulse_half(b["laser"]), 2.0 * math.pi * C0 / lam
    ka = math.pi / T
    th = _window(b)
    r0, u0 = _bunch(b, n_e, _gen(seed))
    t = torch.linspace(-th, th, n_s + 1, dtype=torch.float64, device="cuda")
    R, B, A = (torch.empty(n_e, n_s + 1, 3, dtype=torch.float64, device="cuda")
               for _ in range(3))
    step = max(1, (1 << 22) // (n_s + 1))
    for k in range(0, n_e, step):
        r, u = r0[k:k + step, None, :], u0[k:k + step, None, :]
        amp = a0 * torch.exp(-(r[..., 0] ** 2 + r[..., 1] ** 2) / (w0 * w0))
        ux0, uy = u[..., 0], u[..., 1]
        h = u[..., 2] + torch.sqrt(1.0 + (u * u).sum(-1))
        d = 1.0 + ux0 * ux0 + uy * uy
        xi0 = r[..., 2] / C0

        def i1(x):
            return amp * (torch.sin(om * x) / (2 * om) + torch.sin((om + ka) * x) / (4 * (om + ka))
                          + torch.sin((om - ka) * x) / (4 * (om - ka)))

        def i2(x):
            s = 0.375 * x + torch.sin(ka * x) / (2 * ka) + torch.sin(2 * ka * x) / (16 * ka)
            for c, w in ((0.375, 2 * om), (0.25, 2 * om + ka), (0.25, 2 * om - ka),
                         (0.0625, 2 * om + 2 * ka), (0.0625, 2 * om - 2 * ka)):
                s = s + (c / w) * torch.sin(w * x)
            return 0.5 * amp * amp * s

        h2 = h * h
        free = 2.0 * t[None, :] + xi0 * (1.0 + d / h2)
        xi = free / (1.0 + d / h2)
        for _ in range(5):
            x = xi.clamp(-T, T)
            xi = (free - (2.0 * ux0 * i1(x) + i2(x)) / h2) / (1.0 + d / h2)
        x = xi.clamp(-T, T)
        env = 0.5 * (1.0 + torch.cos(ka * x))
        cw, sw = torch.cos(om * x), torch.sin(om * x)
        a = amp * env * cw
        da = amp * (-0.5 * ka * torch.sin(ka * x) * cw - om * env * sw)
        ux = ux0 + a
        perp = 1.0 + ux * ux + uy * uy
        gam, uz = 0.5 * (h + perp / h), 0.5 * (h - perp / h)
        dg = ux * da / h
        f = h / (gam * gam)
        R[k:k + step, :, 0] = r[..., 0] + (C0 / h) * (ux0 * (xi - xi0) + i1(x))
        R[k:k + step, :, 1] = r[..., 1] + (C0 / h) * uy * (xi - xi0)
        R[k:k + step, :, 2] = C0 * (xi - t[None, :])
        for c, (v, dv) in enumerate(((ux, da), (uy, 0.0), (uz, -dg))):
            B[k:k + step, :, c] = v / gam
            A[k:k + step, :, c] = f * (dv - v * dg / gam)
    return t, R, B, A


def _grid(traj, det, n_bins):
    lo, hi = lw.lw_grid_bounds(traj, det).cpu().tolist()
    return lw.grid_from_bounds(lo, hi, n_bins)


def _sections(prec):
    return lw.LW_SECTION_FP64 if prec == lw.LW_FP64 else lw.LW_SECTION_MIXED


def _push_inputs(case, seed):
    """Initial state of a pushed bunch at the window's start: (r0, u0, laser, t0, t1)."""
    b = BEAMS[case["beam"]]
    th = _window(b)
    r, u = _bunch(b, case["n_e"], _gen(seed))
    v = C0 * u / torch.sqrt(1.0 + (u * u).sum(-1, keepdim=True))
    return (r - v * th).contiguous(), u.contiguous(), b["laser"], -th, th


def _line(b):
    """On-axis fundamental 4 gamma^2 omega_L / (1 + a0^2/2)."""
    lam, a0 = b["laser"][0], b["laser"][1]
    return 4.0 * b["gamma"] ** 2 * (2.0 * math.pi * C0 / lam) / (1.0 + 0.5 * a0 * a0)


def _sweep(case):
    """The variants' sizes: log-spread over the ranges, a fixed design like a user's list."""
    n = case["variants"]
    out = []
    for v in range(n):
        def at(lo, hi, stride):
            f = ((v * stride) % n) / max(1, n - 1)
            return int(round(lo * (hi / lo) ** f))
        out.append((at(case["n_e_lo"], case["n_e_hi"], 1), at(case["n_s_lo"], case["n_s_hi"], 5),
                    at(case["side_lo"], case["side_hi"], 3),
                    1 << (case["log2_lo"] + (v * 3) % (case["log2_hi"] - case["log2_lo"] + 1))))
    return out


def _record(case, seed):
    """A record as the deposit leaves it: per pixel a chirped pulse with noise, x largest."""
    n_pix, N = case["nx"] * case["ny"], case["n_bins"]
    g = _gen(seed)
    j = torch.arange(N, dtype=torch.float64, device="cuda") / N
    p = torch.rand(n_pix, 3, dtype=torch.float64, device="cuda", generator=g)
    scale = torch.tensor([1.0, 0.2, 0.02], dtype=torch.float64, device="cuda") * 1e17
    rec = torch.empty(n_pix, 3, N, dtype=torch.float64, device="cuda")
    for m in range(0, n_pix, 256):
        q = p[m:m + 256, :, None]
        env = torch.exp(-(((j - 0.3 - 0.4 * q) / (0.02 + 0.1 * q)) ** 2))
        x = env * torch.cos(2.0 * math.pi * (0.05 + 0.3 * q) * N * j * (1.0 + 0.1 * j))
        x += 1e-3 * torch.randn(x.shape, dtype=torch.float64, device="cuda", generator=g)
        rec[m:m + 256] = x * scale[:, None]
    return rec


def _as_record(rec, prec):
    if prec in (lw.LW_FP64, lw.LW_MIXED):
        return rec
    if prec == lw.LW_MIXED_F32:
        return rec.float()
    if prec == lw.LW_MIXED_F32X4:
        out = torch.zeros(rec.shape[0], rec.shape[2], 4, dtype=torch.float32, device="cuda")
        out[..., :3] = rec.permute(0, 2, 1)
        return out
    hi = rec.float()
    return torch.stack([hi, (rec - hi.double()).float()], -1).contiguous()


# ------------------------------------------------------------------------------ the calls

def prepare(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        prec = PREC[case["prec"]]
        rec = _as_record(_record(case, seed), prec)
        grid = lw.Grid(0.0, 2.0e-18, case["n_bins"])
        n_pix = case["nx"] * case["ny"]
        ws = lw.workspace(lw.spectrum_workspace_bytes(prec, n_pix, grid))
        S = torch.empty((n_pix, case["n_bins"] // 2 + 1), device="cuda",
                        dtype=torch.float64 if prec == lw.LW_FP64 else torch.float32)
        return dict(case=case, prec=prec, rec=rec, grid=grid, n_pix=n_pix, ws=ws, S=S)
    if kind == "batch":
        b, prec = BEAMS[case["beam"]], PREC[case["prec"]]
        items = []
        for v, (n_e, n_s, side, n_bins) in enumerate(_sweep(case)):
            gamma = 30.0 * (150.0 / 30.0) ** (v / max(1, case["variants"] - 1))
            bv = dict(b, gamma=gamma)
            det = lw.Detector(_detector(side, side, bv["half"] / gamma))
            traj = lw.lw_trajectories_upload(*_trajectories(bv, n_e, n_s, seed * 131 + v),
                                             sections=lw.LW_SECTION_MIXED)
            grid = _grid(traj, det, n_bins)
            del traj._inputs
            shape, dtype = lw.record_shape(det, grid, prec)
            items.append(dict(traj=traj, det=det, grid=grid,
                              rec=torch.empty(shape, dtype=dtype, device="cuda"),
                              S=torch.empty((det.n_pix, n_bins // 2 + 1), dtype=torch.float32,
                                            device="cuda")))
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        plan = lw.lw_batch_plan([i["traj"] for i in items], [i["det"] for i in items],
                                [i["grid"] for i in items], [i["rec"] for i in items],
                                precision=prec, statuses=[status] * len(items))
        ws = lw.workspace(max(lw.spectrum_workspace_bytes(prec, i["det"].n_pix, i["grid"])
                              for i in items))
        return dict(case=case, prec=prec, items=items, plan=plan, ws=ws, status=status)
    b = BEAMS[case["beam"]]
    det = lw.Detector(_detector(case["nx"], case["ny"], b["half"] / b["gamma"]))
    if kind == "in_situ":
        return dict(case=case, det=det, push=_push_inputs(case, seed), prec=PREC[case["prec"]])
    if kind == "chain":
        r0, u0, laser, t0, t1 = _push_inputs(case, seed)
        n_s = case["n_s"]
        r1, u1 = r0.clone(), u0.clone()
        t = torch.empty(n_s + 1, dtype=torch.float64, device="cuda")
        bufs = [torch.empty(case["n_e"], n_s + 1, 3, dtype=torch.float64, device="cuda")
                for _ in range(3)]
        lw.lw_boris_push(r1, u1, t0, (t1 - t0) / n_s, n_s, laser, t, *bufs)
        lo, hi = insitu.grid_bounds_from_ends(t0, t1, r0, r1, det)
        # bounds rounded to single precision, as a user writes them down in a configuration
        lo = float(torch.tensor(lo, dtype=torch.float32))
        hi = float(torch.tensor(hi, dtype=torch.float32))
        grid = lw.grid_from_bounds(lo - 1e-5 * (hi - lo), hi + 1e-5 * (hi - lo), case["n_bins"])
        w = band_mask(grid, _line(b)).cuda() * (2.0 * math.pi / (grid.n_bins * grid.dt_u))
        return dict(case=case, det=det, grid=grid, prec=PREC[case["prec"]], r0=r0, laser=laser,
                    t0=t0, t1=t1, w=w, leaves=(
                        u0, torch.tensor(laser[1], dtype=torch.float64, device="cuda"),
                        torch.tensor(laser[2], dtype=torch.float64, device="cuda")))
    inputs = _trajectories(b, case["n_e"], case["n_s"], seed)
    if kind == "grad":
        traj = lw.lw_trajectories_upload(*inputs, sections=lw.LW_SECTION_FP64)
        grid = _grid(traj, det, case["n_bins"])
        w = band_mask(grid, _line(b)).cuda() * (2.0 * math.pi / (grid.n_bins * grid.dt_u))
        return dict(case=case, det=det, grid=grid, inputs=inputs, w=w)
    if kind == "fdm":
        traj = lw.lw_trajectories_upload(*inputs, sections=lw.LW_SECTION_FP64)
        return dict(case=case, det=det, traj=traj, d_omega=2.0 * _line(b) / case["n_omega"],
                    dt=2.0 * _window(b) / case["n_s"])
    prec = PREC[case["prec"]]
    traj = lw.lw_trajectories_upload(*inputs, sections=_sections(prec))
    grid = _grid(traj, det, case["n_bins"])
    shape, dtype = lw.record_shape(det, grid, prec)
    st = dict(case=case, det=det, grid=grid, prec=prec,
              rec=torch.empty(shape, dtype=dtype, device="cuda"),
              status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if kind == "deposit":
        del traj._inputs
        st["traj"] = traj
        return st
    st.update(inputs=inputs, traj_ws=traj.ws,
              ws=lw.workspace(lw.spectrum_workspace_bytes(prec, det.n_pix, grid)),
              S=torch.empty((det.n_pix, case["n_bins"] // 2 + 1), device="cuda",
                            dtype=torch.float64 if prec == lw.LW_FP64 else torch.float32))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        traj = lw.lw_trajectories_upload(*st["inputs"], sections=_sections(st["prec"]),
                                         ws=st["traj_ws"])
        lw.lw_deposit_time_domain(traj, st["det"], st["grid"], st["prec"], record=st["rec"],
                                  status=st["status"])
        S = lw.lw_spectrum(st["rec"], st["prec"], st["det"].n_pix, st["grid"], ws=st["ws"],
                           out=st["S"])
        return {"S": S, "status": st["status"]}
    if kind == "deposit":
        flags = lw.LW_FIELD_ACCEL | (lw.LW_FIELD_VELOCITY if case["velocity"] else 0)
        rec = lw.lw_deposit_time_domain(st["traj"], st["det"], st["grid"], st["prec"], flags,
                                        record=st["rec"], status=st["status"])
        return {"record": rec, "status": st["status"]}
    if kind == "spectrum":
        out = lw.lw_spectrum(st["rec"], st["prec"], st["n_pix"], st["grid"],
                             want_X=case["want_X"], ws=st["ws"], out=st["S"])
        return {"S": out[0], "X": out[1]} if case["want_X"] else {"S": out}
    if kind == "grad":
        t, *x = st["inputs"]
        x = [v.detach().requires_grad_(True) for v in x]
        S = LWSpectrum.apply(t, *x, st["det"], st["grid"])
        (S * st["w"]).sum().backward()
        return {"S": S.detach(), "dr": x[0].grad, "dbeta": x[1].grad, "dbdot": x[2].grad}
    if kind == "chain":
        u0, a0, w0 = (v.detach().requires_grad_(True) for v in st["leaves"])
        lam, fwhm = st["laser"][0], st["laser"][3]
        S = PushSpectrum.apply(u0, a0, w0, st["r0"], lam, fwhm, st["t0"], st["t1"], case["n_s"],
                               st["det"], st["grid"], lw.Q_E, st["prec"])
        (S.to(torch.float64) * st["w"]).sum().backward()
        return {"S": S.detach(), "du0": u0.grad, "da0": a0.grad, "dw0": w0.grad}
    if kind == "in_situ":
        r0, u0, laser, t0, t1 = st["push"]
        S, grid, rec = insitu.in_situ_spectrum(r0, u0, laser, t0, t1, case["n_s"], st["det"],
                                               case["n_bins"], precision=st["prec"])
        return {"S": S, "t_min": grid.t_min, "dt_u": grid.dt_u, "record": rec}
    if kind == "batch":
        lw.lw_batch_deposit(st["plan"])
        for i in st["items"]:
            lw.lw_spectrum(i["rec"], st["prec"], i["det"].n_pix, i["grid"], ws=st["ws"],
                           out=i["S"])
        return {"S": [i["S"] for i in st["items"]], "status": st["status"]}
    return {"S": lw.lw_spectrum_fdm(st["traj"], st["det"], 0.0, st["d_omega"], case["n_omega"],
                                    st["dt"])}


# ------------------------------------------------------------------------------ the work

def _step_work(n_e, n_s, n_pix, n_bins, prec, points):
    """Bytes and operations of upload + deposit + spectrum of `points` grid points reached:
    inputs read once, spectra written once; two fields (29 each), their interpolation and
    weight (14) and the two bracketing coordinates (14) per grid point, 2.5 N log2 N per
    real row's transform."""
    w = 8 if prec == "fp64" else 4
    return {"bytes": 72.0 * n_e * (n_s + 1) + w * n_pix * (n_bins // 2 + 1.0),
            "flops": 86.0 * points + 7.5 * n_pix * n_bins * math.log2(n_bins)}


def _points(beam, n_e, n_s, n_pix, n_bins):
    """Grid points the electrons reach: each electron's own arrival span (its window's phase
    advance) over the whole grid's span (bunch length added)."""
    b = BEAMS[beam]
    g = b["gamma"]
    own = 2.0 * _window(b) * (1.0 + 0.5 * b["half"] ** 2) / (2.0 * g * g)
    span = own + 8.0 * b["s"][2] / C0
    return n_e * n_pix * n_bins * min(1.0, own / span)


def work(case):
    kind = case["kind"]
    if kind == "spectrum":
        n_pix, N = case["nx"] * case["ny"], case["n_bins"]
        word = {"fp64": 24, "mixed": 24, "kahan": 24, "f32": 12, "f32x4": 16}[case["prec"]]
        out = (8 if case["prec"] == "fp64" else 4) * (7 if case["want_X"] else 1)
        return {"bytes": n_pix * (word * N + out * (N // 2 + 1.0)),
                "flops": 7.5 * n_pix * N * math.log2(N)}
    if kind == "batch":
        tot = {"bytes": 0.0, "flops": 0.0}
        for n_e, n_s, side, n_bins in _sweep(case):
            w = _step_work(n_e, n_s, side * side, n_bins, case["prec"],
                           _points(case["beam"], n_e, n_s, side * side, n_bins))
            tot["bytes"] += w["bytes"] - 32.0 * n_e * (n_s + 1)   # already in the 40 B layout
            tot["flops"] += w["flops"]
        return tot
    n_e, n_s, n_pix = case["n_e"], case["n_s"], case["nx"] * case["ny"]
    if kind == "fdm":
        return {"bytes": 80.0 * n_e * (n_s + 1) + 8.0 * n_pix * case["n_omega"],
                "flops": 16.0 * n_e * (n_s + 1) * n_pix * case["n_omega"]}
    N = case["n_bins"]
    pts = _points(case["beam"], n_e, n_s, n_pix, N)
    if kind == "step":
        return _step_work(n_e, n_s, n_pix, N, case["prec"], pts)
    if kind == "deposit":
        word = {"fp64": 24, "kahan": 24, "f32": 12, "f32x4": 16}[case["prec"]]
        samp = 72 if case["prec"] == "fp64" else 40
        return {"bytes": samp * n_e * (n_s + 1.0) + word * n_pix * float(N), "flops": 86.0 * pts}
    if kind == "in_situ":   # two pushes (trial and real) of about 250 operations a step
        return {"bytes": 48.0 * n_e + 16.0 * n_pix * N + 4.0 * n_pix * (N // 2 + 1),
                "flops": 86.0 * pts + 500.0 * n_e * n_s + 7.5 * n_pix * N * math.log2(N)}
    # gradients: the forward, its transpose at about twice the work
    f = _step_work(n_e, n_s, n_pix, N, "fp64" if kind == "grad" else case["prec"], pts)
    push = 2000.0 * n_e * n_s if kind == "chain" else 0.0
    grads = 72.0 * n_e * (n_s + 1) if kind == "grad" else 24.0 * n_e
    return {"bytes": f["bytes"] + grads, "flops": 3.0 * f["flops"] + push}


# ------------------------------------------------------------------------------ 64-bit values

def _fields64(n, b, a, velocity, R):
    """F = n x ((n - beta) x beta_dot) / D^3 (+ velocity term) in FP64, broadcast."""
    D = 1.0 - (n * b).sum(-1, keepdim=True)
    m = n - b
    F = torch.linalg.cross(n, torch.linalg.cross(m, a.expand(m.shape))) / D ** 3
    if velocity:
        F = F + C0 * m * (1.0 - (b * b).sum(-1, keepdim=True)) / (D ** 3 * R)
    return F


def _deposit64(inputs, n_hat, grid, velocity=False, R=1.0):
    """Algorithm 2 in torch FP64: [n_pix][3][n_bins]; differentiable in (r, beta, beta_dot)."""
    t, r, beta, bdot = inputs
    n_pix, N = n_hat.shape[0], grid.n_bins
    n_e, ns1 = r.shape[0], r.shape[1]
    rec = torch.zeros(n_pix * 3 * N, dtype=torch.float64, device="cuda")
    inv = 1.0 / grid.dt_u
    keep = r.requires_grad
    pstep = n_pix if keep else max(1, (1 << 25) // ns1)
    for k in range(n_e):
        for p in range(0, n_pix, pstep):
            n = n_hat[p:p + pstep]
            ta = t[None, :] - (n @ r[k].T) * (1.0 / C0)
            J = torch.floor((ta.detach() - grid.t_min) * inv).to(torch.int64)
            cnt = (J[:, 1:].clamp(-1, N - 1) - J[:, :-1].clamp(-1, N - 1)).clamp_(min=0)
            q = cnt.reshape(-1)
            seg = torch.repeat_interleave(torch.arange(q.numel(), device="cuda"), q)
            if not seg.numel():
                continue
            first = torch.cumsum(q, 0) - q
            m, i = seg // (ns1 - 1), seg % (ns1 - 1)
            j = J[:, :-1].clamp(-1, N - 1)[m, i] + 1 + torch.arange(
                seg.numel(), device="cuda") - first[seg]
            tb, te = ta[m, i], ta[m, i + 1]
            tj = grid.t_min + j.to(torch.float64) * grid.dt_u
            w = ((tj - tb) / (te - tb))[:, None]
            Fb = _fields64(n[m], beta[k][i], bdot[k][i], velocity, R)
            Fa = _fields64(n[m], beta[k][i + 1], bdot[k][i + 1], velocity, R)
            v = Fb * (1.0 - w) + Fa * w
            at = (((m + p) * 3)[:, None] + torch.arange(3, device="cuda")) * N + j[:, None]
            if keep:
                rec = rec.index_add(0, at.reshape(-1), v.reshape(-1))
            else:
                rec.index_add_(0, at.reshape(-1), v.reshape(-1))
    return rec.view(n_pix, 3, N)


def _spectrum64(rec, dt_u, want_X=False):
    K = Q_E * Q_E / (16.0 * math.pi ** 3 * EPS0 * C0)
    X = torch.conj_physical(torch.fft.rfft(rec, dim=-1)) * (math.sqrt(K) * dt_u)
    S = (X.real ** 2 + X.imag ** 2).sum(1)
    return (S, X) if want_X else S


def _push64(r, u, laser, t0, t1, n_s):
    """The Boris push of the Gaussian beam in torch FP64: samples (t, r, beta, beta_dot)."""
    lam, a0, w0, fwhm = laser
    om = 2.0 * math.pi * C0 / lam
    sig = fwhm / (2.0 * math.sqrt(math.log(2.0)))
    zR = math.pi * w0 * w0 / lam
    E0 = a0 * M_E * C0 * om / Q_E
    qm, dt = -Q_E / M_E, (t1 - t0) / n_s
    t = t0 + dt * torch.arange(n_s + 1, dtype=torch.float64, device="cuda")
    R, U = (torch.empty(n_s + 1, r.shape[0], 3, dtype=torch.float64, device="cuda")
            for _ in range(2))

    def Ex(x, tt):
        z = -x[..., 2]
        w = w0 * torch.sqrt(1.0 + (z / zR) ** 2)
        rho2 = x[..., 0] ** 2 + x[..., 1] ** 2
        xi = tt + x[..., 2] / C0
        ph = om * xi + om / C0 * rho2 * z / (2.0 * (z * z + zR * zR)) - torch.atan(z / zR)
        return (E0 * (w0 / w) * torch.exp(-rho2 / (w * w) - xi * xi / (2.0 * sig * sig))
                * torch.cos(ph))

    R[0], U[0] = r, u
    for s in range(n_s):
        rh = r + (0.5 * dt * C0) * u / torch.sqrt(1.0 + (u * u).sum(-1, keepdim=True))
        E = Ex(rh, t0 + dt * (s + 0.5))
        e = qm * dt / (2.0 * C0) * E
        um = u + torch.stack([e, torch.zeros_like(e), torch.zeros_like(e)], -1)
        tv = qm * dt / (2.0 * torch.sqrt(1.0 + (um * um).sum(-1))) * (-E / C0)
        sv = 2.0 * tv / (1.0 + tv * tv)
        px, pz = um[:, 0] - um[:, 2] * tv, um[:, 2] + um[:, 0] * tv
        u = torch.stack([um[:, 0] - pz * sv + e, um[:, 1], um[:, 2] + px * sv], -1)
        r = rh + (0.5 * dt * C0) * u / torch.sqrt(1.0 + (u * u).sum(-1, keepdim=True))
        R[s + 1], U[s + 1] = r, u
    R, U = R.transpose(0, 1).contiguous(), U.transpose(0, 1).contiguous()
    gam = torch.sqrt(1.0 + (U * U).sum(-1, keepdim=True))
    b = U / gam
    E = Ex(R, t[None, :])[..., None]
    bx, bz = b[..., 0:1], b[..., 2:3]
    ex = torch.cat([E + bz * E, torch.zeros_like(E), -bx * E], -1)   # E + c beta x B, B_y=-E/c
    return t, R, b, qm / (gam * C0) * (ex - b * (bx * E))


def exact(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        prec = PREC[case["prec"]]
        rec = lw.record_value(_as_record(_record(case, seed), prec), prec)
        S, X = _spectrum64(rec, 2.0e-18, want_X=True)
        return {"S": S, "X": X} if case["want_X"] else {"S": S}
    if kind in ("batch", "chain"):
        return None   # many variants / a sequential gradient: minutes in plain torch
    b = BEAMS[case["beam"]]
    n_hat = _detector(case["nx"], case["ny"], b["half"] / b["gamma"])
    det = lw.Detector(n_hat)
    if kind == "fdm":
        t, r, beta, bdot = _trajectories(b, case["n_e"], case["n_s"], seed)
        dw, dt, W = 2.0 * _line(b) / case["n_omega"], 2.0 * _window(b) / case["n_s"], case["n_omega"]
        if case["n_e"] * case["n_s"] * n_hat.shape[0] * W > 4.0e10:
            return None
        out = torch.empty(n_hat.shape[0], W, dtype=torch.float64, device="cuda")
        lo = torch.arange(64, dtype=torch.float64, device="cuda") * dw
        hi = torch.arange(0, W, 64, dtype=torch.float64, device="cuda") * dw
        for m in range(n_hat.shape[0]):
            n = n_hat[m]
            tau = (t[None, :] - (r @ n) / C0).reshape(-1)
            D = 1.0 - beta @ n
            v = n - beta
            A = (torch.linalg.cross(n.expand(v.shape), torch.linalg.cross(v, bdot))
                 / (D * D)[..., None]).reshape(-1, 3)
            e_lo = torch.polar(torch.ones_like(tau[:, None]), tau[:, None] * lo)
            e_hi = torch.polar(torch.ones_like(tau[:, None]), tau[:, None] * hi)
            s = torch.zeros(hi.numel() * 64, dtype=torch.float64, device="cuda")
            for c in range(3):
                X = (e_hi * A[:, c:c + 1]).T @ e_lo
                s += (X.real ** 2 + X.imag ** 2).reshape(-1)
            out[m] = s[:W]
        return {"S": out * (Q_E * Q_E * dt * dt / (16.0 * math.pi ** 3 * EPS0 * C0))}
    deposits = float(case["n_e"]) * case["n_s"] * n_hat.shape[0]
    if kind == "grad":
        if _points(case["beam"], case["n_e"], case["n_s"], n_hat.shape[0], case["n_bins"]) > 2e8:
            return None
        t, *x = _trajectories(b, case["n_e"], case["n_s"], seed)
        traj = lw.lw_trajectories_upload(t, *x, sections=lw.LW_SECTION_FP64)
        grid = _grid(traj, det, case["n_bins"])
        w = band_mask(grid, _line(b)).cuda() * (2.0 * math.pi / (grid.n_bins * grid.dt_u))
        rec = torch.zeros(n_hat.shape[0], 3, grid.n_bins, dtype=torch.float64, device="cuda")
        for k in range(case["n_e"]):
            rec += _deposit64([t] + [v[k:k + 1] for v in x], n_hat, grid)
        rec.requires_grad_(True)
        S = _spectrum64(rec, grid.dt_u)
        (S * w).sum().backward()
        out = [torch.empty_like(v) for v in x]
        for k in range(case["n_e"]):   # the deposit is linear in its electrons
            leaf = [v[k:k + 1].clone().requires_grad_(True) for v in x]
            (_deposit64([t] + leaf, n_hat, grid) * rec.grad).sum().backward()
            for o, v in zip(out, leaf):
                o[k] = v.grad[0]
        return {"S": S.detach(), "dr": out[0], "dbeta": out[1], "dbdot": out[2]}
    points = _points(case["beam"], case["n_e"], case["n_s"], n_hat.shape[0], case["n_bins"])
    if deposits > 2.0e10 or points > 2.0e9:
        return None
    if kind == "in_situ":
        r0, u0, laser, t0, t1 = _push_inputs(case, seed)
        inputs = _push64(r0, u0, laser, t0, t1, case["n_s"])
        ta = [t_ - (r_ @ n_hat.T) / C0 for t_, r_ in ((t0, inputs[1][:, 0]), (t1, inputs[1][:, -1]))]
        grid = lw.grid_from_bounds(float(ta[0].min()), float(ta[1].max()), case["n_bins"])
        rec = _deposit64(inputs, n_hat, grid)
        out = rec
        if case["prec"] == "f32x4":
            out = torch.zeros(rec.shape[0], rec.shape[2], 4, dtype=torch.float64, device="cuda")
            out[..., :3] = rec.permute(0, 2, 1)
        return {"S": _spectrum64(rec, grid.dt_u), "t_min": grid.t_min, "dt_u": grid.dt_u,
                "record": out}
    inputs = _trajectories(b, case["n_e"], case["n_s"], seed)
    traj = lw.lw_trajectories_upload(*inputs, sections=lw.LW_SECTION_FP64)
    grid = _grid(traj, det, case["n_bins"])
    if kind == "step":
        return {"S": _spectrum64(_deposit64(inputs, n_hat, grid), grid.dt_u), "status": None}
    rec = _deposit64(inputs, n_hat, grid, case["velocity"], 1.0)
    if case["prec"] == "kahan":   # the value is sum + compensation: no value for either word
        return None
    if case["prec"] == "f32x4":
        out = torch.zeros(rec.shape[0], rec.shape[2], 4, dtype=torch.float64, device="cuda")
        out[..., :3] = rec.permute(0, 2, 1)
        rec = out
    return {"record": rec, "status": None}
