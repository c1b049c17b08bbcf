// Boris pusher on the GPU (FP64), the trajectory update of Algorithm 2 ("update
// trajectory" in the step loop), for the in-situ form of the time-domain path:
// trajectories are produced one block of steps at a time and deposited at once,
// so only the current block is ever stored.  The same step, differentiated in
// forward mode, gives the gradient of a loss of the samples with respect to the
// initial momenta and the laser's a0 and waist.
//
// Laser: lowest-order paraxial Gaussian beam polarised along x, propagating
// along -z, focused at z = 0 and peaking there at t = 0:
//   E_x = E0 (w0/w) exp(-rho^2/w^2) exp(-(t + z/c)^2/(2 sigma^2))
//         cos(omega (t + z/c) + k rho^2 zeta/(2 (zeta^2 + zR^2)) - atan(zeta/zR)),
//   B_y = -E_x/c0,  zeta = -z,  w = w0 sqrt(1 + zeta^2/zR^2),  zR = pi w0^2/lam,
//   E0 = a0 m c0 omega / e,  sigma = FWHM_intensity / (2 sqrt(ln 2)).
// Step: drift half a step, Boris kick (half electric, magnetic rotation, half
// electric) with the fields at the midpoint, drift half a step; samples hold
// (t, r, beta, beta_dot) with beta_dot the Lorentz-force derivative
//   beta_dot = q/(m gamma c0) [E + c0 beta x B - beta (beta . E)].
#include <math.h>

#include "lw_internal.cuh"

namespace lw {
namespace {

constexpr double kQe = 1.602176634e-19;
constexpr double kMe = 9.1093837015e-31;

// Laser constants of the push.
struct Laser {
    double omega, k, sigma, E0, zR, w0;
};

// ------------------------------------------------------------------ the push
//
// What bounds it: FP64 issue along one chain per electron.  On GB300 one FP64 warp
// instruction occupies its SM sub-partition for 64 cycles, whether or not it depends on the
// one before and however many lanes are active (four busy sub-partitions: 19 cycles per
// instruction and SM), so a step takes the number of FP64 instructions on its longest chain
// within one warp.  A CTA is therefore four warps, one per sub-partition, over the same 32
// electrons, and the step is cut along its data flow:
//   warp 0   phase, cosine, kick, z of the second half drift (the chain);
//   warp 1   the next step's first half drift K v / gamma, beside the second half drift of
//            warps 0 and 2, and the Gouy phase atan(zeta/zR) of the midpoint;
//   warp 2   the midpoint's transverse profile exp(-rho^2/w^2) and amplitude E0 w0/w, and x
//            and y of the second half drift;
//   warp 3   its temporal profile exp(-xi^2/(2 sigma^2)), then the sample (beta, beta_dot) of
//            the state the step started from.
// Positions and momenta are rounded operation by operation as the step was before it was cut
// up: a position's last bit can move a grid point across a sample, which a gradient of the
// spectrum feels.  That fixes where products are fused into sums (gamma of the first half drift
// and of the kick adds rounded squares, gamma of the second half drift fuses them).  A square
// root and the quotients by it share one reciprocal square root, with a residual correction
// for each correctly rounded result; zeta/zR uses the host's reciprocal the same way.  Only
// the samples' beta and beta_dot use a shorter form (beam_value()).
// One warp per 32 electrons doing all of it took 15.7 us per step (1,500 electrons, 10,000
// steps: 157 ms); cut this way it takes 5.0 us (50 ms).
struct Beam {
    double inv_zR, inv_w02, inv_2s2;   // 1/zR, 1/w0^2, 1/(2 sigma^2)
    double om_pi, kz_pi;               // omega/pi, k/(2 pi zR)
    double E0;
};

// E_x / E0 in the form
//   U = exp(-rho^2/(w0^2 q) - xi^2/(2 sigma^2)) (cos phi + s sin phi) / q,
//   s = zeta/zR, q = 1 + s^2, phi = omega xi + k rho^2 s / (2 zR q), xi = t + z/c0,
// from w^2 = w0^2 q and cos(phi - atan s) = (cos phi + s sin phi) / sqrt(q): one exponential,
// one reciprocal and no arc tangent or square root.
struct BeamValue {
    double s, iq, g, xi;    // zeta/zR, 1/q, rho^2/q, xi
    double A, sn, cs;       // exp(...)/q, sin phi, cos phi
};
__device__ __forceinline__ BeamValue beam_value(const Beam& B, double x, double y, double z,
                                                double t) {
    BeamValue b;
    b.s = -z * B.inv_zR;
    b.iq = 1.0 / fma(b.s, b.s, 1.0);
    b.g = fma(x, x, y * y) * b.iq;
    b.xi = fma(z, kInvC0, t);
    b.A = b.iq * exp(-fma(b.g, B.inv_w02, b.xi * b.xi * B.inv_2s2));
    sincospi(fma(B.om_pi, b.xi, B.kz_pi * (b.g * b.s)), &b.sn, &b.cs);
    return b;
}
__device__ __forceinline__ double beam_unit(const BeamValue& b) { return b.A * fma(b.s, b.sn, b.cs); }

// n / d rounded as the division rounds it, given the reciprocal r of d to an ulp: residual correction
// (Markstein), exact while n and the quotient are above 2^-960 in size, 2^-105 of the quotient before
// the last rounding.  Below that (a momentum component of 1e-289) last bits of the quotient differ.
__device__ __forceinline__ double quotient(double n, double d, double r) {
    const double q = __dmul_rn(n, r);
    return fma(fma(-q, d, n), r, q);
}

// gamma = sqrt(a), rounded as the square root rounds it, and its reciprocal to an ulp (a = 1 + u^2 >= 1;
// an infinite or NaN a ends as NaN): residual correction from a reciprocal root good to an ulp
// (Markstein; tests/test_rounding_model.py has its steps)
__device__ __forceinline__ double root(double a, double& inv) {
    const double y = rsqrt(a);
    const double g = __dmul_rn(a, y);
    const double gam = fma(fma(-g, g, a), 0.5 * y, g);
    inv = fma(fma(-gam, y, 1.0), y, y);
    return gam;
}

// 1 + u^2 with every square fused, and with the y and z squares rounded first
__device__ __forceinline__ double gamma2_fused(double u0, double u1, double u2) {
    return fma(u2, u2, fma(u1, u1, fma(u0, u0, 1.0)));
}
__device__ __forceinline__ double gamma2_sum(double u0, double u1, double u2) {
    return __dadd_rn(__dadd_rn(fma(u0, u0, 1.0), __dmul_rn(u1, u1)), __dmul_rn(u2, u2));
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
    __syncwarp();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

constexpr int kPushThreads = 128;
// named barriers of a step: momentum published (warp 0 -> 1, 2), first half drift (1 -> 0, 2),
// midpoint and state published (all four warps), Gouy phase (1 -> 0), profiles (2, 3 -> 0)
enum { kBarKick = 1, kBarDrift = 2, kBarState = 3, kBarGouy = 4, kBarProfile = 5 };

__global__ void __launch_bounds__(kPushThreads)
    push_kernel(double* __restrict__ r, double* __restrict__ u, int64_t n_e, double t0, double dt,
                int64_t step0, int n_steps, Laser L, Beam B, double qm,
                double* __restrict__ t_out, double* __restrict__ ro, double* __restrict__ bo,
                double* __restrict__ ao) {
    // two slots by the parity of the step: a slot is rewritten only after the barrier of the
    // step in between, which every reader passes after its reads
    __shared__ double s_mid[2][3][32];    // midpoint of the step
    __shared__ double s_st[2][6][32];     // state the step starts from
    __shared__ double s_part[2][4][32];   // atan, transverse profile, amplitude, temporal profile
    __shared__ double s_q[2][3][32];      // K v / gamma of the first half drift
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t k = blockIdx.x * (int64_t)32 + lane;
    const int64_t kc = k < n_e ? k : n_e - 1;   // lanes past the end repeat the last electron
    const double hdt = 0.5 * dt;
    const double K = hdt * kC0;
    if (warp == 0) {
        const double eps = qm * dt / (2.0 * kC0), qdt = qm * dt;
        const double zR2 = L.zR * L.zR;
        double z = r[3 * kc + 2];
        double v[3] = {u[3 * kc], u[3 * kc + 1], u[3 * kc + 2]};
        for (int c = 0; c < 3; ++c) s_st[0][3 + c][lane] = v[c];
        bar_arrive(kBarKick, 96);
        for (int s = 0;; ++s) {
            const int p = s & 1;
            const double tm = fma(dt, (double)(step0 + s), t0) + hdt;
            s_st[p][2][lane] = z;
            bar_sync(kBarDrift, 96);
            z = __dadd_rn(z, s_q[p][2][lane]);
            s_mid[p][2][lane] = z;
            bar_sync(kBarState, kPushThreads);
            if (s == n_steps) break;
            const double x = s_mid[p][0][lane], y = s_mid[p][1][lane];
            const double rho2 = fma(x, x, __dmul_rn(y, y));
            const double xi = fma(z, kInvC0, tm);
            const double curv = __dmul_rn(__dmul_rn(L.k, rho2), -z) / (2.0 * fma(z, z, zR2));
            const double ph = fma(L.omega, xi, curv);
            bar_sync(kBarGouy, 64);
            const double cs = cos(__dsub_rn(ph, s_part[p][0][lane]));
            bar_sync(kBarProfile, 96);
            const double env = __dmul_rn(s_part[p][1][lane], s_part[p][3][lane]);
            const double Ex = __dmul_rn(__dmul_rn(s_part[p][2][lane], env), cs);
            const double By = -__dmul_rn(Ex, kInvC0);
            const double um = fma(eps, Ex, v[0]);
            double igm;
            const double gm = root(gamma2_sum(um, v[1], v[2]), igm);
            const double tv = __dmul_rn(quotient(qdt, 2.0 * gm, 0.5 * igm), By);
            // rotation about y: u' = um + um x t, u+ = um + u' x s, s = 2 t / (1 + t^2)
            const double up0 = fma(-v[2], tv, um), up2 = fma(um, tv, v[2]);
            const double sv = 2.0 * tv / fma(tv, tv, 1.0);
            v[0] = fma(eps, Ex, fma(-up2, sv, um));
            v[2] = fma(up0, sv, v[2]);
            s_st[p ^ 1][3][lane] = v[0];
            s_st[p ^ 1][4][lane] = v[1];
            s_st[p ^ 1][5][lane] = v[2];
            bar_arrive(kBarKick, 96);
            double ig;
            const double gam = root(gamma2_fused(v[0], v[1], v[2]), ig);
            z = __dadd_rn(z, quotient(__dmul_rn(K, v[2]), gam, ig));
        }
        if (k < n_e) {
            r[3 * k + 2] = s_st[n_steps & 1][2][lane];
            for (int c = 0; c < 3; ++c) u[3 * k + c] = v[c];
        }
    } else if (warp == 1) {
        const double izR = 1.0 / L.zR;
        for (int s = 0; s <= n_steps; ++s) {
            const int p = s & 1;
            bar_sync(kBarKick, 96);
            const double v0 = s_st[p][3][lane], v1 = s_st[p][4][lane], v2 = s_st[p][5][lane];
            double ig;
            const double gam = root(gamma2_sum(v0, v1, v2), ig);
            s_q[p][2][lane] = quotient(__dmul_rn(K, v2), gam, ig);
            s_q[p][0][lane] = quotient(__dmul_rn(K, v0), gam, ig);
            s_q[p][1][lane] = quotient(__dmul_rn(K, v1), gam, ig);
            bar_arrive(kBarDrift, 96);
            bar_sync(kBarState, kPushThreads);
            if (s < n_steps) {
                s_part[p][0][lane] = atan(quotient(-s_mid[p][2][lane], L.zR, izR));
                bar_arrive(kBarGouy, 64);
            }
        }
    } else if (warp == 2) {
        const double izR = 1.0 / L.zR;
        double x = r[3 * kc], y = r[3 * kc + 1];
        bar_sync(kBarKick, 96);
        for (int s = 0;; ++s) {
            const int p = s & 1;
            s_st[p][0][lane] = x;
            s_st[p][1][lane] = y;
            bar_sync(kBarDrift, 96);
            x = __dadd_rn(x, s_q[p][0][lane]);
            y = __dadd_rn(y, s_q[p][1][lane]);
            s_mid[p][0][lane] = x;
            s_mid[p][1][lane] = y;
            bar_sync(kBarState, kPushThreads);
            if (s == n_steps) break;
            const double zn = quotient(-s_mid[p][2][lane], L.zR, izR);
            double iw;
            const double w = __dmul_rn(L.w0, root(fma(zn, zn, 1.0), iw));
            s_part[p][1][lane] = exp(-fma(x, x, __dmul_rn(y, y)) / __dmul_rn(w, w));
            s_part[p][2][lane] = __dmul_rn(L.E0, L.w0 / w);
            bar_arrive(kBarProfile, 96);
            bar_sync(kBarKick, 96);
            const double v0 = s_st[p ^ 1][3][lane], v1 = s_st[p ^ 1][4][lane];
            double ig;
            const double gam = root(gamma2_fused(v0, v1, s_st[p ^ 1][5][lane]), ig);
            x = __dadd_rn(x, quotient(__dmul_rn(K, v0), gam, ig));
            y = __dadd_rn(y, quotient(__dmul_rn(K, v1), gam, ig));
        }
        if (k < n_e) {
            r[3 * k] = s_st[n_steps & 1][0][lane];
            r[3 * k + 1] = s_st[n_steps & 1][1][lane];
        }
    } else {
        const double two_s2 = 2.0 * L.sigma * L.sigma;
        const double f0 = qm / kC0;
        const int64_t base = 3 * kc * (int64_t)(n_steps + 1);
        for (int s = 0; s <= n_steps; ++s) {
            const int p = s & 1;
            const double t = fma(dt, (double)(step0 + s), t0);
            bar_sync(kBarState, kPushThreads);
            if (s < n_steps) {
                const double xi = fma(s_mid[p][2][lane], kInvC0, t + hdt);
                s_part[p][3][lane] = exp(-__dmul_rn(xi, xi) / two_s2);
                bar_arrive(kBarProfile, 96);
            }
            const double x = s_st[p][0][lane], y = s_st[p][1][lane], z = s_st[p][2][lane];
            const double u0 = s_st[p][3][lane], u1 = s_st[p][4][lane], u2 = s_st[p][5][lane];
            const double ig = rsqrt(fma(u2, u2, fma(u1, u1, fma(u0, u0, 1.0))));
            const double b0 = u0 * ig, b1 = u1 * ig, b2 = u2 * ig;
            // E = (Ex, 0, 0), c0 B = (0, -Ex, 0):
            // E + c0 beta x B - beta (beta . E) = Ex (1 + b_z - b_x^2, -b_x b_y, -b_x (1 + b_z))
            const double f = f0 * ig * (B.E0 * beam_unit(beam_value(B, x, y, z, t)));
            const double g = f * b0, h = 1.0 + b2;
            if (k < n_e) {
                const int64_t o = base + 3 * (int64_t)s;
                ro[o] = x;
                ro[o + 1] = y;
                ro[o + 2] = z;
                bo[o] = b0;
                bo[o + 1] = b1;
                bo[o + 2] = b2;
                ao[o] = fma(f, h, -g * b0);
                ao[o + 1] = -g * b1;
                ao[o + 2] = -g * h;
                if (k == 0) t_out[s] = t;
            }
        }
    }
}

// ------------------------------------------------------------------ its gradient
//
// Gradient of a loss L(samples) with respect to each electron's initial momentum u0 and the
// laser's a0 and w0, in forward mode: the derivative of an electron's state along u0_x, u0_y,
// u0_z, a0 and w0 is carried through the push and contracted with dL/d(r, beta, beta_dot) of
// every sample.  Bound as the push is: FP64 instructions of the busiest warp.  Everything that
// the five directions share is computed once per electron, by the warps of a CTA over the same
// 32 electrons, as a pipeline over the steps with one barrier per step (ring of four slots):
//   warp 0   the push itself (step n);
//   warp 1   the sample's adjoint (sample n): dL/d(sample) pulled back to the state and the
//            laser, W . (dx, du, da0, dw0);
//   warp 2   directions a0 and w0 (step n - 2), and the gradient of the field at the midpoint
//            (step n - 1);
//   warp 3   directions u0_x, u0_y, u0_z (step n - 2).
// A direction costs 33 operations per step (the step linearised with coefficients from warps 0
// and 2) and 6 for the contraction.  One thread per electron and direction, each pushing the
// electron again in derivative numbers, took 26.6 us per step (2,048 electrons x 4,096 steps:
// 109 ms); this form 4.6 us (19.0 ms).

// Gradient of E_x = E0 U with respect to (x, y, z), and along a0 and w0.
struct BeamGrad {
    double x, y, z, a0, w0;
};
struct TanLaser {   // constants of the gradient
    double kz, om_c, inv_s2c, e0_per_a0, two_over_w0;   // k/(2 zR), omega/c0, 1/(sigma^2 c0)
};
// With A the amplitude, P = dE/dphi and g = rho^2/q: dE = Cg dg + Cs ds + (P omega - E xi/sigma^2)
// dxi, where dg = 2 (x dx + y dy)/q - 2 s g ds/q is already part of Cs; zR varies as w0^2.
__device__ __forceinline__ BeamGrad beam_grad(const Beam& B, const TanLaser& T,
                                              const BeamValue& b, double x, double y) {
    const double U = beam_unit(b), E = B.E0 * U, a = B.E0 * b.A;
    const double P = a * fma(b.s, b.cs, -b.sn);
    const double Pk = P * T.kz;
    const double Ew = E * B.inv_w02;
    const double Cg = fma(Pk, b.s, -Ew);
    const double Cs = fma(Pk, b.g, fma(a, b.sn, -2.0 * b.s * b.iq * fma(Cg, b.g, E)));
    const double c2 = 2.0 * Cg * b.iq;
    BeamGrad G;
    G.x = c2 * x;
    G.y = c2 * y;
    G.z = fma(P, T.om_c, fma(-E * b.xi, T.inv_s2c, -Cs * B.inv_zR));
    G.a0 = T.e0_per_a0 * U;
    G.w0 = T.two_over_w0 * fma(Ew, b.g, -b.s * fma(Pk, b.g, Cs));
    return G;
}

constexpr int kTanThreads = 128;
constexpr int kTanSlots = 4;
// one slot of the ring (doubles per electron)
enum {
    kX = 0, kV = 3, kIg = 6,                     // state n (x, u, 1/gamma)
    kMx = 7, kMy, kBs, kBiq, kBg, kBxi, kBA, kBsn, kBcs,   // midpoint of step n
    kUm = 16, kTa, kTb, kTr, kRc, kRs, kV0r,     // kick of step n
    kG = 23,                                     // field gradient of step n (x, y, z, a0, w0)
    kW = 28,                                     // adjoint of sample n (x, u, a0, w0)
    kSlotVals = 36
};

__global__ void __launch_bounds__(kTanThreads)
    push_tangent_kernel(const double* __restrict__ r0, const double* __restrict__ u0, int64_t n_e,
                        double t0, double dt, int n_steps, Beam B, TanLaser T, double qm,
                        const double* __restrict__ g_r, const double* __restrict__ g_b,
                        const double* __restrict__ g_a, double* __restrict__ dL_du0,
                        double* __restrict__ dL_dlaser) {
    __shared__ double s_ring[kTanSlots][kSlotVals][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t k = blockIdx.x * (int64_t)32 + lane;
    const int64_t kc = k < n_e ? k : n_e - 1;   // lanes past the end repeat the last electron
    const double kd = 0.5 * dt * kC0, eps = qm * dt / (2.0 * kC0);
    auto at = [&](int n, int i) -> double& { return s_ring[n & (kTanSlots - 1)][i][lane]; };
    auto inv_gamma = [](const double (&u)[3]) {
        return rsqrt(fma(u[2], u[2], fma(u[1], u[1], fma(u[0], u[0], 1.0))));
    };
    // warp 0: state of the step; warp 1: the next sample's dL/d(sample)
    double x[3], v[3], ig = 1.0;
    double g[9];
    // warps 2 and 3: state derivatives of up to three directions, their half drifts' delta and sums
    constexpr int kDirs = 3;
    double dx[kDirs][3], dv[kDirs][3], de[kDirs][3], acc[kDirs];
    const int n_dir = warp == 2 ? 2 : 3;
    if (warp == 0) {
        for (int c = 0; c < 3; ++c) {
            x[c] = r0[3 * kc + c];
            v[c] = u0[3 * kc + c];
            at(0, kX + c) = x[c];
            at(0, kV + c) = v[c];
        }
        ig = inv_gamma(v);
        at(0, kIg) = ig;
    }
    auto load_g = [&](int n) {   // dL/d(sample n)
        const int64_t o = 3 * (kc * (int64_t)(n_steps + 1) + n);
        for (int c = 0; c < 3; ++c) {
            g[c] = g_r[o + c];
            g[3 + c] = g_b[o + c];
            g[6 + c] = g_a[o + c];
        }
    };
    if (warp == 1) load_g(0);
    for (int d = 0; d < kDirs; ++d) {
        acc[d] = 0.0;
        for (int c = 0; c < 3; ++c) {
            dx[d][c] = de[d][c] = 0.0;
            dv[d][c] = warp == 3 && d == c ? 1.0 : 0.0;
        }
    }
    __syncthreads();
    // delta of a half drift, d(K u/gamma) = K/gamma du - K/gamma^3 (u . du) u, at state n
    auto half_drift = [&](int n) {
        const double i1 = at(n, kIg), c1 = kd * i1, c2 = c1 * i1 * i1;
        const double w0 = at(n, kV), w1 = at(n, kV + 1), w2 = at(n, kV + 2);
#pragma unroll
        for (int d = 0; d < kDirs; ++d) {
            if (d >= n_dir) break;
            const double w = -c2 * fma(w2, dv[d][2], fma(w1, dv[d][1], w0 * dv[d][0]));
            de[d][0] = fma(c1, dv[d][0], w * w0);
            de[d][1] = fma(c1, dv[d][1], w * w1);
            de[d][2] = fma(c1, dv[d][2], w * w2);
        }
    };
    if (warp >= 2) half_drift(0);

    for (int it = 0; it <= n_steps + 2; ++it) {
        if (warp == 0) {
            if (it < n_steps) {   // step it: drift, kick, drift, as the push
                const double d = kd * ig;
                const double h0 = fma(v[0], d, x[0]), h1 = fma(v[1], d, x[1]),
                             h2 = fma(v[2], d, x[2]);
                const BeamValue b = beam_value(B, h0, h1, h2, fma(dt, (double)it + 0.5, t0));
                at(it, kMx) = h0;
                at(it, kMy) = h1;
                at(it, kBs) = b.s;
                at(it, kBiq) = b.iq;
                at(it, kBg) = b.g;
                at(it, kBxi) = b.xi;
                at(it, kBA) = b.A;
                at(it, kBsn) = b.sn;
                at(it, kBcs) = b.cs;
                const double e = eps * (B.E0 * beam_unit(b));
                const double um[3] = {v[0] + e, v[1], v[2]};
                const double igm = inv_gamma(um);
                // rotation in the (z, x) plane by theta, tan(theta/2) = tv
                const double tv = -e * igm;
                const double rr = 2.0 / fma(tv, tv, 1.0);
                const double sn = rr * tv, cs = fma(-tv, sn, 1.0);
                const double v0r = fma(cs, um[0], -sn * v[2]);
                at(it, kUm) = um[0];
                at(it, kTa) = -eps * igm;          // dtv = kTa dE - kTb (um . dum)
                at(it, kTb) = tv * igm * igm;
                at(it, kTr) = rr;
                at(it, kRc) = cs;
                at(it, kRs) = sn;
                at(it, kV0r) = v0r;
                v[2] = fma(cs, v[2], sn * um[0]);
                v[0] = v0r + e;
                ig = inv_gamma(v);
                const double d2 = kd * ig;
                x[0] = fma(v[0], d2, h0);
                x[1] = fma(v[1], d2, h1);
                x[2] = fma(v[2], d2, h2);
                for (int c = 0; c < 3; ++c) {
                    at(it + 1, kX + c) = x[c];
                    at(it + 1, kV + c) = v[c];
                }
                at(it + 1, kIg) = ig;
            }
        } else if (warp == 1) {
            if (it <= n_steps) {   // sample it: psi = g_r . r + g_b . beta + g_a . beta_dot
                const double gr[3] = {g[0], g[1], g[2]}, gb[3] = {g[3], g[4], g[5]},
                             ga[3] = {g[6], g[7], g[8]};
                if (it < n_steps) load_g(it + 1);
                const double sx = at(it, kX), sy = at(it, kX + 1), sz = at(it, kX + 2);
                const double u_0 = at(it, kV), u_1 = at(it, kV + 1), u_2 = at(it, kV + 2);
                const double i1 = at(it, kIg);
                const BeamValue b = beam_value(B, sx, sy, sz, fma(dt, (double)it, t0));
                const BeamGrad G = beam_grad(B, T, b, sx, sy);
                const double b0 = u_0 * i1, b1 = u_1 * i1, b2 = u_2 * i1, h = 1.0 + b2;
                // beta_dot = f (h - b0^2, -b0 b1, -b0 h), f = q/(m c0) E / gamma
                const double fe = qm / kC0 * i1, f = fe * (B.E0 * beam_unit(b));
                const double m = fma(ga[1], b1, ga[2] * h);
                const double y = fma(ga[0], fma(-b0, b0, h), -b0 * m);   // dpsi/df
                const double q = fe * y;                                  // dpsi/dE
                const double B0 = fma(f, fma(-2.0 * b0, ga[0], -m), gb[0]);
                const double B1 = fma(-f * b0, ga[1], gb[1]);
                const double B2 = fma(f, fma(-b0, ga[2], ga[0]), gb[2]);
                // 1/gamma enters beta = u/gamma and f: d(1/gamma) = -(1/gamma)^2 beta . du
                const double ki = fma(f, y, fma(B2, b2, fma(B1, b1, B0 * b0)));
                at(it, kW) = fma(q, G.x, gr[0]);
                at(it, kW + 1) = fma(q, G.y, gr[1]);
                at(it, kW + 2) = fma(q, G.z, gr[2]);
                at(it, kW + 3) = i1 * fma(-ki, b0, B0);
                at(it, kW + 4) = i1 * fma(-ki, b1, B1);
                at(it, kW + 5) = i1 * fma(-ki, b2, B2);
                at(it, kW + 6) = q * G.a0;
                at(it, kW + 7) = q * G.w0;
            }
        } else {
            if (warp == 2 && it >= 1 && it - 1 < n_steps) {
                const int n = it - 1;
                BeamValue b;
                b.s = at(n, kBs);
                b.iq = at(n, kBiq);
                b.g = at(n, kBg);
                b.xi = at(n, kBxi);
                b.A = at(n, kBA);
                b.sn = at(n, kBsn);
                b.cs = at(n, kBcs);
                const BeamGrad G = beam_grad(B, T, b, at(n, kMx), at(n, kMy));
                at(n, kG) = G.x;
                at(n, kG + 1) = G.y;
                at(n, kG + 2) = G.z;
                at(n, kG + 3) = G.a0;
                at(n, kG + 4) = G.w0;
            }
            const int n = it - 2;
            if (n >= 0) {
                const double W0 = at(n, kW), W1 = at(n, kW + 1), W2 = at(n, kW + 2);
                const double W3 = at(n, kW + 3), W4 = at(n, kW + 4), W5 = at(n, kW + 5);
#pragma unroll
                for (int d = 0; d < kDirs; ++d) {
                    if (d >= n_dir) break;
                    if (warp == 2) acc[d] += at(n, kW + 6 + d);
                    acc[d] = fma(W0, dx[d][0], fma(W1, dx[d][1], fma(W2, dx[d][2], acc[d])));
                    acc[d] = fma(W3, dv[d][0], fma(W4, dv[d][1], fma(W5, dv[d][2], acc[d])));
                }
                if (n < n_steps) {
                    const double Gx = at(n, kG), Gy = at(n, kG + 1), Gz = at(n, kG + 2);
                    const double um = at(n, kUm), ta = at(n, kTa), tb = at(n, kTb);
                    const double rr = at(n, kTr), cs = at(n, kRc), sn = at(n, kRs);
                    const double v0r = at(n, kV0r), v1 = at(n, kV + 1), v2 = at(n, kV + 2);
                    const double v2n = at(n + 1, kV + 2);
#pragma unroll
                    for (int d = 0; d < kDirs; ++d) {
                        if (d >= n_dir) break;
                        for (int c = 0; c < 3; ++c) dx[d][c] += de[d][c];   // midpoint
                        double dE = Gx * dx[d][0];
                        if (warp == 2) dE += at(n, kG + 3 + d);
                        dE = fma(Gz, dx[d][2], fma(Gy, dx[d][1], dE));
                        const double dum = fma(eps, dE, dv[d][0]);
                        const double dot = fma(v2, dv[d][2], fma(v1, dv[d][1], um * dum));
                        const double dth = rr * fma(ta, dE, -tb * dot);
                        dv[d][0] = fma(eps, dE, fma(-v2n, dth, fma(-sn, dv[d][2], cs * dum)));
                        dv[d][2] = fma(v0r, dth, fma(cs, dv[d][2], sn * dum));
                    }
                    half_drift(n + 1);
#pragma unroll
                    for (int d = 0; d < kDirs; ++d)
                        for (int c = 0; c < 3; ++c) dx[d][c] += de[d][c];
                }
            }
        }
        __syncthreads();   // slots it and it + 1 are readable, slot it - 2 is free
    }
    if (warp == 3 && k < n_e)
        for (int c = 0; c < 3; ++c) dL_du0[3 * k + c] += acc[c];
    if (warp == 2)
        for (int d = 0; d < 2; ++d) {
            double a = k < n_e ? acc[d] : 0.0;
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (lane == 0) atomicAdd(dL_dlaser + d, a);
        }
}

Laser laser_constants(const lw_laser& l) {
    Laser L;
    L.omega = 2.0 * kPi * kC0 / l.lam;
    L.k = L.omega * kInvC0;
    L.sigma = l.fwhm / (2.0 * sqrt(log(2.0)));
    L.E0 = l.a0 * kMe * kC0 * L.omega / kQe;
    // finite, so that zeta/zR by its reciprocal is (a plane wave given as a huge waist; the product
    // overflows from w0 = 1e151 on): at 1e300 zeta/zR and its square add nothing
    L.zR = fmin(kPi * l.w0 * l.w0 / l.lam, 1.0e300);
    L.w0 = l.w0;
    return L;
}

Beam beam_constants(const Laser& L) {
    Beam B;
    B.inv_zR = 1.0 / L.zR;
    B.inv_w02 = 1.0 / (L.w0 * L.w0);
    B.inv_2s2 = 1.0 / (2.0 * L.sigma * L.sigma);
    B.om_pi = L.omega / kPi;
    B.kz_pi = L.k / (2.0 * kPi * L.zR);
    B.E0 = L.E0;
    return B;
}

}  // namespace
}  // namespace lw

using namespace lw;

extern "C" int lw_boris_push(double* r, double* u, int64_t n_e, double t0, double dt,
                             int64_t step0, int32_t n_steps, const lw_laser* laser,
                             double charge, double mass,
                             double* t_out, double* r_out, double* beta_out, double* bdot_out,
                             void* stream) {
    if (!r || !u || !laser || !t_out || !r_out || !beta_out || !bdot_out) return LW_EINVAL;
    if (n_e < 1 || n_steps < 1 || step0 < 0 || step0 > (int64_t(1) << 52) || !(dt > 0.0) ||
        !isfinite(t0) || !(mass > 0.0))
        return LW_EINVAL;
    if (!(laser->lam > 0.0) || !(laser->w0 > 0.0) || !(laser->fwhm > 0.0)) return LW_EINVAL;
    const Laser L = laser_constants(*laser);
    const Beam B = beam_constants(L);
    const int blocks = (int)((n_e + 31) / 32);
    push_kernel<<<blocks, kPushThreads, 0, as_stream(stream)>>>(
        r, u, n_e, t0, dt, step0, n_steps, L, B, charge / mass, t_out, r_out, beta_out, bdot_out);
    return launch_status();
}

extern "C" int lw_boris_push_grad(const double* r0, const double* u0, int64_t n_e, double t0,
                                  double dt, int32_t n_steps, const lw_laser* laser,
                                  double charge, double mass, const double* dL_dr,
                                  const double* dL_dbeta, const double* dL_dbeta_dot,
                                  double* dL_du0, double* dL_dlaser, void* stream) {
    if (!r0 || !u0 || !laser || !dL_dr || !dL_dbeta || !dL_dbeta_dot || !dL_du0 || !dL_dlaser)
        return LW_EINVAL;
    if (n_e < 1 || n_steps < 1 || !(dt > 0.0) || !isfinite(t0) || !(mass > 0.0))
        return LW_EINVAL;
    if (!(laser->lam > 0.0) || !(laser->w0 > 0.0) || !(laser->fwhm > 0.0)) return LW_EINVAL;
    const Laser L = laser_constants(*laser);
    TanLaser T;
    T.kz = L.k / (2.0 * L.zR);
    T.om_c = L.omega * kInvC0;
    T.inv_s2c = kInvC0 / (L.sigma * L.sigma);
    T.e0_per_a0 = kMe * kC0 * L.omega / kQe;
    T.two_over_w0 = 2.0 / L.w0;
    const int blocks = (int)((n_e + 31) / 32);
    push_tangent_kernel<<<blocks, kTanThreads, 0, as_stream(stream)>>>(
        r0, u0, n_e, t0, dt, n_steps, beam_constants(L), T, charge / mass, dL_dr, dL_dbeta,
        dL_dbeta_dot, dL_du0, dL_dlaser);
    return launch_status();
}
