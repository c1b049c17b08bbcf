// Boris pusher on the GPU (FP64), the trajectory update of Algorithm 2 ("update
// trajectory" in the step loop), for the in-situ form of the time-domain path:
// trajectories are produced one block of steps at a time and deposited at once,
// so only the current block is ever stored.  The same step, carried out on
// forward-mode derivative numbers, gives the gradient of a loss of the samples
// with respect to the initial momenta and the laser's a0 and waist.
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

using ::atan;
using ::cos;
using ::exp;
using ::sqrt;

// Forward-mode derivative numbers: a value and its derivatives along N directions.
template <int N>
struct Dual {
    double v;
    double d[N];
};
template <int N>
__device__ __forceinline__ Dual<N> mk(double v) {
    Dual<N> r;
    r.v = v;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = 0.0;
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> operator+(const Dual<N>& a, const Dual<N>& b) {
    Dual<N> r;
    r.v = a.v + b.v;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = a.d[i] + b.d[i];
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> operator-(const Dual<N>& a, const Dual<N>& b) {
    Dual<N> r;
    r.v = a.v - b.v;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = a.d[i] - b.d[i];
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> operator-(const Dual<N>& a) {
    Dual<N> r;
    r.v = -a.v;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = -a.d[i];
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> operator*(const Dual<N>& a, const Dual<N>& b) {
    Dual<N> r;
    r.v = a.v * b.v;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * b.v + a.v * b.d[i];
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> operator/(const Dual<N>& a, const Dual<N>& b) {
    Dual<N> r;
    r.v = a.v / b.v;
    const double ib = 1.0 / b.v;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = (a.d[i] - r.v * b.d[i]) * ib;
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> operator+(const Dual<N>& a, double b) {
    Dual<N> r = a;
    r.v = a.v + b;
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> operator+(double a, const Dual<N>& b) { return b + a; }
template <int N>
__device__ __forceinline__ Dual<N> operator-(const Dual<N>& a, double b) { return a + (-b); }
template <int N>
__device__ __forceinline__ Dual<N> operator-(double a, const Dual<N>& b) { return (-b) + a; }
template <int N>
__device__ __forceinline__ Dual<N> operator*(const Dual<N>& a, double b) {
    Dual<N> r;
    r.v = a.v * b;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * b;
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> operator*(double a, const Dual<N>& b) { return b * a; }
template <int N>
__device__ __forceinline__ Dual<N> operator/(const Dual<N>& a, double b) { return a * (1.0 / b); }
template <int N>
__device__ __forceinline__ Dual<N> operator/(double a, const Dual<N>& b) { return mk<N>(a) / b; }
template <int N>
__device__ __forceinline__ Dual<N> sqrt(const Dual<N>& a) {
    Dual<N> r;
    r.v = sqrt(a.v);
    const double h = 0.5 / r.v;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * h;
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> exp(const Dual<N>& a) {
    Dual<N> r;
    r.v = exp(a.v);
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * r.v;
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> cos(const Dual<N>& a) {
    Dual<N> r;
    double sn, cs;
    sincos(a.v, &sn, &cs);
    r.v = cs;
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = -a.d[i] * sn;
    return r;
}
template <int N>
__device__ __forceinline__ Dual<N> atan(const Dual<N>& a) {
    Dual<N> r;
    r.v = atan(a.v);
    const double h = 1.0 / (1.0 + a.v * a.v);
#pragma unroll
    for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * h;
    return r;
}

// Laser constants (T = double, or Dual when derivatives along a0 and w0 are carried).
template <typename T>
struct LaserT {
    double omega, k, sigma;
    T E0, zR, w0;
};
using Laser = LaserT<double>;

template <typename T>
__device__ __forceinline__ void fields(const LaserT<T>& L, const T& x, const T& y, const T& z,
                                       double t, T& Ex, T& By) {
    const T zeta = -z;
    const T w = L.w0 * sqrt(1.0 + (zeta / L.zR) * (zeta / L.zR));
    const T rho2 = x * x + y * y;
    const T xi = t + z * kInvC0;
    const T env = exp(-rho2 / (w * w)) * exp(-(xi * xi) / (2.0 * L.sigma * L.sigma));
    const T phase =
        L.omega * xi + L.k * rho2 * zeta / (2.0 * (zeta * zeta + L.zR * L.zR)) - atan(zeta / L.zR);
    Ex = L.E0 * (L.w0 / w) * env * cos(phase);
    By = -Ex * kInvC0;
}

// The sample at (r, u): beta = u / gamma and the Lorentz-force beta_dot.
template <typename T>
__device__ __forceinline__ void sample(const LaserT<T>& L, double qm, const T r[3], const T u[3],
                                       double t, T b[3], T a[3]) {
    const T gam = sqrt(1.0 + u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    b[0] = u[0] / gam;
    b[1] = u[1] / gam;
    b[2] = u[2] / gam;
    T Ex, By;
    fields(L, r[0], r[1], r[2], t, Ex, By);
    // E = (Ex, 0, 0), B = (0, By, 0): beta x B = (-b_z By, 0, b_x By)
    const T bE = b[0] * Ex;
    const T f = qm / (gam * kC0);
    a[0] = f * (Ex + kC0 * (-b[2] * By) - b[0] * bE);
    a[1] = f * (-b[1] * bE);
    a[2] = f * (kC0 * (b[0] * By) - b[2] * bE);
}

// One Boris step from time ti: drift dt/2, kick with the fields at the midpoint, drift.
template <typename T>
__device__ __forceinline__ void boris_step(const LaserT<T>& L, double qm, double dt, double ti,
                                           T x[3], T v[3]) {
    const double eps = qm * dt / (2.0 * kC0);
    T gam = sqrt(1.0 + v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    const T rh[3] = {x[0] + 0.5 * dt * kC0 * v[0] / gam, x[1] + 0.5 * dt * kC0 * v[1] / gam,
                     x[2] + 0.5 * dt * kC0 * v[2] / gam};
    T Ex, By;
    fields(L, rh[0], rh[1], rh[2], ti + 0.5 * dt, Ex, By);
    const T um[3] = {v[0] + eps * Ex, v[1], v[2]};
    const T gm = sqrt(1.0 + um[0] * um[0] + um[1] * um[1] + um[2] * um[2]);
    const T tv = qm * dt / (2.0 * gm) * By;   // t vector = (0, tv, 0)
    // u' = um + um x t ; s = 2 t / (1 + t^2) ; u+ = um + u' x s
    const T up[3] = {um[0] - um[2] * tv, um[1], um[2] + um[0] * tv};
    const T sv = 2.0 * tv / (1.0 + tv * tv);
    v[0] = um[0] - up[2] * sv + eps * Ex;
    v[1] = um[1];
    v[2] = um[2] + up[0] * sv;
    gam = sqrt(1.0 + v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    x[0] = rh[0] + 0.5 * dt * kC0 * v[0] / gam;
    x[1] = rh[1] + 0.5 * dt * kC0 * v[1] / gam;
    x[2] = rh[2] + 0.5 * dt * kC0 * v[2] / gam;
}

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
// the samples' beta and beta_dot use a shorter form (sample_beam()).
// One warp per 32 electrons doing all of it took 15.7 us per step (1,500 electrons, 10,000
// steps: 157 ms); cut this way it takes 5.0 us (50 ms).
struct Beam {
    double inv_zR, inv_w02, inv_2s2;   // 1/zR, 1/w0^2, 1/(2 sigma^2)
    double om_pi, kz_pi;               // omega/pi, k/(2 pi zR)
    double E0;
};

// E_x of fields() in the form
//   E0 exp(-rho^2/(w0^2 q) - xi^2/(2 sigma^2)) (cos phi + s sin phi) / q,
//   s = zeta/zR, q = 1 + s^2, phi = omega xi + k rho^2 s / (2 zR q), xi = t + z/c0,
// from w^2 = w0^2 q and cos(phi - atan s) = (cos phi + s sin phi) / sqrt(q): one exponential,
// one reciprocal and no arc tangent or square root.
__device__ __forceinline__ double sample_beam(const Beam& B, double x, double y, double z,
                                              double t) {
    const double s = -z * B.inv_zR;
    const double iq = 1.0 / fma(s, s, 1.0);
    const double g = fma(x, x, y * y) * iq;
    const double xi = fma(z, kInvC0, t);
    const double env = exp(-fma(g, B.inv_w02, xi * xi * B.inv_2s2));
    double sn, cs;
    sincospi(fma(B.om_pi, xi, B.kz_pi * (g * s)), &sn, &cs);
    return B.E0 * iq * env * fma(s, sn, cs);
}

// n / d correctly rounded, given the reciprocal r of d to an ulp (residual correction; the
// error left before the last rounding is 2^-105 of the quotient)
__device__ __forceinline__ double quotient(double n, double d, double r) {
    const double q = __dmul_rn(n, r);
    return fma(fma(-q, d, n), r, q);
}

// gamma = sqrt(a), correctly rounded, and its reciprocal to an ulp (a = 1 + u^2 >= 1; an
// infinite or NaN a ends as NaN)
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
            const double f = f0 * ig * sample_beam(B, x, y, z, t), g = f * b0, h = 1.0 + b2;
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

// Gradient of a loss L(samples) with respect to each electron's initial momentum u0 and
// the laser's a0 and w0, by forward-mode differentiation of the push: one thread per
// (electron, direction) pushes the electron again carrying the derivative of its state
// along one of u0_x, u0_y, u0_z, a0 and w0 (Dual<1>) and contracts each sample's
// derivative with dL/d(r, beta, beta_dot) of that sample.  Five threads per electron
// rather than one thread with all five directions: the push is a sequential FP64 chain
// per electron, and GB300's FP64 rate per SM sub-partition makes a single warp's
// instructions slow, so the work is spread over five times as many warps.  Per-electron
// a0 and w0 parts are added to dL_dlaser with FP64 atomics.
constexpr int kTan = 5;
__global__ void push_tangent_kernel(const double* __restrict__ r0, const double* __restrict__ u0,
                                    int64_t n_e, double t0, double dt, int n_steps, Laser L0,
                                    double e0_per_a0, double zr_per_w0, double qm,
                                    const double* __restrict__ g_r, const double* __restrict__ g_b,
                                    const double* __restrict__ g_a, double* __restrict__ dL_du0,
                                    double* __restrict__ dL_dlaser) {
    using D = Dual<1>;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n_e * kTan;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = t / kTan;
        const int dir = (int)(t - k * kTan);   // 0..2: u0 components, 3: a0, 4: w0
        LaserT<D> L;
        L.omega = L0.omega;
        L.k = L0.k;
        L.sigma = L0.sigma;
        L.E0 = D{L0.E0, {dir == 3 ? e0_per_a0 : 0.0}};
        L.zR = D{L0.zR, {dir == 4 ? zr_per_w0 : 0.0}};
        L.w0 = D{L0.w0, {dir == 4 ? 1.0 : 0.0}};
        D x[3], v[3];
        for (int c = 0; c < 3; ++c) {
            x[c] = mk<1>(r0[3 * k + c]);
            v[c] = mk<1>(u0[3 * k + c]);
            v[c].d[0] = dir == c ? 1.0 : 0.0;
        }
        double acc = 0.0;
        const int64_t base = k * (int64_t)(n_steps + 1);
        auto contract = [&](int64_t o, double tt) {
            D b[3], a[3];
            sample(L, qm, x, v, tt, b, a);
            for (int c = 0; c < 3; ++c)
                acc = fma(g_r[3 * o + c], x[c].d[0],
                          fma(g_b[3 * o + c], b[c].d[0], fma(g_a[3 * o + c], a[c].d[0], acc)));
        };
        contract(base, t0);
        for (int s = 0; s < n_steps; ++s) {
            boris_step(L, qm, dt, t0 + dt * (double)s, x, v);
            contract(base + s + 1, t0 + dt * (double)(s + 1));
        }
        if (dir < 3)
            dL_du0[3 * k + dir] += acc;
        else
            atomicAdd(dL_dlaser + (dir - 3), acc);
    }
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
    Laser L;
    L.omega = 2.0 * kPi * kC0 / laser->lam;
    L.k = L.omega * kInvC0;
    L.sigma = laser->fwhm / (2.0 * sqrt(log(2.0)));
    L.E0 = laser->a0 * kMe * kC0 * L.omega / kQe;
    L.zR = kPi * laser->w0 * laser->w0 / laser->lam;
    L.w0 = laser->w0;
    Beam B;
    B.inv_zR = 1.0 / L.zR;
    B.inv_w02 = 1.0 / (L.w0 * L.w0);
    B.inv_2s2 = 1.0 / (2.0 * L.sigma * L.sigma);
    B.om_pi = L.omega / kPi;
    B.kz_pi = L.k / (2.0 * kPi * L.zR);
    B.E0 = L.E0;
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
    Laser L;
    L.omega = 2.0 * kPi * kC0 / laser->lam;
    L.k = L.omega * kInvC0;
    L.sigma = laser->fwhm / (2.0 * sqrt(log(2.0)));
    const double e0_per_a0 = kMe * kC0 * L.omega / kQe;
    L.E0 = laser->a0 * e0_per_a0;
    L.zR = kPi * laser->w0 * laser->w0 / laser->lam;
    L.w0 = laser->w0;
    const double zr_per_w0 = 2.0 * kPi * laser->w0 / laser->lam;
    // one warp per block: the warps spread over the SMs' sub-partitions
    const int threads = 32;
    const int64_t work = n_e * kTan;
    const int blocks = (int)std::min<int64_t>((work + threads - 1) / threads, 1 << 20);
    push_tangent_kernel<<<blocks, threads, 0, as_stream(stream)>>>(
        r0, u0, n_e, t0, dt, n_steps, L, e0_per_a0, zr_per_w0, charge / mass, dL_dr, dL_dbeta,
        dL_dbeta_dot, dL_du0, dL_dlaser);
    return launch_status();
}
