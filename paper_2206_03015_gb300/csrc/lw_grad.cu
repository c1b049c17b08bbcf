// Adjoint of lw_deposit_time_domain followed by lw_spectrum (FP64, and mixed precision below).
//
// Given g = dL/dS and the saved X' = sqrt(K) dt_u X, the record gradient is
//   dL/drec_c[j] = 2 sqrt(K) dt_u Re( sum_{l=0}^{N/2} g_l conj(X'_c(l)) e^{+2 pi i j l/N} ),
// evaluated as one complex FFT of two Hermitian-extended rows (both outputs
// are real, so they travel as the real and imaginary part of one transform).
// The deposit's adjoint is its transpose: a gather over the same
// (electron, step, pixel) intervals.  For grid point j in (t_b, t_a] with
// w = (t_j - t_b)/(t_a - t_b) the record received F_b (1 - w) + F_a w, so
//   dL/dF_b += R (1 - w),  dL/dF_a += R w,
//   dL/dt_a += -(R.(F_a - F_b)) w / (t_a - t_b),
//   dL/dt_b += -(R.(F_a - F_b)) (1 - w) / (t_a - t_b),
// and, per sample, with t_a = t - n.r/c0 and F = [(n-beta)(n.bdot) - D bdot]/D^3:
//   dL/dr    = -(dL/dt_a) n / c0,
//   dL/dbdot = [n ((n-beta).G) - D G] / D^3,
//   dL/dbeta = [-(n.bdot) G + n (bdot.G)] / D^3 + 3 n (F.G) / D,     G = dL/dF.
// Contributions of the 32 pixels of a warp to the same sample are summed with
// shuffles before one atomic add per component.
#include <math.h>

#include "lw_fft.cuh"

namespace lw {
namespace {

// ------------------------------------------------------------ adjoint FFT

struct AdjLoader {
    const double2* X;     // [n_pix][3][nl] (FP64 forward)
    const float2* Xf;     // the same from a mixed-precision forward (X unused when set)
    const double* g;      // [n_pix][nl]
    int64_t rows;         // 3 * n_pix
    int64_t nl;
    double two_sigma;     // 2 sqrt(K) dt_u

    __device__ double2 H(int64_t row, int64_t l) const {   // 2 sigma g_l conj(X'_l)
        double2 h;
        if (row >= rows) {
            h.x = h.y = 0.0;
            return h;
        }
        const int64_t m = row / 3;
        double2 x;
        if (Xf) {
            const float2 xf = Xf[row * nl + l];
            x.x = xf.x;
            x.y = xf.y;
        } else {
            x = X[row * nl + l];
        }
        const double s = two_sigma * g[m * nl + l];
        h.x = s * x.x;
        h.y = -s * x.y;
        return h;
    }
    // Hermitian extension of H at index l of a length-N transform
    __device__ double2 Ht(int64_t row, int64_t l, int64_t N) const {
        const int64_t half = N / 2;
        double2 h;
        if (l == 0 || l == half) {
            h = H(row, l);
            h.y = 0.0;
        } else if (l < half) {
            h = H(row, l);
            h.x *= 0.5;
            h.y *= 0.5;
        } else {
            h = H(row, N - l);
            h.x *= 0.5;
            h.y = -0.5 * h.y;
        }
        return h;
    }
    __device__ double2 operator()(int64_t pair, int64_t l, int64_t N) const {
        const double2 a = Ht(2 * pair, l, N), b = Ht(2 * pair + 1, l, N);
        double2 z;
        z.x = a.x - b.y;
        z.y = a.y + b.x;
        return z;
    }
};

__device__ __forceinline__ void adj_store(double* out, int64_t rows, int64_t pair, int64_t N,
                                          int64_t j, double2 z) {
    const int64_t ra = 2 * pair, rb = 2 * pair + 1;
    out[ra * N + j] = z.x;
    if (rb < rows) out[rb * N + j] = z.y;
}

__global__ void adj_direct_kernel(AdjLoader ld, int N, int logN, const double2* __restrict__ tw,
                                  double* __restrict__ out) {
    extern __shared__ unsigned char smem_raw[];
    double2* buf = reinterpret_cast<double2*>(smem_raw);
    const int64_t pair = blockIdx.x;
    for (int l = threadIdx.x; l < N; l += blockDim.x) buf[bitrev(l, logN)] = ld(pair, l, N);
    __syncthreads();
    fft_smem<double2, 1, false>(buf, N, logN, tw, N);
    for (int j = threadIdx.x; j < N; j += blockDim.x) adj_store(out, ld.rows, pair, N, j, buf[j]);
}

template <int CT>
__global__ void adj_pass1_kernel(AdjLoader ld, int N, int N1, int logN1, int N2,
                                 const double2* __restrict__ tw, double2* __restrict__ Y) {
    extern __shared__ unsigned char smem_raw[];
    double2* buf = reinterpret_cast<double2*>(smem_raw);   // [N1][CT]
    const int64_t pair = blockIdx.y;
    const int c0 = blockIdx.x * CT;
    for (int t = threadIdx.x; t < N1 * CT; t += blockDim.x) {
        const int c = t % CT, n1 = t / CT;
        buf[bitrev(n1, logN1) * CT + c] = ld(pair, (int64_t)n1 * N2 + c0 + c, N);
    }
    __syncthreads();
    fft_smem<double2, CT, false>(buf, N1, logN1, tw, N);
    double2* Yp = Y + pair * (int64_t)N;
    for (int t = threadIdx.x; t < N1 * CT; t += blockDim.x) {
        const int c = t % CT, k1 = t / CT;
        const int n2 = c0 + c;
        Yp[(int64_t)k1 * N2 + n2] = cmul(buf[k1 * CT + c], tw[((int64_t)n2 * k1) & (N - 1)]);
    }
}

// rows k1 .. k1+CT-1 of the pass-1 output: transform over n2, write X[k1 + N1 k2]
template <int CT>
__global__ void adj_pass2_kernel(int64_t rows, int N, int N1, int N2, int logN2,
                                 const double2* __restrict__ tw, const double2* __restrict__ Y,
                                 double* __restrict__ out) {
    extern __shared__ unsigned char smem_raw[];
    double2* buf = reinterpret_cast<double2*>(smem_raw);   // [N2][CT]
    const int64_t pair = blockIdx.y;
    const int k10 = blockIdx.x * CT;
    const double2* Yp = Y + pair * (int64_t)N;
    for (int t = threadIdx.x; t < N2 * CT; t += blockDim.x) {
        const int n2 = t % N2, c = t / N2;
        buf[bitrev(n2, logN2) * CT + c] = Yp[(int64_t)(k10 + c) * N2 + n2];
    }
    __syncthreads();
    fft_smem<double2, CT, false>(buf, N2, logN2, tw, N);
    for (int t = threadIdx.x; t < N2 * CT; t += blockDim.x) {
        const int c = t % CT, k2 = t / CT;
        adj_store(out, rows, pair, N, (int64_t)(k10 + c) + (int64_t)N1 * k2, buf[k2 * CT + c]);
    }
}

// ------------------------------------------------------------ adjoint deposit

struct AdjArgs {
    int64_t n_e, ns1;
    int t_per_e;
    const double* t;
    const double* r;
    const double* beta;
    const double* bdot;
    const double* n_hat;
    int64_t n_pix;
    double t_min, dt_u, inv_dtu;
    int64_t n_bins;
    const double* dLdrec;   // [n_pix][3][n_bins]
    const float* dLdrec_f;  // mixed: dLdrec * 2^-e in FP32 (|values| < 2)
    const double* rscale;   // mixed: 2^e (device scalar)
    float* f_grad;          // mixed: per sample 12 floats, (dL/du_a n, dL/dbeta, dL/dbdot, 0)
                            // on the record gradient's scale, FP32 sums
    double* g_r;
    double* g_beta;
    double* g_bdot;
    int e_chunk;
};

constexpr int kAdjThreads = 128;
constexpr int kAdjTile = 64;

// One sample seen from one pixel: m = n - beta, nm = n . m, k = n . beta_dot and D = 1 - n . beta
// give the acceleration field F = (k m - nm beta_dot) / D^3 (Eq. far_efield expanded); zero, with
// iD = 0, when |beta| >= 1 or D <= 0.
struct SampleField {
    double m[3], a[3], F[3];
    double nm, k, iD, iD3;
};
__device__ __forceinline__ void sample_field(double nx, double ny, double nz,
                                             const double* __restrict__ b,
                                             const double* __restrict__ a, SampleField& f) {
    const double b0 = b[0], b1 = b[1], b2 = b[2];
    for (int c = 0; c < 3; ++c) f.a[c] = a[c];
    f.m[0] = nx - b0;
    f.m[1] = ny - b1;
    f.m[2] = nz - b2;
    f.nm = fma(nz, f.m[2], fma(ny, f.m[1], nx * f.m[0]));
    f.k = fma(nz, f.a[2], fma(ny, f.a[1], nx * f.a[0]));
    // the forward's D to the bit: 1e-16 of rounding in n . beta is 1e-12 of D at gamma 60
    const double D = __dsub_rn(1.0, __dadd_rn(__dadd_rn(__dmul_rn(nx, b0), __dmul_rn(ny, b1)),
                                              __dmul_rn(nz, b2)));
    // the forward's test too: a sample whose field it takes as zero has no gradient
    const bool ok = D > 0.0 && subluminal(b0, b1, b2);
    f.iD = ok ? __drcp_rn(D) : 0.0;
    f.iD3 = f.iD * f.iD * f.iD;
    for (int c = 0; c < 3; ++c) f.F[c] = fma(f.m[c], f.k, -f.a[c] * f.nm) * f.iD3;
}

// (dL/dF, dL/dt_a) of one sample -> (dL/dr, dL/dbeta, dL/dbdot)
__device__ __forceinline__ void sample_chain(double nx, double ny, double nz, const SampleField& f,
                                             const double G[3], double gta, double out[9]) {
    const double gc = -gta * kInvC0;
    out[0] = gc * nx;
    out[1] = gc * ny;
    out[2] = gc * nz;
    const double aG = fma(f.a[2], G[2], fma(f.a[1], G[1], f.a[0] * G[0]));
    const double mG = fma(f.m[2], G[2], fma(f.m[1], G[1], f.m[0] * G[0]));
    const double FG = fma(f.F[2], G[2], fma(f.F[1], G[1], f.F[0] * G[0]));
    const double sn = fma(aG, f.iD3, 3.0 * f.iD * FG), sG = f.k * f.iD3;
    const double tn = mG * f.iD3, tG = f.nm * f.iD3;
    out[3] = fma(nx, sn, -sG * G[0]);
    out[4] = fma(ny, sn, -sG * G[1]);
    out[5] = fma(nz, sn, -sG * G[2]);
    out[6] = fma(nx, tn, -tG * G[0]);
    out[7] = fma(ny, tn, -tG * G[1]);
    out[8] = fma(nz, tn, -tG * G[2]);
}

// Sums of nine values over the warp: eight by halving (each exchange sends the half of the
// values that the partner keeps: 4 + 2 + 1 exchanges, then two for the group of four lanes), the
// ninth by five exchanges -- 14 additions instead of 45.  Lane 4 g holds the sum of value g in the
// result, lane 1 that of value 8; the index is `which` (-1 on the other lanes).
template <typename T>
__device__ __forceinline__ T warp_sum9(const T (&o)[9], int& which) {
    const int lane = threadIdx.x & 31;
    T v[4], w[2];
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        v[c] = (h16 ? o[c + 4] : o[c]) + __shfl_xor_sync(0xffffffffu, h16 ? o[c] : o[c + 4], 16);
#pragma unroll
    for (int c = 0; c < 2; ++c)
        w[c] = (h8 ? v[c + 2] : v[c]) + __shfl_xor_sync(0xffffffffu, h8 ? v[c] : v[c + 2], 8);
    T x = (h4 ? w[1] : w[0]) + __shfl_xor_sync(0xffffffffu, h4 ? w[0] : w[1], 4);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    T y = o[8];
    for (int s = 16; s > 0; s >>= 1) y += __shfl_xor_sync(0xffffffffu, y, s);
    which = (lane & 3) == 0 ? lane >> 2 : (lane == 1 ? 8 : -1);
    return lane == 1 ? y : x;
}

// finish sample i: chain rule, warp sum over pixels, atomics into the gradients
__device__ __forceinline__ void flush_sample(const AdjArgs& p, double nx, double ny, double nz,
                                             int64_t s, const SampleField& f, const double G[3],
                                             double gta, bool nonzero) {
    if (!__any_sync(0xffffffffu, nonzero)) return;
    double o[9];
    if (nonzero) {
        sample_chain(nx, ny, nz, f, G, gta, o);
    } else {
        for (int c = 0; c < 9; ++c) o[c] = 0.0;
    }
    int which;
    const double v = warp_sum9(o, which);
    if (which >= 0) {
        double* g = which < 3 ? p.g_r + which : which < 6 ? p.g_beta + (which - 3)
                                                          : p.g_bdot + (which - 6);
        atomicAdd(g + 3 * s, v);
    }
}

// Transpose of the FP64 deposit: thread = pixel, a CTA walks part of an electron's steps (grid z)
// in order.  Bound by the FP64 pipe (19 cycles per warp instruction and SM), so within a step the
// sums over its grid points are S0 = sum R and S1 = sum R w only: with dF = Fa - Fb the rest is
// per step,
//   dL/dF_b += S0 - S1,  dL/dF_a += S1,  dL/dt_a -= dF.S1/(t_a - t_b),
//   dL/dt_b -= dF.(S0 - S1)/(t_a - t_b),
// and a sample's field, Doppler factor and products serve its chain rule too.  64 electrons x
// 1,200 steps x 400 pixels x 4,096 bins: 22.9 ms with these sums per grid point, the field
// evaluated again in the chain rule and 45 additions per sample in the warp sums; now 10.0.
__global__ void __launch_bounds__(kAdjThreads) adj_deposit_kernel(AdjArgs p) {
    __shared__ double s_t[kAdjTile];
    __shared__ double s_r[kAdjTile * 3];
    const int64_t m = (int64_t)blockIdx.x * kAdjThreads + threadIdx.x;
    const bool active = m < p.n_pix;
    double nx = 0.0, ny = 0.0, nz = 1.0;
    if (active) {
        nx = p.n_hat[3 * m];
        ny = p.n_hat[3 * m + 1];
        nz = p.n_hat[3 * m + 2];
    }
    const double* R = p.dLdrec + (active ? m * 3 * p.n_bins : 0);
    const int64_t k0 = (int64_t)blockIdx.y * p.e_chunk;
    const int64_t k1 = min(k0 + p.e_chunk, p.n_e);
    // this CTA's steps end at samples i_lo + 1 .. i_hi: whole tiles
    const int64_t n_tiles = (p.ns1 + kAdjTile - 1) / kAdjTile;
    const int64_t i_lo = n_tiles * blockIdx.z / gridDim.z * kAdjTile;
    const int64_t i_hi = min(n_tiles * (blockIdx.z + 1) / gridDim.z * kAdjTile, p.ns1 - 1);
    for (int64_t k = k0; k < k1; ++k) {
        const double* tk = p.t + (p.t_per_e ? k * p.ns1 : 0);
        const double* rk = p.r + 3 * k * p.ns1;
        const double* bk = p.beta + 3 * k * p.ns1;
        const double* ak = p.bdot + 3 * k * p.ns1;
        double tb = 0.0;
        int64_t jb = 0;   // floor of the coordinate of sample i-1
        bool ok_b = false;
        SampleField fb = {};   // sample i-1 (valid when fb_step == i-1)
        int64_t fb_step = -1;
        double Gc[3] = {0.0, 0.0, 0.0}, gtc = 0.0;   // carry: sample i-1 so far
        bool nzc = false;
        for (int64_t i0 = i_lo; i0 <= i_hi; i0 += kAdjTile) {
            const int n = (int)min((int64_t)kAdjTile, i_hi + 1 - i0);
            __syncthreads();
            for (int q = threadIdx.x; q < n; q += kAdjThreads) {
                s_t[q] = tk[i0 + q];
                s_r[3 * q] = rk[3 * (i0 + q)];
                s_r[3 * q + 1] = rk[3 * (i0 + q) + 1];
                s_r[3 * q + 2] = rk[3 * (i0 + q) + 2];
            }
            __syncthreads();
            for (int q = 0; q < n; ++q) {
                const int64_t i = i0 + q;
                const double ta = advanced_time_fp64(nx, ny, nz, s_r[3 * q], s_r[3 * q + 1],
                                                     s_r[3 * q + 2], s_t[q]);
                const double ua = __dmul_rn(__dsub_rn(ta, p.t_min), p.inv_dtu);
                // |u| < 2^62 on the bits
                const bool ok_a = (__double2hiint(ua) & 0x7fffffff) < 0x43d00000;
                const int64_t je = __double2ll_rd(ua);
                double Gn[3] = {0.0, 0.0, 0.0}, gtn = 0.0;   // contributions to sample i
                SampleField fa;
                bool step = false;   // the step holds grid points
                if (i > i_lo && active && ok_a && ok_b) {
                    int64_t ja = jb + 1, jz = je;
                    if (ja < 0) ja = 0;
                    if (jz > p.n_bins - 1) jz = p.n_bins - 1;
                    if (ja <= jz) {
                        step = true;
                        if (fb_step != i - 1)
                            sample_field(nx, ny, nz, bk + 3 * (i - 1), ak + 3 * (i - 1), fb);
                        sample_field(nx, ny, nz, bk + 3 * i, ak + 3 * i, fa);
                        const double iden = 1.0 / __dsub_rn(ta, tb);
                        double S0[3] = {0.0, 0.0, 0.0}, S1[3] = {0.0, 0.0, 0.0};
                        double jd = (double)ja;
                        for (int64_t j = ja; j <= jz; ++j, jd += 1.0) {
                            const double w = (fma(jd, p.dt_u, p.t_min) - tb) * iden;
                            const double R0 = R[j], R1 = R[p.n_bins + j], R2 = R[2 * p.n_bins + j];
                            S0[0] += R0;
                            S0[1] += R1;
                            S0[2] += R2;
                            S1[0] = fma(R0, w, S1[0]);
                            S1[1] = fma(R1, w, S1[1]);
                            S1[2] = fma(R2, w, S1[2]);
                        }
                        double d0 = 0.0, d1 = 0.0;   // dF . (S0 - S1), dF . S1
                        for (int c = 0; c < 3; ++c) {
                            const double dF = fa.F[c] - fb.F[c], g = S0[c] - S1[c];
                            d0 = fma(dF, g, d0);
                            d1 = fma(dF, S1[c], d1);
                            Gc[c] += g;
                            Gn[c] = S1[c];
                        }
                        gtc = fma(-d0, iden, gtc);
                        gtn = -d1 * iden;
                    }
                }
                if (i > i_lo)
                    flush_sample(p, nx, ny, nz, k * p.ns1 + i - 1, fb, Gc, gtc, nzc || step);
                for (int c = 0; c < 3; ++c) Gc[c] = Gn[c];
                gtc = gtn;
                nzc = step;
                if (step) {
                    fb = fa;
                    fb_step = i;
                }
                tb = ta;
                jb = je;
                ok_b = ok_a;
            }
        }
        flush_sample(p, nx, ny, nz, k * p.ns1 + i_hi, fb, Gc, gtc, nzc);
    }
}

// ------------------------------------------------------------ mixed-precision adjoint
//
// Bound by issue and latency.  2,048 electrons x 4,096 steps x 1,024 pixels x 16,384 bins: 269 ms
// with 64-bit grid indices (their conversions held the FP64 pipe at 71 %), a second field
// evaluation in the chain rule and 45 shuffles per sample; 197 ms with 32-bit indices, one
// evaluation and warp_sum9; 152 ms with FP32 constants that are not converted again per step and
// the exact coordinate out of line, so that seven CTAs per SM are resident instead of four.
//
// The same transpose in mixed precision: the bin coordinate of each tile's first sample in
// FP64 and, within the tile of 64 samples, each sample's as an integer plus an FP32
// fraction advanced by the step's FP32 increment (from FP64-differenced samples), so the
// weights are computed from numbers of the size of a step; everything else in FP32:
// the fields in the stable form
// D = (1 - n_z) + n_z (1 - beta_z) - n_perp . beta_perp, the weights from bin coordinates
// relative to the step's first grid point, the sums over grid points and the per-sample
// chain rule.  The record gradient enters scaled by a power of two 2^-e (|values| < 2,
// e from its largest magnitude), so that its products with fields of up to ~1e30 /s stay
// in FP32 range; the warp sums are added to per-sample FP32 sums, which a last pass unscales
// in FP64 into the caller's gradients.

// largest |dL/drec| as ordered bits (non-negative doubles compare as integers)
__global__ void adj_absmax_kernel(const double* __restrict__ R, int64_t n,
                                  unsigned long long* __restrict__ mx) {
    unsigned long long v = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(R[i]));
        v = b > v ? b : v;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(mx, v);
}

// 2^e >= the largest |dL/drec| / 2 (1 when it is zero or not finite)
__device__ __forceinline__ int adj_exponent(unsigned long long mx) {
    const int e = (int)(mx >> 52) - 1023;
    return (mx == 0 || e > 1000 || e < -1000) ? 0 : e;
}

// dL/drec scaled and rounded to FP32.  With n_bins a multiple of 4 a pixel's three rows are
// interleaved in groups of four bins (x, y, z of bins 4 q .. 4 q + 3: 48 bytes), so that the lanes
// of a warp, each walking its own pixel, keep one cache line in use instead of three: the
// adjoint's L1 working set is what limits its resident warps.
__global__ void adj_to_f32_kernel(const double* __restrict__ R, int64_t n_pix, int64_t n_bins,
                                  const unsigned long long* __restrict__ mx,
                                  float* __restrict__ Rf, double* __restrict__ rscale) {
    const int e = adj_exponent(*mx);
    const double down = ldexp(1.0, -e);
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if ((n_bins & 3) == 0) {
        const int64_t per = n_bins / 4;
        for (int64_t g = i0; g < n_pix * per; g += step) {
            const int64_t m = g / per, q = g - m * per;
            for (int c = 0; c < 3; ++c) {
                const double* r = R + (3 * m + c) * n_bins + 4 * q;
                reinterpret_cast<float4*>(Rf)[3 * g + c] =
                    make_float4((float)(r[0] * down), (float)(r[1] * down), (float)(r[2] * down),
                                (float)(r[3] * down));
            }
        }
    } else {
        for (int64_t i = i0; i < 3 * n_pix * n_bins; i += step) Rf[i] = (float)(R[i] * down);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *rscale = ldexp(1.0, e);
}

struct NF {   // a pixel direction in FP32 with 1 - n_z kept exactly
    float x, y, z, omz;
};

// One sample seen from one pixel: acceleration field ((n - beta) (n . bdot) - D bdot) / D^3 in FP32
// and what its chain rule shares with it; all zero when |beta| >= 1 (b.w == 0) or D <= 0
struct SampleF {
    float mx, my, mz, nbd, D, iD, iD3;
    float F[3];
};
__device__ __forceinline__ void sample_field_f32(const NF& n, float4 b, float4 a, SampleF& f) {
    f.D = fmaf(-n.y, b.y, fmaf(-n.x, b.x, fmaf(n.z, b.z, n.omz)));
    f.mx = n.x - b.x;
    f.my = n.y - b.y;
    f.mz = b.z - n.omz;
    f.nbd = fmaf(n.z, a.z, fmaf(n.y, a.y, n.x * a.x));
    const bool ok = b.w != 0.0f && f.D > 0.0f;
    f.iD = ok ? __fdividef(1.0f, f.D) : 0.0f;
    f.iD3 = f.iD * f.iD * f.iD;
    f.F[0] = fmaf(f.mx, f.nbd, -f.D * a.x) * f.iD3;
    f.F[1] = fmaf(f.my, f.nbd, -f.D * a.y) * f.iD3;
    f.F[2] = fmaf(f.mz, f.nbd, -f.D * a.z) * f.iD3;
}

// (dL/dF, dL/du_a) of one sample -> (dL/du_a n, dL/dbeta, dL/dbdot) in FP32, on the scale
// of the record gradient; dL/dr = -(dL/du_a) n / (c0 dt_u) is completed by the caller
__device__ __forceinline__ void sample_chain_f32(const NF& n, const SampleF& f, float4 a,
                                                 const float G[3], float gu, float o[9]) {
    o[0] = gu * n.x;
    o[1] = gu * n.y;
    o[2] = gu * n.z;
    const float bG = fmaf(a.z, G[2], fmaf(a.y, G[1], a.x * G[0]));
    const float mG = fmaf(f.mz, G[2], fmaf(f.my, G[1], f.mx * G[0]));
    const float FG3 = 3.0f * fmaf(f.F[2], G[2], fmaf(f.F[1], G[1], f.F[0] * G[0])) * f.iD;
    o[3] = fmaf(fmaf(-f.nbd, G[0], n.x * bG), f.iD3, n.x * FG3);
    o[4] = fmaf(fmaf(-f.nbd, G[1], n.y * bG), f.iD3, n.y * FG3);
    o[5] = fmaf(fmaf(-f.nbd, G[2], n.z * bG), f.iD3, n.z * FG3);
    o[6] = fmaf(n.x, mG, -f.D * G[0]) * f.iD3;
    o[7] = fmaf(n.y, mG, -f.D * G[1]) * f.iD3;
    o[8] = fmaf(n.z, mG, -f.D * G[2]) * f.iD3;
}

__device__ __forceinline__ void flush_sample_f32(const AdjArgs& p, const NF& n, int64_t s,
                                                 const SampleF& f, float4 a, const float G[3],
                                                 float gu, bool nonzero) {
    if (!__any_sync(0xffffffffu, nonzero)) return;
    float o[9];
    if (nonzero) {
        sample_chain_f32(n, f, a, G, gu, o);
    } else {
        for (int c = 0; c < 9; ++c) o[c] = 0.0f;
    }
    int which;
    const float v = warp_sum9(o, which);
    if (which >= 0) atomicAdd(p.f_grad + 12 * s + which, v);   // one FP32 reduction of nine lanes
}

// the FP32 sums in FP64, unscaled, added to the caller's gradients
__global__ void adj_finish_kernel(const float* __restrict__ f, int64_t n_samples,
                                  const double* __restrict__ rscale, double inv_dtu,
                                  double* __restrict__ g_r, double* __restrict__ g_b,
                                  double* __restrict__ g_a) {
    const double r_scale = *rscale;
    const double u_scale = -r_scale * inv_dtu * kInvC0;   // dL/dr = -(dL/du_a) n / (c0 dt_u)
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n_samples;
         s += (int64_t)gridDim.x * blockDim.x) {
        const float* q = f + 12 * s;
        for (int c = 0; c < 3; ++c) {
            g_r[3 * s + c] += (double)q[c] * u_scale;
            g_b[3 * s + c] += (double)q[3 + c] * r_scale;
            g_a[3 * s + c] += (double)q[6 + c] * r_scale;
        }
    }
}

// Half-width of the band around an integer inside which a sample's bin coordinate is
// recomputed in FP64: far above the FP32 chain's rounding over a tile (64 steps of a few
// ulps of the step's terms).
constexpr float kAdjGuard = 1.0f / (1 << 12);

// The FP64 adjoint's bin coordinate of a sample (t, x) for the direction n, as floor + FP32
// fraction.  32-bit: conversions from and to 64-bit integers run on the FP64 pipe; coordinates are
// clamped to +-1e9, far beyond any grid.  Out of line, reading its direction again: inlined it
// keeps doubles in registers throughout.
__device__ __noinline__ int2 adj_exact_coord(const double* n, const double* x, double t,
                                             double t_min, double inv_dtu) {
    double u = __dmul_rn(__dsub_rn(advanced_time_fp64(n[0], n[1], n[2], x[0], x[1], x[2], t), t_min),
                         inv_dtu);
    u = fmin(fmax(u, -1.0e9), 1.0e9);
    const double fl = floor(u);
    return make_int2((int)fl, __float_as_int((float)(u - fl)));
}

__global__ void __launch_bounds__(kAdjThreads, 7) adj_deposit_mixed_kernel(AdjArgs p) {
    // one tile of samples i0 .. i0 + kAdjTile - 1, staged once per CTA: each sample's step
    // from the previous one (FP64 differences rounded to FP32) and its fields' inputs
    __shared__ float4 s_d[kAdjTile];   // (tau_i - tau_i-1, r_i - r_i-1), tau = t - z/c0
    // (slot q + 1: sample i0 + q, slot 0: the sample before the tile)
    __shared__ float4 s_b[kAdjTile + 1];   // (beta_x, beta_y, 1 - beta_z, |beta| < 1)
    __shared__ float4 s_a[kAdjTile + 1];   // (beta_dot, 0)
    const int64_t m = (int64_t)blockIdx.x * kAdjThreads + threadIdx.x;
    const bool active = m < p.n_pix;
    const double* n_hat = p.n_hat + (active ? 3 * m : 0);   // inactive lanes follow pixel 0
    NF nf;
    float s32, wx32, wy32, wz32;
    {
        const double nx = n_hat[0], ny = n_hat[1], nz = n_hat[2];
        nf.x = (float)nx;
        nf.y = (float)ny;
        nf.z = (float)nz;
        nf.omz = (float)(1.0 - nz);
        // bin coordinate u = (t_a - t_min)/dt_u = (tau - t_min)/dt_u + w . r with the pixel's slope
        // w = (-n_x, -n_y, 1 - n_z) / (c0 dt_u): in FP64 at each tile's first sample; from there on
        // as J + f (integer, FP32 fraction) advanced by each step's FP32 increment s dtau + w . dr,
        // so that the weights see small numbers
        const double sw = kInvC0 * p.inv_dtu;
        s32 = (float)p.inv_dtu;
        wx32 = (float)(-nx * sw);
        wy32 = (float)(-ny * sw);
        wz32 = (float)((1.0 - nz) * sw);
    }
    // the rounded values are made opaque: the compiler otherwise converts the doubles again in
    // every step to save registers (FP64 pipe 71-80 % busy at 96 registers)
    asm volatile("" : "+f"(s32), "+f"(wx32), "+f"(wy32), "+f"(wz32));
    asm volatile("" : "+f"(nf.x), "+f"(nf.y), "+f"(nf.z), "+f"(nf.omz));
    const float* R = p.dLdrec_f + (active ? m * 3 * p.n_bins : 0);
    const bool vec = (p.n_bins & 3) == 0;
    const int nb1 = (int)p.n_bins - 1;
    const int64_t k0 = (int64_t)blockIdx.y * p.e_chunk;
    const int64_t k1 = min(k0 + p.e_chunk, p.n_e);
    for (int64_t k = k0; k < k1; ++k) {
        const double* tk = p.t + (p.t_per_e ? k * p.ns1 : 0);
        const double* rk = p.r + 3 * k * p.ns1;
        const double* bk = p.beta + 3 * k * p.ns1;
        const double* ak = p.bdot + 3 * k * p.ns1;
        SampleF fb = {};   // sample i-1 (valid when fb_step == i-1)
        int64_t fb_step = -1;
        float Gc[3] = {0.0f, 0.0f, 0.0f}, guc = 0.0f;   // carry: sample i-1 so far
        bool nzc = false;
        int J = 0;   // sample i-1 at J + f
        // the record gradient is read in increasing j: with n_bins a multiple of 4 a lane keeps
        // the group of four bins holding the current j, three vector loads per group instead
        // of three scalars per bin (the lanes of a warp read 32 different pixels, so loads
        // cost one L1 wavefront per lane)
        int jc = -4;
        float4 c0 = make_float4(0.f, 0.f, 0.f, 0.f), c1 = c0, c2 = c0;
        float f = 0.0f;
        for (int64_t i0 = 0; i0 < p.ns1; i0 += kAdjTile) {
            const int n = (int)min((int64_t)kAdjTile, p.ns1 - i0);
            __syncthreads();
            for (int q = (i0 > 0 ? -1 : 0) + (int)threadIdx.x; q < n; q += kAdjThreads) {
                const int64_t i = i0 + q;
                const double* rq = rk + 3 * i;
                const double* bq = bk + 3 * i;
                const double* aq = ak + 3 * i;
                if (i > 0 && q >= 0) {
                    const double tau = tk[i] - rq[2] * kInvC0;
                    const double taup = tk[i - 1] - rq[-1] * kInvC0;
                    s_d[q] = make_float4((float)(tau - taup), (float)(rq[0] - rq[-3]),
                                         (float)(rq[1] - rq[-2]), (float)(rq[2] - rq[-1]));
                }
                const double bb = __dadd_rn(__dadd_rn(__dmul_rn(bq[0], bq[0]),
                                                      __dmul_rn(bq[1], bq[1])),
                                            __dmul_rn(bq[2], bq[2]));
                s_b[q + 1] = make_float4((float)bq[0], (float)bq[1], (float)(1.0 - bq[2]),
                                     bb < 1.0 ? 1.0f : 0.0f);
                s_a[q + 1] = make_float4((float)aq[0], (float)aq[1], (float)aq[2], 0.0f);
            }
            __syncthreads();
            for (int q = 0; q < n; ++q) {
                const int64_t i = i0 + q;
                // sample i at Ji + fi: the tile's first from the FP64 anchor, the others
                // advanced from sample i-1 by the step's FP32 increment, and recomputed in
                // FP64 when the fraction lies within kAdjGuard of an integer, so that the
                // floors -- which grid points a step holds -- are those of the FP64 adjoint
                int Ji;
                float fi;
                bool exact = q == 0;
                if (!exact) {
                    const float4 d = s_d[q];
                    float u = f + fmaf(wz32, d.w, fmaf(wy32, d.z, fmaf(wx32, d.y, s32 * d.x)));
                    u = fminf(fmaxf(u, -1.0e9f), 1.0e9f);
                    const float fl = floorf(u);
                    Ji = min(max(J + (int)fl, -1000000000), 1000000000);
                    fi = u - fl;
                    // (a clamped coordinate is no start to add to)
                    exact = fi < kAdjGuard || fi > 1.0f - kAdjGuard || abs(J) > 900000000 ||
                            abs(Ji) > 900000000;
                }
                if (exact) {
                    const int2 e = adj_exact_coord(n_hat, rk + 3 * i, tk[i], p.t_min, p.inv_dtu);
                    Ji = e.x;
                    fi = __int_as_float(e.y);
                }
                // the step (i-1, i] relative to Jf = J_(i-1): ub = f_(i-1), ua = u_i - Jf
                const int dJ = Ji - J;
                const float ub = f;
                const float ua = (dJ > -(1 << 24) && dJ < (1 << 24)) ? (float)dJ + fi : 1.0e9f;
                float Gn[3] = {0.0f, 0.0f, 0.0f}, gun = 0.0f;   // contributions to sample i
                SampleF fa;
                const int ja = max(J + 1, 0), jz = min(Ji, nb1);
                const bool step = i > 0 && active && ja <= jz;   // the step holds grid points
                if (step) {
                    if (fb_step != i - 1) sample_field_f32(nf, s_b[q], s_a[q], fb);
                    sample_field_f32(nf, s_b[q + 1], s_a[q + 1], fa);
                    const float iden = __fdividef(1.0f, ua - ub);
                    const float d0 = fa.F[0] - fb.F[0], d1 = fa.F[1] - fb.F[1],
                                d2 = fa.F[2] - fb.F[2];
                    float tj = (float)(ja - J);
                    for (int j = ja; j <= jz; ++j, tj += 1.0f) {
                        const float wa = (ua - tj) * iden, wb = (tj - ub) * iden;
                        float R0, R1, R2;
                        if (vec) {   // a group of four bins of the three rows, reloaded when left
                            if ((j & ~3) != jc) {
                                jc = j & ~3;
                                const float4* g = reinterpret_cast<const float4*>(R + 3 * jc);
                                c0 = __ldg(g);
                                c1 = __ldg(g + 1);
                                c2 = __ldg(g + 2);
                            }
                            const int e = j & 3;
                            R0 = e == 0 ? c0.x : e == 1 ? c0.y : e == 2 ? c0.z : c0.w;
                            R1 = e == 0 ? c1.x : e == 1 ? c1.y : e == 2 ? c1.z : c1.w;
                            R2 = e == 0 ? c2.x : e == 1 ? c2.y : e == 2 ? c2.z : c2.w;
                        } else {
                            R0 = R[j];
                            R1 = R[p.n_bins + j];
                            R2 = R[2 * p.n_bins + j];
                        }
                        Gc[0] = fmaf(R0, wa, Gc[0]);
                        Gc[1] = fmaf(R1, wa, Gc[1]);
                        Gc[2] = fmaf(R2, wa, Gc[2]);
                        Gn[0] = fmaf(R0, wb, Gn[0]);
                        Gn[1] = fmaf(R1, wb, Gn[1]);
                        Gn[2] = fmaf(R2, wb, Gn[2]);
                        const float dw = fmaf(R2, d2, fmaf(R1, d1, R0 * d0)) * iden;
                        gun = fmaf(-dw, wb, gun);
                        guc = fmaf(-dw, wa, guc);
                    }
                }
                if (i > 0)
                    flush_sample_f32(p, nf, k * p.ns1 + i - 1, fb, s_a[q], Gc, guc, nzc || step);
                Gc[0] = Gn[0];
                Gc[1] = Gn[1];
                Gc[2] = Gn[2];
                guc = gun;
                nzc = step;
                if (step) {
                    fb = fa;
                    fb_step = i;
                }
                J = Ji;
                f = fi;
            }
        }
        flush_sample_f32(p, nf, k * p.ns1 + p.ns1 - 1, fb, s_a[(p.ns1 - 1) % kAdjTile + 1], Gc, guc, nzc);
    }
}

int pick_chunk(int64_t n_e, int64_t tiles) {
    const int64_t target = (int64_t)kSms * 64;
    int64_t chunk = (n_e * tiles + target - 1) / target;
    if (chunk < 1) chunk = 1;
    if (chunk > n_e) chunk = n_e;
    return (int)chunk;
}

}  // namespace
}  // namespace lw

using namespace lw;

extern "C" int lw_spectrum_grad(const lw_traj* traj, const lw_detector* det, const lw_grid* grid,
                                int32_t precision, uint32_t field_flags, const void* X_save,
                                const double* dL_dS, double q, double* dL_dr, double* dL_dbeta,
                                double* dL_dbeta_dot, void* ws, size_t* ws_bytes, void* stream) {
    if (!traj || !det || !grid || !ws_bytes || !det->n_hat || det->n_pix < 1) return LW_EINVAL;
    const bool mixed = precision == LW_MIXED || precision == LW_MIXED_KAHAN ||
                       precision == LW_MIXED_F32 || precision == LW_MIXED_F32X4;
    if (precision != LW_FP64 && !mixed) return LW_EUNSUPPORTED;
    if (field_flags != LW_FIELD_ACCEL) return LW_EUNSUPPORTED;
    if (!(traj->sections & LW_SECTION_FP64)) return LW_EINVAL;
    const int64_t N = grid->n_bins;
    if (N < 2 || N > (int64_t(1) << 18) || (N & (N - 1))) return LW_EUNSUPPORTED;
    if (!(grid->dt_u > 0.0) || !isfinite(q)) return LW_EINVAL;
    int logN = 0;
    while ((int64_t(1) << logN) < N) ++logN;
    const bool direct = N <= 4096;
    const int64_t rows = 3 * det->n_pix;
    const int64_t pairs = (rows + 1) / 2;
    const size_t rec_bytes = align256(sizeof(double) * (size_t)(rows * N));
    const size_t tw_bytes = align256(sizeof(double2) * (size_t)N);
    const size_t y_bytes = direct ? 0 : align256(sizeof(double2) * (size_t)(pairs * N));
    // mixed: the scaled FP32 record gradient, its largest magnitude and the scale
    const size_t gsum_bytes = mixed ? align256(sizeof(float) * 12 * (size_t)(traj->n_e * (traj->n_s + 1))) : 0;
    const size_t f_bytes = mixed ? align256(sizeof(float) * (size_t)(rows * N)) + 256 + gsum_bytes : 0;
    const size_t need = rec_bytes + tw_bytes + y_bytes + f_bytes;
    if (!ws) {
        *ws_bytes = need;
        return LW_OK;
    }
    if (*ws_bytes < need) {
        *ws_bytes = need;
        return LW_ESIZE;
    }
    if (!X_save || !dL_dS || !dL_dr || !dL_dbeta || !dL_dbeta_dot) return LW_EINVAL;
    cudaStream_t st = as_stream(stream);
    char* base = static_cast<char*>(ws);
    double* dLdrec = reinterpret_cast<double*>(base);
    double2* tw = reinterpret_cast<double2*>(base + rec_bytes);
    double2* Y = reinterpret_cast<double2*>(base + rec_bytes + tw_bytes);
    const double K = q * q / (16.0 * kPi * kPi * kPi * kEps0 * kC0);
    AdjLoader ld;
    ld.X = mixed ? nullptr : static_cast<const double2*>(X_save);
    ld.Xf = mixed ? static_cast<const float2*>(X_save) : nullptr;
    ld.g = dL_dS;
    ld.rows = rows;
    ld.nl = N / 2 + 1;
    ld.two_sigma = 2.0 * sqrt(K) * grid->dt_u;

    const int tw_grid = (int)((N + 255) / 256 < 1024 ? (N + 255) / 256 : 1024);
    twiddle_kernel<double><<<tw_grid, 256, 0, st>>>(tw, N);
    if (launch_status() != LW_OK) return LW_ECUDA;
    if (direct) {
        const size_t smem = sizeof(double2) * (size_t)N;
        if (smem > 48 * 1024 &&
            cudaFuncSetAttribute(adj_direct_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem) != cudaSuccess)
            return LW_ECUDA;
        adj_direct_kernel<<<(unsigned)pairs, 256, smem, st>>>(ld, (int)N, logN, tw, dLdrec);
    } else {
        const int logN2 = (logN + 1) / 2, logN1 = logN - logN2;
        const int N1 = 1 << logN1, N2 = 1 << logN2;
        constexpr int CT = 16;
        size_t smem = sizeof(double2) * (size_t)N1 * CT;
        if (smem > 48 * 1024 &&
            cudaFuncSetAttribute(adj_pass1_kernel<CT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem) != cudaSuccess)
            return LW_ECUDA;
        adj_pass1_kernel<CT><<<dim3((unsigned)(N2 / CT), (unsigned)pairs), 256, smem, st>>>(
            ld, (int)N, N1, logN1, N2, tw, Y);
        if (launch_status() != LW_OK) return LW_ECUDA;
        smem = sizeof(double2) * (size_t)N2 * CT;
        if (smem > 48 * 1024 &&
            cudaFuncSetAttribute(adj_pass2_kernel<CT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem) != cudaSuccess)
            return LW_ECUDA;
        adj_pass2_kernel<CT><<<dim3((unsigned)(N1 / CT), (unsigned)pairs), 256, smem, st>>>(
            rows, (int)N, N1, N2, logN2, tw, Y, dLdrec);
    }
    if (launch_status() != LW_OK) return LW_ECUDA;

    AdjArgs a{};
    a.n_e = traj->n_e;
    a.ns1 = traj->n_s + 1;
    a.t_per_e = traj->t_per_electron;
    a.t = traj->t;
    a.r = traj->r;
    a.beta = traj->beta;
    a.bdot = traj->beta_dot;
    a.n_hat = det->n_hat;
    a.n_pix = det->n_pix;
    a.t_min = grid->t_min;
    a.dt_u = grid->dt_u;
    a.inv_dtu = 1.0 / grid->dt_u;
    a.n_bins = N;
    a.dLdrec = dLdrec;
    a.g_r = dL_dr;
    a.g_beta = dL_dbeta;
    a.g_bdot = dL_dbeta_dot;
    const int64_t tiles = (det->n_pix + kAdjThreads - 1) / kAdjThreads;
    a.e_chunk = pick_chunk(traj->n_e, tiles);
    dim3 g((unsigned)tiles, (unsigned)((traj->n_e + a.e_chunk - 1) / a.e_chunk));
    if (!mixed) {
        // parts of an electron's steps until there are about 24 CTAs per SM (few electrons)
        const int64_t n_tiles = (a.ns1 + kAdjTile - 1) / kAdjTile, ctas = (int64_t)g.x * g.y;
        g.z = (unsigned)std::min<int64_t>(std::min<int64_t>(n_tiles, 65535),
                                          (kSms * 24 + ctas - 1) / ctas);
        adj_deposit_kernel<<<g, kAdjThreads, 0, st>>>(a);
        return launch_status();
    }
    char* fbase = base + rec_bytes + tw_bytes + y_bytes;
    float* Rf = reinterpret_cast<float*>(fbase);
    unsigned long long* mx =
        reinterpret_cast<unsigned long long*>(fbase + align256(sizeof(float) * (size_t)(rows * N)));
    double* rscale = reinterpret_cast<double*>(mx + 1);
    if (cudaMemsetAsync(mx, 0, sizeof(unsigned long long), st) != cudaSuccess) return LW_ECUDA;
    const int64_t n_rec = rows * N;
    const int rg = (int)std::min<int64_t>((n_rec + 255) / 256, (int64_t)kSms * 8);
    adj_absmax_kernel<<<rg, 256, 0, st>>>(dLdrec, n_rec, mx);
    adj_to_f32_kernel<<<rg, 256, 0, st>>>(dLdrec, det->n_pix, N, mx, Rf, rscale);
    if (launch_status() != LW_OK) return LW_ECUDA;
    a.dLdrec_f = Rf;
    a.rscale = rscale;
    a.f_grad = reinterpret_cast<float*>(fbase + align256(sizeof(float) * (size_t)(rows * N)) + 256);
    const int64_t n_samples = traj->n_e * (traj->n_s + 1);
    if (cudaMemsetAsync(a.f_grad, 0, sizeof(float) * 12 * (size_t)n_samples, st) != cudaSuccess)
        return LW_ECUDA;
    adj_deposit_mixed_kernel<<<g, kAdjThreads, 0, st>>>(a);
    if (launch_status() != LW_OK) return LW_ECUDA;
    const int fg = (int)std::min<int64_t>((n_samples + 255) / 256, (int64_t)kSms * 8);
    adj_finish_kernel<<<fg, 256, 0, st>>>(a.f_grad, n_samples, rscale, a.inv_dtu, a.g_r, a.g_beta,
                                          a.g_bdot);
    return launch_status();
}
