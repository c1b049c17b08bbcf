// Frequency-domain method (Eq. inty_dft / Algorithm 1 of the paper), the
// comparison method of the time-domain path, on a uniform frequency grid
// omega_w = omega0 + w * d_omega:
//   S(n, omega) = q^2 dt^2 / (16 pi^3 eps0 c0)
//                 | sum_k sum_i A_k(n, t_i) exp(j omega (t_i - n.r_ki / c0)) |^2,
//   A = n x ((n - beta) x beta_dot) / (1 - n.beta)^2.
//
// Per sample one thread computes in FP64 the phase time tau, the vector A (then rounded to
// FP32) and the phases omega_base tau (one per block of 1,024 frequencies), 32 d_omega tau and
// d_omega tau, reduced modulo 2 pi and kept as FP32 hi + lo pairs.  The twiddles
// exp(j (omega_base + 32 a d_omega) tau) and exp(j b d_omega tau), a, b = 0..31, follow in
// double-FP32 arithmetic (exact products, reduction by a two-float 2 pi) and one FP32 sincos
// each; a thread's twiddle for frequency w = 32 a + b is one complex product.  Per sample and
// frequency that leaves one complex product and six FMAs; partial sums over 16 samples are FP32
// and are added to compensated (two-float) totals.
//
// Bound: the FP32 pipe, busy 66 % of the active cycles, beside instruction issue at 56 %
// (32 electrons x 1,000 steps x 144 pixels x 2,048 frequencies; 10 operations per sample and
// frequency, 42 more per 16 samples).  The rest is kept off it or beside it: two warps of a CTA do
// the FP64 part ahead of the others through a ring of groups of 32 samples (an FP64 instruction
// holds a warp for 64 cycles), a CTA takes two blocks of frequencies so that they share it, two
// frequencies go into one packed FP32x2 instruction, and the CTAs of a cluster divide the samples
// and add their totals through distributed shared memory, so that few pixels fill the GPU.  64 electrons x 1,000 steps x 144
// pixels x 2,048 frequencies: 21.0 ms (16 threads per CTA doing the FP64 part between barriers)
// -> 11.1 ms.
#include <cooperative_groups.h>
#include <math.h>

#include "lw_internal.cuh"

namespace lw {
namespace {

constexpr int kFdmBlock = 1024;         // frequencies sharing a base phase
constexpr int kFdmGroup = 32;           // samples per ring slot (two partial sums of 16)
constexpr int kFdmSlots = 4;
constexpr int kFdmProducers = 2;        // warps
// named barriers: slot filled, slot free (one per slot), consumers
constexpr int kBarFull = 1, kBarFree = 1 + kFdmSlots, kBarCons = 1 + 2 * kFdmSlots;

struct FdmArgs {
    int64_t n_e, ns1;
    int t_per_e;
    const double* t;
    const double* r;
    const double* beta;
    const double* bdot;
    const double* n_hat;
    int64_t n_pix;
    double omega0, d_omega;
    int64_t n_omega;
    double scale;   // q^2 dt^2 / (16 pi^3 eps0 c0)
    double* S;
};

__device__ __forceinline__ double mod2pi(double x) {
    constexpr double two_pi = 2.0 * kPi;
    constexpr double inv_two_pi = 1.0 / (2.0 * kPi);
    return x - two_pi * floor(x * inv_two_pi);
}

// exp(j (base + a * step)) with base, step in [0, 2 pi) given as FP32 hi + lo pairs
__device__ __forceinline__ float2 twiddle(float bh, float bl, float sh, float sl, float a) {
    constexpr float two_pi_hi = 6.28318548202514648f;              // fl(2 pi)
    constexpr float two_pi_lo = -1.7484555314695172e-7f;           // 2 pi - fl(2 pi)
    const float p = a * sh;
    const float e = fmaf(a, sh, -p);                                // exact product error
    const float hi = __fadd_rn(p, bh);
    const float bb = __fsub_rn(hi, p);
    const float err = __fadd_rn(__fsub_rn(p, __fsub_rn(hi, bb)), __fsub_rn(bh, bb));
    const float lo = fmaf(a, sl, e) + bl + err;
    const float kq = rintf(hi * 0.159154943091895336f);
    const float ph = fmaf(-kq, two_pi_lo, fmaf(-kq, two_pi_hi, hi)) + lo;
    float s, c;
    sincosf(ph, &s, &c);
    return make_float2(c, s);
}

// hi, lo += v exactly (two-sum), for two totals at once
__device__ __forceinline__ void two_sum_add(float2& hi, float2& lo, float2 v) {
    const float2 m1 = make_float2(-1.0f, -1.0f);   // a - b as the exact b (-1) + a
    const float2 s = __fadd2_rn(hi, v);
    const float2 bb = __ffma2_rn(hi, m1, s);
    const float2 a = __ffma2_rn(__ffma2_rn(bb, m1, s), m1, hi);
    const float2 c = __ffma2_rn(bb, m1, v);
    hi = s;
    lo = __fadd2_rn(lo, __fadd2_rn(a, c));
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
    __syncwarp();
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// BLOCKS blocks of 1,024 frequencies per CTA, 256 threads each with four frequencies per thread:
// consumer warp v holds a = 4 v .. 4 v + 3 (of all its blocks' 32 BLOCKS values), lane b.
template <int BLOCKS>
struct FdmShared {
    float2 ph[kFdmSlots][kFdmGroup][BLOCKS + 2];   // base phases, 32 d_omega, d_omega (hi, lo)
    float4 A01[kFdmSlots][kFdmGroup];              // (A0, A0, A1, A1)
    float2 A2[kFdmSlots][kFdmGroup];               // (A2, A2)
    float4 e1[2][kFdmGroup][16 * BLOCKS];          // pairs of a: (x_a, x_a+1, y_a, y_a+1)
    float4 e2[2][kFdmGroup][32];                   // (x, x, y, y)
};
template <int BLOCKS>
constexpr int fdm_threads() { return 256 * BLOCKS + 32 * kFdmProducers; }
// the ring, reused at the end for six doubles per frequency
template <int BLOCKS>
constexpr size_t fdm_smem() {
    return sizeof(FdmShared<BLOCKS>) > 48 * (size_t)kFdmBlock * BLOCKS
               ? sizeof(FdmShared<BLOCKS>)
               : 48 * (size_t)kFdmBlock * BLOCKS;
}

template <int BLOCKS>
__global__ void __launch_bounds__(fdm_threads<BLOCKS>(), 3 - BLOCKS) fdm_kernel(FdmArgs p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FdmShared<BLOCKS>& sh = *reinterpret_cast<FdmShared<BLOCKS>*>(smem_raw);
    constexpr int kCons = 256 * BLOCKS;   // consumer threads
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t m = blockIdx.x;
    const int64_t w0 = (int64_t)blockIdx.y * kFdmBlock * BLOCKS;
    // this CTA's samples: whole groups
    const int64_t total = p.n_e * p.ns1;
    const int64_t groups = (total + kFdmGroup - 1) / kFdmGroup;
    const int64_t g0 = groups * blockIdx.z / gridDim.z, g1 = groups * (blockIdx.z + 1) / gridDim.z;
    if (warp >= kCons / 32) {   // ---- producers: FP64 per sample
        const double nx = p.n_hat[3 * m], ny = p.n_hat[3 * m + 1], nz = p.n_hat[3 * m + 2];
        for (int64_t g = g0 + (warp - kCons / 32); g < g1; g += kFdmProducers) {
            const int slot = (int)((g - g0) % kFdmSlots);
            if (g - g0 >= kFdmSlots) bar_sync(kBarFree + slot, kCons + 32);
            const int64_t q = g * kFdmGroup + lane;
            float2 ph[BLOCKS + 2];
            float A0f = 0.0f, A1f = 0.0f, A2f = 0.0f;
#pragma unroll
            for (int c = 0; c < BLOCKS + 2; ++c) ph[c] = make_float2(0.0f, 0.0f);
            if (q < total) {
                const int64_t k = q / p.ns1, i = q - k * p.ns1;
                const double* x = p.r + 3 * q;
                const double tt = p.t_per_e ? p.t[q] : p.t[i];
                const double tau = tt - ((nx * x[0] + ny * x[1]) + nz * x[2]) * kInvC0;
#pragma unroll
                for (int c = 0; c < BLOCKS + 2; ++c) {
                    const double f = c < BLOCKS ? p.omega0 + (double)(w0 + c * kFdmBlock) * p.d_omega
                                     : c == BLOCKS ? 32.0 * p.d_omega : p.d_omega;
                    const double v = mod2pi(f * tau);
                    const float h = (float)v;
                    ph[c] = make_float2(h, (float)(v - (double)h));
                }
                const double* b = p.beta + 3 * q;
                const double* a = p.bdot + 3 * q;
                const double D = 1.0 - ((nx * b[0] + ny * b[1]) + nz * b[2]);
                const double bb = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
                if (D > 0.0 && bb < 1.0) {
                    const double m0 = nx - b[0], m1 = ny - b[1], m2 = nz - b[2];
                    const double i0 = m1 * a[2] - m2 * a[1];
                    const double i1 = m2 * a[0] - m0 * a[2];
                    const double i2 = m0 * a[1] - m1 * a[0];
                    const double iD2 = 1.0 / (D * D);
                    A0f = (float)((ny * i2 - nz * i1) * iD2);
                    A1f = (float)((nz * i0 - nx * i2) * iD2);
                    A2f = (float)((nx * i1 - ny * i0) * iD2);
                }
            }
#pragma unroll
            for (int c = 0; c < BLOCKS + 2; ++c) sh.ph[slot][lane][c] = ph[c];
            sh.A01[slot][lane] = make_float4(A0f, A0f, A1f, A1f);
            sh.A2[slot][lane] = make_float2(A2f, A2f);
            bar_arrive(kBarFull + slot, kCons + 32);
        }
        // the slots still to be released
        for (int64_t g = g0 + (warp - kCons / 32); g < g1; g += kFdmProducers)
            if (g + kFdmSlots >= g1) bar_sync(kBarFree + (int)((g - g0) % kFdmSlots), kCons + 32);
    }
    // compensated totals of two frequencies each: [pair][component] real and imaginary
    float2 hr[2][3], hi[2][3], lr[2][3], li[2][3];
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            hr[f][c] = hi[f][c] = lr[f][c] = li[f][c] = make_float2(0.0f, 0.0f);
    if (warp < kCons / 32) {   // ---- consumers
        // twiddles of group g into buffer g & 1: 32 BLOCKS values of a and 32 of b per sample
        auto twiddles = [&](int64_t g) {
            const int slot = (int)((g - g0) % kFdmSlots), buf = (int)((g - g0) & 1);
            bar_sync(kBarFull + slot, kCons + 32);
            for (int job = threadIdx.x; job < kFdmGroup * 32; job += kCons) {
                const int s = job >> 5, b = job & 31;
                const float2 ph = sh.ph[slot][s][BLOCKS + 1];
                const float2 e = twiddle(0.0f, 0.0f, ph.x, ph.y, (float)b);
                sh.e2[buf][s][b] = make_float4(e.x, e.x, e.y, e.y);
            }
            for (int job = threadIdx.x; job < kFdmGroup * 32 * BLOCKS; job += kCons) {
                const int s = job / (32 * BLOCKS), a = job % (32 * BLOCKS);
                const float2 base = sh.ph[slot][s][a >> 5], st = sh.ph[slot][s][BLOCKS];
                const float2 e = twiddle(base.x, base.y, st.x, st.y, (float)(a & 31));
                float* d = reinterpret_cast<float*>(&sh.e1[buf][s][a >> 1]) + (a & 1);
                d[0] = e.x;
                d[2] = e.y;
            }
        };
        const bool any = w0 + 128 * warp < p.n_omega;   // the warp's 128 frequencies
        if (g0 < g1) twiddles(g0);
        for (int64_t g = g0; g < g1; ++g) {
            const int slot = (int)((g - g0) % kFdmSlots), buf = (int)((g - g0) & 1);
            bar_sync(kBarCons, kCons);   // twiddles of g complete, buffer of g - 1 free
            if (any) {
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
                    float2 pr[2][3], pi[2][3];
#pragma unroll
                    for (int f = 0; f < 2; ++f)
#pragma unroll
                        for (int c = 0; c < 3; ++c) pr[f][c] = pi[f][c] = make_float2(0.0f, 0.0f);
#pragma unroll 4
                    for (int s = 16 * half; s < 16 * half + 16; ++s) {
                        const float4 a01 = sh.A01[slot][s];
                        const float2 A[3] = {make_float2(a01.x, a01.y), make_float2(a01.z, a01.w),
                                             sh.A2[slot][s]};
                        const float4 e2 = sh.e2[buf][s][lane];
                        const float2 x2 = make_float2(e2.x, e2.y), y2 = make_float2(e2.z, e2.w);
                        const float2 n2 = make_float2(-e2.z, -e2.w);
#pragma unroll
                        for (int f = 0; f < 2; ++f) {
                            const float4 e1 = sh.e1[buf][s][2 * warp + f];
                            const float2 x1 = make_float2(e1.x, e1.y), y1 = make_float2(e1.z, e1.w);
                            // e1 e2, each part one product and one fused sum
                            const float2 tx = __ffma2_rn(x1, x2, __fmul2_rn(y1, n2));
                            const float2 ty = __ffma2_rn(x1, y2, __fmul2_rn(y1, x2));
#pragma unroll
                            for (int c = 0; c < 3; ++c) {
                                pr[f][c] = __ffma2_rn(A[c], tx, pr[f][c]);
                                pi[f][c] = __ffma2_rn(A[c], ty, pi[f][c]);
                            }
                        }
                    }
#pragma unroll
                    for (int f = 0; f < 2; ++f)
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            two_sum_add(hr[f][c], lr[f][c], pr[f][c]);
                            two_sum_add(hi[f][c], li[f][c], pi[f][c]);
                        }
                }
            }
            if (g + 1 < g1) twiddles(g + 1);
            bar_arrive(kBarFree + slot, kCons + 32);   // A of g and phases of g are used
        }
    }
    // totals in FP64, added over the cluster's CTAs; each CTA finishes a share of the frequencies
    __syncthreads();
    double* tot = reinterpret_cast<double*>(smem_raw);   // [frequency][6]
    if (warp < kCons / 32) {
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                double* d = tot + 6 * ((4 * warp + 2 * f + e) * 32 + lane);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    d[2 * c] = e ? (double)hr[f][c].y + (double)lr[f][c].y
                                 : (double)hr[f][c].x + (double)lr[f][c].x;
                    d[2 * c + 1] = e ? (double)hi[f][c].y + (double)li[f][c].y
                                     : (double)hi[f][c].x + (double)li[f][c].x;
                }
            }
    }
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int ranks = (int)cl.num_blocks(), share = kFdmBlock * BLOCKS / ranks;
    for (int q = threadIdx.x; q < share; q += blockDim.x) {
        const int idx = (int)cl.block_rank() * share + q;
        const int64_t w = w0 + idx;
        if (w >= p.n_omega) continue;
        double v[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int r = 0; r < ranks; ++r) {
            const double* o = cl.map_shared_rank(tot, r) + 6 * idx;
            for (int c = 0; c < 6; ++c) v[c] += o[c];
        }
        double sum = 0.0;
        for (int c = 0; c < 6; ++c) sum += v[c] * v[c];
        p.S[m * p.n_omega + w] = p.scale * sum;
    }
    cl.sync();   // the totals stay readable until every CTA has read them
}

template <int BLOCKS>
int launch_fdm(const FdmArgs& a, int64_t blocks, cudaStream_t st) {
    const auto kern = fdm_kernel<BLOCKS>;
    const size_t smem = fdm_smem<BLOCKS>();
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return LW_ECUDA;
    const int64_t gy = (blocks + BLOCKS - 1) / BLOCKS, ctas = a.n_pix * gy;
    const int64_t groups = (a.n_e * a.ns1 + kFdmGroup - 1) / kFdmGroup;
    // samples divided over clusters of 1, 2, 4 or 8 CTAs (at least 16 groups each), whichever
    // leaves the fewest idle SMs: CTAs fill an SM's registers, and clusters of 4 or 8 do not use every
    // SM of a GPC (eight parts on 144 pixels: a quarter of the SMs idle, 14.2 ms instead of 11.1)
    const int resident = 3 - BLOCKS;
    int parts = 1;
    double best = 1e300;
    for (int z = 1; z <= 8 && (z == 1 || groups >= 16 * z); z *= 2) {
        const int64_t slots = (int64_t)resident * (z <= 2 ? kSms : z == 4 ? 144 : 128);
        const double t = (double)((ctas * z + slots - 1) / slots) / z;
        if (t < 0.999 * best) {
            best = t;
            parts = z;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.n_pix, (unsigned)gy, (unsigned)parts);
    cfg.blockDim = dim3(fdm_threads<BLOCKS>());
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = (unsigned)parts;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, a) != cudaSuccess) return LW_ECUDA;
    return launch_status();
}

}  // namespace
}  // namespace lw

using namespace lw;

extern "C" int lw_spectrum_fdm(const lw_traj* traj, const lw_detector* det, double omega0,
                               double d_omega, int64_t n_omega, double dt, double q,
                               double* spectrum, void* stream) {
    if (!traj || !det || !spectrum || !det->n_hat || det->n_pix < 1 || n_omega < 1)
        return LW_EINVAL;
    if (!(traj->sections & LW_SECTION_FP64) || !traj->t || !traj->r) return LW_EINVAL;
    if (!isfinite(omega0) || !isfinite(d_omega) || !(dt > 0.0) || !isfinite(q)) return LW_EINVAL;
    if (det->n_pix > 2147483647LL || (n_omega + kFdmBlock - 1) / kFdmBlock > 65535)
        return LW_EUNSUPPORTED;
    FdmArgs a{};
    a.n_e = traj->n_e;
    a.ns1 = traj->n_s + 1;
    a.t_per_e = traj->t_per_electron;
    a.t = traj->t;
    a.r = traj->r;
    a.beta = traj->beta;
    a.bdot = traj->beta_dot;
    a.n_hat = det->n_hat;
    a.n_pix = det->n_pix;
    a.omega0 = omega0;
    a.d_omega = d_omega;
    a.n_omega = n_omega;
    a.scale = q * q * dt * dt / (16.0 * kPi * kPi * kPi * kEps0 * kC0);
    a.S = spectrum;
    // two blocks of 1,024 frequencies per CTA where their number is even
    const int64_t blocks = (n_omega + kFdmBlock - 1) / kFdmBlock;
    return blocks % 2 ? launch_fdm<1>(a, blocks, as_stream(stream))
                      : launch_fdm<2>(a, blocks, as_stream(stream));
}
