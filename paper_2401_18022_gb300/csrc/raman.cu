// Tabulated power profile from the Raman ODEs, and the quadratures that use it
// (arXiv 2401.18022, Sec. III and App. A: the profile term of Eq. pk comes
// from the Raman power-evolution ODEs, with the gain scaled by the effective
// area at the channel frequency).
//
// Model.  Channel k is a line of power P_k at f_k; with y_i = ln P_i
//   dy_i/dz = -alpha_i + s_i C_r sum_{k != i} h(f_k, f_i) P_k,
//   h = f_k - f_i               for 0 < f_k - f_i <= df_max  (k pumps i)
//   h = (f_k - f_i) f_i / f_k   for 0 < f_i - f_k <= df_max  (photon ratio;
//                                                              1 if disabled)
// so the partners of channel i form one index window [lo_i, hi_i] of the
// sorted plan, and the sum splits into prefix sums over the window:
//   above i:  sum (fr_k - fr_i) P_k = S(fr P) - fr_i S(P)
//   below i:  sum (fr_k - fr_i) (f_i / f_k) P_k = f_i (S(fr P / f) - fr_i S(P / f))
// (fr = f - f_ref), i.e. four block-wide scans per right-hand side instead of
// an n x n sum.  A slot with P = 0 pumps nothing and follows the gain of a
// zero-power probe (its y starts at 0).
//
// k_raman_ode   one block per profile: classical RK4 through the nodes
//               e_m -> z_m -> e_{m+1} of every z-step, each half in
//               half_steps[m] equal steps; tables
//                 a_c(m) = y_c(z_m) - y_c(0),  ln rho_c(L) = y_c(L) - y_c(0),
//                 b_c(m) = central difference over the neighbouring channels
//                          of the Raman part a + alpha z_m (one-sided at the
//                          plan's ends),
//               so that ln rho(z_m, F) = a_c(m) + b_c(m) (F - f_c) in channel c.
// k_quad_f32_tab, k_quad_f64_tab
//               the persistent quadratures of the closed-form kernels with
//               this profile.  For a grid point of piece (a, b) of CUT i with
//               F_c in candidate channel c,
//                 ln p_m = 1/2 [ln rho(F_a) + ln rho(F_b) + ln rho(F_c) - ln rho(f_i)]
//                        = A_c(m) + Sa_c(m) da + Sb_c(m) db,
//               da = F_a - f_a, db = F_b - f_b, A = (a_a + a_b + a_c - a_i +
//               b_c (f_a + f_b - f_i - f_c)) / 2, Sa = (b_a + b_c)/2,
//               Sb = (b_b + b_c)/2, tabulated per piece and candidate, so a
//               grid point costs the same two FMAs per step as the closed form.
#include <cuda_runtime.h>

#include <algorithm>

#include "isrs_internal.cuh"
#include "isrs_kernels.h"
#include "quad_common.cuh"
#include "quad_nodes.cuh"
#include "quad_tab.cuh"
#include "quad_zsum.cuh"

namespace isrs {

namespace {

constexpr int kOdeThreads = 1024;

// Exclusive prefix sums of four arrays v0..v3 [0, n) into x0..x3 [0, n]
// (x[k] = sum_{j<k} v[j]), all in shared memory.  Each thread scans a run of
// ceil(n / blockDim) consecutive entries; run totals are scanned by warp
// shuffles.  Called by every thread of the block.
__device__ void scan4(const double *v0, const double *v1, const double *v2, const double *v3, double *x0,
                      double *x1, double *x2, double *x3, int n, double *wsum /* [4 * 32] */)
{
    const int per = (n + blockDim.x - 1) / blockDim.x;
    const int b = threadIdx.x * per, e = min(n, b + per);
    double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;
    for (int k = b; k < e; ++k) {
        t0 += v0[k];
        t1 += v1[k];
        t2 += v2[k];
        t3 += v3[k];
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    double i0 = t0, i1 = t1, i2 = t2, i3 = t3;            // inclusive within the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u0 = __shfl_up_sync(0xffffffffu, i0, o), u1 = __shfl_up_sync(0xffffffffu, i1, o);
        const double u2 = __shfl_up_sync(0xffffffffu, i2, o), u3 = __shfl_up_sync(0xffffffffu, i3, o);
        if (lane >= o) {
            i0 += u0;
            i1 += u1;
            i2 += u2;
            i3 += u3;
        }
    }
    if (lane == 31) {
        wsum[wid] = i0;
        wsum[32 + wid] = i1;
        wsum[64 + wid] = i2;
        wsum[96 + wid] = i3;
    }
    __syncthreads();
    if (wid == 0) {
        double w0 = lane < nw ? wsum[lane] : 0.0, w1 = lane < nw ? wsum[32 + lane] : 0.0;
        double w2 = lane < nw ? wsum[64 + lane] : 0.0, w3 = lane < nw ? wsum[96 + lane] : 0.0;
        const double s0 = w0, s1 = w1, s2 = w2, s3 = w3;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double u0 = __shfl_up_sync(0xffffffffu, w0, o), u1 = __shfl_up_sync(0xffffffffu, w1, o);
            const double u2 = __shfl_up_sync(0xffffffffu, w2, o), u3 = __shfl_up_sync(0xffffffffu, w3, o);
            if (lane >= o) {
                w0 += u0;
                w1 += u1;
                w2 += u2;
                w3 += u3;
            }
        }
        if (lane < nw) {                                  // exclusive warp offsets
            wsum[lane] = w0 - s0;
            wsum[32 + lane] = w1 - s1;
            wsum[64 + lane] = w2 - s2;
            wsum[96 + lane] = w3 - s3;
        }
    }
    __syncthreads();
    double r0 = wsum[wid] + i0 - t0, r1 = wsum[32 + wid] + i1 - t1;
    double r2 = wsum[64 + wid] + i2 - t2, r3 = wsum[96 + wid] + i3 - t3;
    for (int k = b; k < e; ++k) {
        x0[k] = r0;
        x1[k] = r1;
        x2[k] = r2;
        x3[k] = r3;
        r0 += v0[k];
        r1 += v1[k];
        r2 += v2[k];
        r3 += v3[k];
    }
    if (threadIdx.x == blockDim.x - 1) {                  // its running sum is the total
        x0[n] = r0;
        x1[n] = r1;
        x2[n] = r2;
        x3[n] = r3;
    }
    __syncthreads();
}

struct OdeShared {
    double *y, *yt, *kacc, *ev0, *ev1, *ev2, *ev3, *x0, *x1, *x2, *x3;
};

// dy/dz at state Y into K (shared arrays; every thread calls).
__device__ void raman_rhs(const RamanParams &rp, int coff, int poff, int n, const double *Y, double *K,
                          const OdeShared &s, double *wsum)
{
    const double *fr = rp.ch_frel + coff;
    const double *P0 = rp.P + poff;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const double e = P0[k] > 0.0 ? exp(Y[k]) : 0.0;
        const double invf = 1.0 / (fr[k] + rp.f_ref);
        s.ev0[k] = e;
        s.ev1[k] = fr[k] * e;
        s.ev2[k] = e * invf;
        s.ev3[k] = fr[k] * e * invf;
    }
    __syncthreads();
    scan4(s.ev0, s.ev1, s.ev2, s.ev3, s.x0, s.x1, s.x2, s.x3, n, wsum);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int lo = rp.win_lo[coff + i], hi = rp.win_hi[coff + i];
        const double fri = fr[i];
        // partners above i: k in (i, hi]
        double g = 0.0;
        if (hi > i) g += (s.x1[hi + 1] - s.x1[i + 1]) - fri * (s.x0[hi + 1] - s.x0[i + 1]);
        // partners below i: k in [lo, i)
        if (lo < i) {
            if (rp.photon)
                g += (fri + rp.f_ref) * ((s.x3[i] - s.x3[lo]) - fri * (s.x2[i] - s.x2[lo]));
            else
                g += (s.x1[i] - s.x1[lo]) - fri * (s.x0[i] - s.x0[lo]);
        }
        K[i] = -rp.ch_alpha[coff + i] + rp.ch_scale[coff + i] * rp.Cr * g;
    }
    __syncthreads();
}

}  // namespace

__global__ void __launch_bounds__(kOdeThreads) k_raman_ode(RamanParams rp)
{
    extern __shared__ double smem_d[];
    __shared__ double wsum[128];
    const int p = blockIdx.x;
    const int plan = rp.prof_plan[p];
    const int n = rp.plan_n[plan];
    const int coff = rp.plan_ch_off[plan];
    const int poff = rp.prof_ch_off[p];
    const int M = rp.n_steps;
    OdeShared s;
    s.y = smem_d;
    s.yt = s.y + n;
    s.kacc = s.yt + n;
    s.ev0 = s.kacc + n;
    s.ev1 = s.ev0 + n;
    s.ev2 = s.ev1 + n;
    s.ev3 = s.ev2 + n;
    s.x0 = s.ev3 + n;
    s.x1 = s.x0 + n + 1;
    s.x2 = s.x1 + n + 1;
    s.x3 = s.x2 + n + 1;
    double *K = s.x3 + n + 1;                 // [n] stage slope
    double *y0 = K + n;                       // [n] initial state
    const double *P0 = rp.P + poff;
    double2 *ab = rp.ab + (size_t)poff * M;
    double *yn = (p == 0) ? rp.y_nodes : nullptr;

    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        const double v = P0[c] > 0.0 ? log(P0[c]) : 0.0;
        s.y[c] = v;
        y0[c] = v;
    }
    __syncthreads();
    int node = 0;
    for (int m = 0; m < M; ++m) {
        const int ns = rp.half_steps[m];
        const double h = 0.5 * rp.zs_d[m].y / ns;
        for (int half = 0; half < 2; ++half) {
            for (int t = 0; t < ns; ++t) {
                if (yn)
                    for (int c = threadIdx.x; c < n; c += blockDim.x) yn[(size_t)node * n + c] = s.y[c];
                ++node;
                raman_rhs(rp, coff, poff, n, s.y, K, s, wsum);                   // k1
                for (int c = threadIdx.x; c < n; c += blockDim.x) {
                    s.kacc[c] = K[c];
                    s.yt[c] = s.y[c] + 0.5 * h * K[c];
                }
                __syncthreads();
                raman_rhs(rp, coff, poff, n, s.yt, K, s, wsum);                  // k2
                for (int c = threadIdx.x; c < n; c += blockDim.x) {
                    s.kacc[c] += 2.0 * K[c];
                    s.yt[c] = s.y[c] + 0.5 * h * K[c];
                }
                __syncthreads();
                raman_rhs(rp, coff, poff, n, s.yt, K, s, wsum);                  // k3
                for (int c = threadIdx.x; c < n; c += blockDim.x) {
                    s.kacc[c] += 2.0 * K[c];
                    s.yt[c] = s.y[c] + h * K[c];
                }
                __syncthreads();
                raman_rhs(rp, coff, poff, n, s.yt, K, s, wsum);                  // k4
                for (int c = threadIdx.x; c < n; c += blockDim.x) s.y[c] += h / 6.0 * (s.kacc[c] + K[c]);
                __syncthreads();
            }
            if (half == 0)
                for (int c = threadIdx.x; c < n; c += blockDim.x) ab[(size_t)c * M + m].x = s.y[c] - y0[c];
        }
    }
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        rp.lnrho_L[poff + c] = s.y[c] - y0[c];
        if (yn) yn[(size_t)node * n + c] = s.y[c];
    }
    __syncthreads();
    // in-channel slopes: central differences of a + alpha z_m
    const double *fr = rp.ch_frel + coff;
    const double *al = rp.ch_alpha + coff;
    for (int t = threadIdx.x; t < n * M; t += blockDim.x) {
        const int c = t / M, m = t - c * M;
        const int lo = c > 0 ? c - 1 : 0, hi = c < n - 1 ? c + 1 : n - 1;
        double b = 0.0;
        if (hi != lo) {
            const double zm = rp.zs_d[m].x;
            const double rlo = ab[(size_t)lo * M + m].x + al[lo] * zm;
            const double rhi = ab[(size_t)hi * M + m].x + al[hi] * zm;
            b = (rhi - rlo) / (fr[hi] - fr[lo]);
        }
        ab[(size_t)c * M + m].y = b;
    }
}

size_t raman_smem_bytes(int n_ch)
{
    return sizeof(double) * (size_t)(13 * n_ch + 4);
}

cudaError_t launch_raman(const RamanParams &rp, int n_prof, int max_n, cudaStream_t st)
{
    const size_t smem = raman_smem_bytes(max_n);
    cudaError_t e = cudaFuncSetAttribute(k_raman_ode, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_raman_ode<<<n_prof, kOdeThreads, smem, st>>>(rp);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Discrete adjoint of the profile (single profile, plan 0).
//
// T depends on the tables through a_c(m) = y_c(z_m) - y_c(0), b_c(m) (central
// differences of a + alpha z) and ln rho_c(L) = y_c(L) - y_c(0).  k_fold_slope
// moves dT/db onto dT/da (the stencil), k_raman_adj runs the RK4 steps
// backwards: with lambda = dT/dy after a step y' = y + h/6 (k1 + 2k2 + 2k3 + k4),
//   mu4 = J(Y4)^T (h/6 lambda),            mu3 = J(Y3)^T (h/3 lambda + h mu4),
//   mu2 = J(Y2)^T (h/3 lambda + h/2 mu3),  mu1 = J(Y1)^T (h/6 lambda + h/2 mu2),
//   dT/dy = lambda + mu1 + mu2 + mu3 + mu4,
// with the stage states Y recomputed from the stored step states, the table
// sensitivities injected at the nodes z_m and L, and
//   (J^T v)_k = C_r e^{Y_k} sum_i s_i v_i h(f_k, f_i)
// again by prefix sums over the partner window of k:
//   i below k:  sum u_i (fr_k - fr_i)              = fr_k S(u) - S(fr u)
//   i above k:  sum u_i (fr_k - fr_i) f_i / f_k    = (fr_k S(f u) - S(fr f u)) / f_k
// (u = s v; the ratio f_i/f_k is 1 without the photon term).  Finally
//   dT/dP_j = (dT/dy_j(0) + dT/d ln P_j|_PSD) / P_j + dT/dSNR_j dSNR_j/dP_j|_N.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_fold_slope(RamanAdjParams ap)
{
    const int n = ap.n, M = ap.r.n_steps;
    const double *fr = ap.r.ch_frel;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * M; t += gridDim.x * blockDim.x) {
        const int c = t / M, m = t - c * M;
        double g = ap.gAB[t].x;
        for (int q = max(0, c - 1); q <= min(n - 1, c + 1); ++q) {
            const int lo = q > 0 ? q - 1 : 0, hi = q < n - 1 ? q + 1 : n - 1;
            if (lo == hi) continue;
            const double gb = ap.gAB[(size_t)q * M + m].y / (fr[hi] - fr[lo]);
            if (hi == c) g += gb;
            if (lo == c) g -= gb;
        }
        ap.gAt[t] = g;
    }
}

namespace {

// out = J(Y)^T v (shared arrays; every thread calls)
__device__ void raman_jt(const RamanParams &rp, int n, const double *Y, const double *v, double *out,
                         const OdeShared &s, double *wsum)
{
    const double *fr = rp.ch_frel;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double u = rp.ch_scale[i] * v[i];
        const double f = fr[i] + rp.f_ref;
        s.ev0[i] = u;
        s.ev1[i] = fr[i] * u;
        s.ev2[i] = f * u;
        s.ev3[i] = fr[i] * f * u;
    }
    __syncthreads();
    scan4(s.ev0, s.ev1, s.ev2, s.ev3, s.x0, s.x1, s.x2, s.x3, n, wsum);
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        double r = 0.0;
        if (rp.P[k] > 0.0) {
            const int lo = rp.win_lo[k], hi = rp.win_hi[k];
            const double frk = fr[k];
            double g = 0.0;
            if (lo < k) g += frk * (s.x0[k] - s.x0[lo]) - (s.x1[k] - s.x1[lo]);
            if (hi > k) {
                if (rp.photon)
                    g += (frk * (s.x2[hi + 1] - s.x2[k + 1]) - (s.x3[hi + 1] - s.x3[k + 1])) / (frk + rp.f_ref);
                else
                    g += frk * (s.x0[hi + 1] - s.x0[k + 1]) - (s.x1[hi + 1] - s.x1[k + 1]);
            }
            r = rp.Cr * exp(Y[k]) * g;
        }
        out[k] = r;
    }
    __syncthreads();
}

}  // namespace

__global__ void __launch_bounds__(kOdeThreads) k_raman_adj(RamanAdjParams ap)
{
    extern __shared__ double smem_d[];
    __shared__ double wsum[128];
    const RamanParams &rp = ap.r;
    const int n = ap.n, M = rp.n_steps;
    double *lam = smem_d, *acc = lam + n, *w = acc + n, *mu = w + n, *Y2 = mu + n, *Y3 = Y2 + n, *Y4 = Y3 + n;
    OdeShared s;
    s.y = s.yt = s.kacc = nullptr;
    s.ev0 = Y4 + n;
    s.ev1 = s.ev0 + n;
    s.ev2 = s.ev1 + n;
    s.ev3 = s.ev2 + n;
    s.x0 = s.ev3 + n;
    s.x1 = s.x0 + n + 1;
    s.x2 = s.x1 + n + 1;
    s.x3 = s.x2 + n + 1;

    for (int c = threadIdx.x; c < n; c += blockDim.x)
        lam[c] = ap.with_direct ? -ap.aase[c] : 0.0;                               // dT/d ln rho(L)
    __syncthreads();
    int node = ap.n_rk;
    for (int m = M - 1; m >= 0; --m) {
        const int ns = rp.half_steps[m];
        const double h = 0.5 * rp.zs_d[m].y / ns;
        for (int half = 1; half >= 0; --half) {
            for (int t = 0; t < ns; ++t) {
                --node;
                const double *Y1 = ap.y_nodes + (size_t)node * n;
                // stage states of this step
                raman_rhs(rp, 0, 0, n, Y1, mu, s, wsum);
                for (int c = threadIdx.x; c < n; c += blockDim.x) Y2[c] = Y1[c] + 0.5 * h * mu[c];
                __syncthreads();
                raman_rhs(rp, 0, 0, n, Y2, mu, s, wsum);
                for (int c = threadIdx.x; c < n; c += blockDim.x) Y3[c] = Y1[c] + 0.5 * h * mu[c];
                __syncthreads();
                raman_rhs(rp, 0, 0, n, Y3, mu, s, wsum);
                for (int c = threadIdx.x; c < n; c += blockDim.x) {
                    Y4[c] = Y1[c] + h * mu[c];
                    acc[c] = lam[c];
                    w[c] = h / 6.0 * lam[c];
                }
                __syncthreads();
                raman_jt(rp, n, Y4, w, mu, s, wsum);                         // mu4
                for (int c = threadIdx.x; c < n; c += blockDim.x) {
                    acc[c] += mu[c];
                    w[c] = h / 3.0 * lam[c] + h * mu[c];
                }
                __syncthreads();
                raman_jt(rp, n, Y3, w, mu, s, wsum);                         // mu3
                for (int c = threadIdx.x; c < n; c += blockDim.x) {
                    acc[c] += mu[c];
                    w[c] = h / 3.0 * lam[c] + 0.5 * h * mu[c];
                }
                __syncthreads();
                raman_jt(rp, n, Y2, w, mu, s, wsum);                         // mu2
                for (int c = threadIdx.x; c < n; c += blockDim.x) {
                    acc[c] += mu[c];
                    w[c] = h / 6.0 * lam[c] + 0.5 * h * mu[c];
                }
                __syncthreads();
                raman_jt(rp, n, Y1, w, mu, s, wsum);                         // mu1
                for (int c = threadIdx.x; c < n; c += blockDim.x) lam[c] = acc[c] + mu[c];
                __syncthreads();
            }
            if (half == 1)
                for (int c = threadIdx.x; c < n; c += blockDim.x) lam[c] += ap.gAt[(size_t)c * M + m];
            __syncthreads();
        }
    }
    // a = y - y(0): every table entry also depends on y(0) directly
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        double direct = ap.with_direct ? ap.aase[j] : 0.0;             // - dT/d ln rho(L)
        for (int m = 0; m < M; ++m) direct -= ap.gAt[(size_t)j * M + m];
        const double P = rp.P[j];
        double g = (lam[j] + direct + ap.gV[j]) / P;
        if (ap.with_direct) {                                          // the SNR numerator
            const double snr = ap.snr[j], B = ap.ch_B[j];
            const double N = ap.pnli[j] + ap.pase[j];
            const double dTds = 2.0 * B / (0.69314718055994530942 * (1.0 + snr));
            g += dTds * snr * snr * N / (P * P);
        }
        ap.dT_dP[j] = g;
    }
}

size_t raman_adj_smem_bytes(int n_ch)
{
    return sizeof(double) * (size_t)(15 * n_ch + 4);
}

cudaError_t launch_raman_adj(const RamanAdjParams &ap, cudaStream_t st)
{
    const int nm = ap.n * ap.r.n_steps;
    k_fold_slope<<<(nm + 255) / 256, 256, 0, st>>>(ap);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t smem = raman_adj_smem_bytes(ap.n);
    e = cudaFuncSetAttribute(k_raman_adj, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_raman_adj<<<1, kOdeThreads, smem, st>>>(ap);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Quadratures with the tabulated profile.
// ---------------------------------------------------------------------------
constexpr int kTabSlots = 192;       // node slots of a chunk
constexpr int kTabCand = 2;          // F_c candidates swept together (most pieces have two)
using TabNodes = WarpNodes<kTabSlots>;

// Dynamic shared memory of k_quad_f32_tab: zt [M], then per warp the nodes and
// the candidates' step rows.
__host__ __device__ constexpr size_t tab_warp_bytes(int n_steps)
{
    return sizeof(TabNodes) + sizeof(float4) * kTabCand * (size_t)n_steps;
}

// As k_quad_f32 (quad_fwd.cu: one warp per tile, row sums from nodes), with the
// step rows of the tabulated profile.  The low rows' blocks replace the 2-D
// contraction of the small-phase moments (176 coefficients per candidate and
// piece) that this kernel used to build.
__global__ void __launch_bounds__(256, 4) k_quad_f32_tab(QuadParams qp)
{
    extern __shared__ float4 smem_f4[];
    const int M = qp.n_steps, G = qp.G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4 *zt = smem_f4;                              // [M] {edge(m+1)/2pi hi, lo, z, dz}
    unsigned char *mine = reinterpret_cast<unsigned char *>(zt + M) + tab_warp_bytes(M) * warp;
    TabNodes &ns = *reinterpret_cast<TabNodes *>(mine);
    float4 *Q = reinterpret_cast<float4 *>(mine + sizeof(TabNodes));   // [kTabCand][M]

    for (int m = threadIdx.x; m < M; m += blockDim.x) {
        const float4 za = qp.zs_a[m], zb = qp.zs_b[m];
        zt[m] = make_float4(zb.x, zb.y, za.x, za.w);
    }
    __syncthreads();
    const float phi_direct = 3.14159265f / qp.dz_max;
    const float phi_small = kBlkPhiL / qp.L;
    unsigned long long n_small = 0;
    unsigned n_direct = 0, n_tele = 0;

    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(qp.counter, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= qp.n_items) break;
        const DevItem item = qp.items[it];
        const int part = item.part & 0xffff, parts = item.part >> 16;
        double acc = 0.0;
        for (int k = item.piece0; k < item.piece1; ++k) {
            const DevPiece &pc = qp.pieces[dbg_clamp(k, qp.n_pieces, kDbgPiece, qp.dbg)];
            __syncwarp();
            const bool sw = node_geo(qp, pc, item.prof, 0.0f, qp.pd_f, 0.0f, ns.geo);
            const TabPiece tp = tab_piece(qp, pc, item.prof, sw);
            const int coff = qp.plan_ch_off[pc.plan];
            __syncwarp();
            PieceGeo &g = ns.geo;
            float sum = 0.0f, comp = 0.0f;
            for (int ca = 0; ca < g.nc; ca += kTabCand) {
                const int cb = min(g.nc, ca + kTabCand);
                float tilt = 0.0f;
                for (int c = ca; c < cb; ++c) {
                    const double fc = qp.ch_frel[coff + pc.c_lo + c];
                    for (int m = lane; m < M; m += 32) {
                        const float4 r = tab_row(tp, pc.c_lo + c, fc, m, M);
                        Q[(c - ca) * M + m] = r;
                        tilt = fmaxf(tilt, fmaxf(fabsf(r.y), fabsf(r.z)));
                    }
                }
                // the largest slope of ln p bounds its swing along a row
                tilt = 0.69314718f * __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(tilt)));
                if (lane == 0) g.tilt = tilt;
                __syncwarp();
                int small;
                piece_nodes(ns, qp.gauss, G, ca, cb, small, [&](int nq) {
                    for (int q = lane + 32 * part; q < nq; q += 32 * parts) {
                        Node nd;
                        if (!node_get(ns, qp.gauss, q, nd)) continue;
                        const int ci = dbg_clamp(nd.ci, g.nc, kDbgCand, qp.dbg);
                        const float aphi = fabsf(nd.phi);
                        const float dl = tp.ol + nd.x, dd = tp.od + nd.y;
                        const float4 *e = Q + (ci - ca) * M;
                        const bool direct = aphi <= phi_direct;
                        const float S2 = direct ? zsum_direct_nt(nd.phi, dl, dd, zt, e, M)
                                                : zsum_tele_nt(nd.phi, nd.phi_lo, dl, dd, zt, e, M);
                        n_small += aphi <= phi_small ? nd.N : 0;
                        n_direct += aphi > phi_small && direct ? nd.N : 0;
                        n_tele += direct ? 0 : nd.N;
                        const float y = nd.wq * g.pd[ci] * S2 * array_factor_f(nd.phi, qp, nd.phi_lo) - comp;
                        const float t = sum + y;
                        comp = (t - sum) - y;
                        sum = t;
                    }
                });
                n_small += lane == 0 && part == 0 ? small : 0;
            }
            acc += (double)(g.mult * g.wab) * ((double)sum - (double)comp);
        }
        const double tot = warp_sum_d(acc);
        if (lane == 0) qp.partial[it] = tot;
    }
    if (qp.path_count) {
        unsigned long long c0 = n_small, c1 = n_direct, c2 = n_tele;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            c0 += __shfl_xor_sync(0xffffffffu, c0, o);
            c1 += __shfl_xor_sync(0xffffffffu, c1, o);
            c2 += __shfl_xor_sync(0xffffffffu, c2, o);
        }
        if (lane == 0) {
            atomicAdd(&qp.path_count[0], c0);
            atomicAdd(&qp.path_count[1], c1);
            atomicAdd(&qp.path_count[2], c2);
        }
    }
}

// Plain FP64 quadrature with the tabulated profile (direct form, libm).
__global__ void __launch_bounds__(256) k_quad_f64_tab(QuadParams qp)
{
    extern __shared__ double2 smem_d2[];
    const int M = qp.n_steps, G = qp.G;
    double2 *sz = smem_d2;                              // [M] {z_m, dz_m}
    double2 *sQ = sz + M;                               // [nc_max][M][2] {A, Sa}, {Sb, 0}
    RowD *rows = reinterpret_cast<RowD *>(sQ + (size_t)2 * qp.nc_max * M);
    __shared__ PieceConst<double> kc;
    __shared__ double s_d0[2];
    __shared__ double scratch[32];
    __shared__ int s_item;

    for (int m = threadIdx.x; m < M; m += blockDim.x) sz[m] = qp.zs_d[m];
    const double c3 = kPi * qp.beta3;
    const double c4 = 2.0 * kPi * kPi / 3.0 * qp.beta4;

    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(qp.counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= qp.n_items) break;
        const DevItem item = qp.items[it];
        double acc = 0.0;
        for (int k = item.piece0; k < item.piece1; ++k) {
            const DevPiece pc = qp.pieces[dbg_clamp(k, qp.n_pieces, kDbgPiece, qp.dbg)];
            piece_rows<RowD>(pc, G, qp.eps_v1, rows);
            piece_consts<double>(qp, pc, item.prof, 0.0, qp.pd_d, kc);
            const int coff = qp.plan_ch_off[pc.plan];
            const double fa = qp.ch_frel[coff + pc.a], fb = qp.ch_frel[coff + pc.b];
            const double fic = qp.ch_frel[coff + pc.cut];
            if (threadIdx.x == 0) {
                s_d0[0] = fa - fic;
                s_d0[1] = fb - fic;
            }
            {
                const double2 *T = qp.ab + (size_t)qp.prof_ch_off[item.prof] * M;
                const int nc = min(pc.c_hi - pc.c_lo + 1, kMaxCand);
                for (int t = threadIdx.x; t < nc * M; t += blockDim.x) {
                    const int ci = t / M, m = t - ci * M;
                    const int c = pc.c_lo + ci;
                    const double2 ta = T[(size_t)pc.a * M + m], tb = T[(size_t)pc.b * M + m];
                    const double2 ti = T[(size_t)pc.cut * M + m], tc = T[(size_t)c * M + m];
                    const double D = (fa + fb) - (fic + qp.ch_frel[coff + c]);
                    sQ[2 * t] = make_double2(0.5 * (ta.x + tb.x + tc.x - ti.x + tc.y * D), 0.5 * (ta.y + tc.y));
                    sQ[2 * t + 1] = make_double2(0.5 * (tb.y + tc.y), 0.0);
                }
            }
            __syncthreads();
            const double fi = kc.fi;
            const double da0 = s_d0[0], db0 = s_d0[1];
            double sum = 0.0;
            const int npts = G * G;
            for (int q = threadIdx.x + (item.part & 0xffff) * blockDim.x; q < npts; q += (item.part >> 16) * blockDim.x) {
                const int r = q / G;
                const int j = q - r * G;
                const RowD rw = rows[dbg_clamp(r, G, kDbgRow, qp.dbg)];
                if (rw.w == 0.0) continue;
                const double d = ((double)j + 0.5 - 0.5 * (double)G) * rw.du2;
                const double f1 = kc.s1 * (rw.xc * exp(d));
                const double f2 = kc.s2 * (rw.yc * exp(-d));
                const double u = f1 + f2;
                int ci = -1;
                for (int c = 0; c < kc.nc; ++c) {
                    if (u >= kc.lo[c] && u < kc.hi[c]) { ci = c; break; }
                }
                if (ci < 0) continue;
                const double W = kc.wab * kc.pd[ci];
                const double da = f1 - da0, db = f2 - db0;
                const double br = qp.beta2 + c3 * (u + 2.0 * fi) +
                                  c4 * (f1 * f1 + 1.5 * f1 * f2 + 3.0 * fi * u + f2 * f2 + 3.0 * fi * fi);
                const double phi = -4.0 * kPi * kPi * f1 * f2 * br;
                const double2 *Q = sQ + (size_t)2 * ci * M;
                double Sr = 0.0, Si = 0.0;
                for (int m = 0; m < M; ++m) {
                    const double2 zz = sz[m];
                    const double2 q0 = Q[2 * m], q1 = Q[2 * m + 1];
                    const double p = exp(q0.x + q0.y * da + q1.x * db);
                    const double amp = p * zz.y * sinc_d(0.5 * phi * zz.y);
                    double sn, cs;
                    sincos(phi * zz.x, &sn, &cs);
                    Sr += amp * cs;
                    Si += amp * sn;
                }
                sum += rw.w * W * (Sr * Sr + Si * Si) * array_factor_d(phi, qp);
            }
            acc += kc.mult * sum;
            __syncthreads();
        }
        const double tot = block_sum_d(acc, scratch);
        if (threadIdx.x == 0) qp.partial[it] = tot;
    }
}

size_t quad_tab_limit_bytes(int precision, int n_steps, int G, int nc_max)
{
    if (precision == 0)
        return (size_t)n_steps * (6 + nc_max) * 16 + (size_t)nc_max * 704 + (size_t)n_steps * 80 + (size_t)G * 16;
    return (size_t)n_steps * (1 + 2 * nc_max) * sizeof(double2) + (size_t)G * sizeof(RowD);
}

cudaError_t launch_quad_tab(const QuadParams &qp, int precision, int num_sms, int block, cudaStream_t st)
{
    int nb = 0, tiles = qp.n_items;
    size_t smem = quad_tab_limit_bytes(1, qp.n_steps, qp.G, qp.nc_max);
    const void *fn = (const void *)k_quad_f64_tab;
    if (precision == 0) {
        // as launch_quad: any number of warps to a block
        const auto bytes = [&](int b) { return sizeof(float4) * (size_t)qp.n_steps + tab_warp_bytes(qp.n_steps) * (b / 32); };
        fn = (const void *)k_quad_f32_tab;
        if (qp.n_items < num_sms * (block / 32)) block = 32;
        while (block > 32 && bytes(block) > 200 * 1024) block -= 32;
        smem = bytes(block);
        tiles = (qp.n_items + block / 32 - 1) / (block / 32);
    }
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, block, smem);
    if (e != cudaSuccess) return e;
    const int grid = std::max(1, std::min(tiles, num_sms * std::max(1, nb)));
    void *args[] = {(void *)&qp};
    return cudaLaunchKernel(fn, dim3(grid), dim3(block), args, smem, st);
}

}  // namespace isrs
