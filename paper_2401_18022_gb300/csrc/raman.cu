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
// (fr = f - f_ref), i.e. four prefix sums per right-hand side instead of an
// n x n sum.  A slot with P = 0 pumps nothing and follows the gain of a
// zero-power probe (its y starts at 0).
//
// k_raman_ode   one cluster per profile: classical RK4 through the nodes
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
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "isrs_internal.cuh"
#include "isrs_kernels.h"
#include "quad_common.cuh"
#include "quad_nodes.cuh"
#include "quad_tab.cuh"
#include "quad_zsum.cuh"

namespace isrs {

namespace cg = cooperative_groups;

namespace {

// The ODE kernels run one thread-block cluster per profile, one lane per
// channel.  A right-hand side is a chain of short FP64 steps (exp, prefix sums,
// combination), ~1,800 of them one after another over 80 km.  On one SM the
// FP64 pipe (2 lanes a clock) and the block barriers of a 1,024-thread scan took
// 18 us each on the 557-channel plan (12.5 us on 41 channels); with two warps to an
// SM and one cluster barrier a stage they take 3.5 us (2.7 us).
constexpr int kOdeWarps = 2;             // warps of a block at most 32 warps of channels
constexpr int kOdeMaxCluster = 16;
constexpr int kOdeMaxWarps = kMaxRamanCh / 32;

// Window sums over the sorted plan, one channel per lane.  Every warp scans its
// 32 channels; the in-warp inclusive prefixes stay in their block's shared
// memory (read remotely at the window's two ends), the warps' totals are pushed
// to every block.  Double-buffered, so one cluster barrier per call suffices: a
// buffer is written again two calls later, after the barrier in between.  (The first
// stores wait for the cluster at the end of ode_lane.)
struct OdeWindow {
    double2 x[2][2][32 * kOdeMaxWarps / 8];      // [buffer][pair][channel of the block]
    double2 tot[2][2][kOdeMaxWarps];             // [buffer][pair][warp of the plan]
};

struct OdeLane {
    int n, i, wpc;                // channels, this lane's, warps per block
    bool live;
    bool one;                     // the cluster is one block: its own barrier and shared memory do
    int jhi, jlo;                 // hi and lo - 1
    int wi, whi, wlo;             // warps of i, of the window's last, of the one before its first
    bool has_lo;                  // the window does not start at channel 0
    const double2 *xhi, *xlo;     // remote prefixes at hi and lo - 1 (buffer 0, pair 0)
    double fr, f, invf, alpha, sc, P0;
};

__device__ __forceinline__ OdeLane ode_lane(cg::cluster_group &cl, OdeWindow &win, const RamanParams &rp, int coff,
                                            int poff, int n)
{
    OdeLane L;
    L.n = n;
    L.wpc = blockDim.x >> 5;
    L.i = (int)cl.block_rank() * blockDim.x + threadIdx.x;
    L.live = L.i < n;
    const int i = min(L.i, n - 1);
    const int lo = rp.win_lo[coff + i], hi = rp.win_hi[coff + i];
    const auto at = [&](int j) {
        const int r = j / (32 * L.wpc);
        return cl.map_shared_rank(&win.x[0][0][0], r) + (j - r * 32 * L.wpc);
    };
    L.one = cl.num_blocks() == 1;
    L.jhi = hi;
    L.jlo = max(lo - 1, 0);
    L.wi = L.i >> 5;
    L.has_lo = lo > 0;
    L.xhi = at(hi);
    L.xlo = at(max(lo - 1, 0));
    L.whi = L.live ? hi >> 5 : L.wi;
    L.wlo = L.live ? max(lo - 1, 0) >> 5 : L.wi;
    L.fr = rp.ch_frel[coff + i];
    L.f = L.fr + rp.f_ref;
    L.invf = 1.0 / L.f;
    L.alpha = rp.ch_alpha[coff + i];
    L.sc = rp.ch_scale[coff + i];
    L.P0 = L.live ? rp.P[poff + i] : 0.0;
    // the first ode_window stores into every block of the cluster: only once all of
    // them run is their shared memory theirs
    if (!L.one) cl.sync();
    return L;
}

// Sums of pair (v0, v1) [or (v2, v3)] over the channels above i in its window
// (up), and below (dn): up from pair pu, dn from pair pd.
__device__ __forceinline__ void ode_window(cg::cluster_group &cl, OdeWindow &win, const OdeLane &L, int buf, double v0,
                                           double v1, double v2, double v3, int pu, int pd, double2 &up, double2 &dn)
{
    const int lane = threadIdx.x & 31;
    double x0 = v0, x1 = v1, x2 = v2, x3 = v3;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u0 = __shfl_up_sync(0xffffffffu, x0, o), u1 = __shfl_up_sync(0xffffffffu, x1, o);
        const double u2 = __shfl_up_sync(0xffffffffu, x2, o), u3 = __shfl_up_sync(0xffffffffu, x3, o);
        if (lane >= o) {
            x0 += u0;
            x1 += u1;
            x2 += u2;
            x3 += u3;
        }
    }
    win.x[buf][0][threadIdx.x] = make_double2(x0, x1);
    win.x[buf][1][threadIdx.x] = make_double2(x2, x3);
    // totals of this warp to every block: lane r (r + 16) takes pair 0 (1) of block r
    const double2 t0 = make_double2(__shfl_sync(0xffffffffu, x0, 31), __shfl_sync(0xffffffffu, x1, 31));
    const double2 t1 = make_double2(__shfl_sync(0xffffffffu, x2, 31), __shfl_sync(0xffffffffu, x3, 31));
    double2 h, l;
    if (L.one) {
        if ((lane & 15) == 0) win.tot[buf][lane >> 4][L.wi] = lane < 16 ? t0 : t1;
        __syncthreads();
        h = win.x[buf][pu][L.jhi];
        l = win.x[buf][pd][L.jlo];
    } else {
        const int r = lane & 15;
        if (r < (int)cl.num_blocks()) {
            double2 *dst = cl.map_shared_rank(&win.tot[buf][lane >> 4][0], r);
            dst[L.wi] = lane < 16 ? t0 : t1;
        }
        cl.sync();
        const int per = 2 * (int)(sizeof(win.x[0][0]) / sizeof(double2));      // entries of one buffer
        const int one = per / 2;
        h = L.xhi[buf * per + pu * one];
        l = L.xlo[buf * per + pd * one];
    }
    const double2 iu = pu ? make_double2(x2, x3) : make_double2(x0, x1);
    const double2 id = pd ? make_double2(x2, x3) : make_double2(x0, x1);
    up = make_double2(h.x - iu.x, h.y - iu.y);
    for (int w = L.wi; w < L.whi; ++w) {
        const double2 t = win.tot[buf][pu][w];
        up.x += t.x;
        up.y += t.y;
    }
    dn = make_double2(id.x - (pd ? v2 : v0), id.y - (pd ? v3 : v1));
    if (L.has_lo) {
        dn.x -= l.x;
        dn.y -= l.y;
    }
    for (int w = L.has_lo ? L.wlo : 0; w < L.wi; ++w) {
        const double2 t = win.tot[buf][pd][w];
        dn.x += t.x;
        dn.y += t.y;
    }
}

// dy/dz of the lane's channel, P its power e^y (0 for an empty slot)
__device__ __forceinline__ double ode_rhs(cg::cluster_group &cl, OdeWindow &win, const OdeLane &L,
                                          const RamanParams &rp, int &buf, double P)
{
    double2 up, dn;
    const double q = P * L.invf;
    ode_window(cl, win, L, buf, P, L.fr * P, q, L.fr * q, 0, rp.photon ? 1 : 0, up, dn);
    buf ^= 1;
    const double below = fma(-L.fr, dn.x, dn.y);
    const double g = fma(-L.fr, up.x, up.y) + (rp.photon ? L.f * below : below);
    return fma(L.sc * rp.Cr, g, -L.alpha);
}

}  // namespace

__global__ void __launch_bounds__(256) k_raman_ode(RamanParams rp)
{
    __shared__ OdeWindow win;
    cg::cluster_group cl = cg::this_cluster();
    const int p = blockIdx.x / cl.num_blocks();
    const int plan = rp.prof_plan[p];
    const int n = rp.plan_n[plan], coff = rp.plan_ch_off[plan], poff = rp.prof_ch_off[p];
    const int M = rp.n_steps;
    const OdeLane L = ode_lane(cl, win, rp, coff, poff, n);
    double2 *ab = rp.ab + (size_t)poff * M;
    double *sp = p == 0 ? rp.stage_P : nullptr;
    const double y0 = L.P0 > 0.0 ? log(L.P0) : 0.0;
    double y = y0;
    int buf = 0;
    size_t node = 0;
    const auto keep = [&](int s, double P) {
        if (sp && L.live) sp[(4 * node + s) * n + L.i] = P;
    };
    for (int m = 0; m < M; ++m) {
        const int ns = rp.half_steps[m];
        const double h = 0.5 * rp.zs_d[m].y / ns;
        for (int half = 0; half < 2; ++half) {
            for (int t = 0; t < ns; ++t) {
                const double P1 = L.P0 > 0.0 ? exp(y) : 0.0;
                const double k1 = ode_rhs(cl, win, L, rp, buf, P1);
                const double P2 = P1 * exp_small(0.5 * h * k1);
                const double k2 = ode_rhs(cl, win, L, rp, buf, P2);
                const double P3 = P1 * exp_small(0.5 * h * k2);
                const double k3 = ode_rhs(cl, win, L, rp, buf, P3);
                const double P4 = P1 * exp_small(h * k3);
                const double k4 = ode_rhs(cl, win, L, rp, buf, P4);
                y += h / 6.0 * ((k1 + 2.0 * k2) + 2.0 * k3 + k4);
                keep(0, P1);
                keep(1, P2);
                keep(2, P3);
                keep(3, P4);
                ++node;
            }
            if (half == 0 && L.live) ab[(size_t)L.i * M + m].x = y - y0;
        }
    }
    if (L.live) rp.lnrho_L[poff + L.i] = y - y0;
    cl.sync();                       // the tables of every block; no block leaves while others read its prefixes
    // in-channel slopes: central differences of a + alpha z_m
    const double *fr = rp.ch_frel + coff;
    const double *al = rp.ch_alpha + coff;
    for (int t = (int)cl.thread_rank(); t < n * M; t += (int)cl.num_threads()) {
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

namespace {

// One cluster per profile: warps of 32 channels, kOdeWarps to a block where 16
// blocks (8 if the device cannot place 16) hold them, else more.
template <typename Params>
cudaError_t launch_clusters(void (*fn)(Params), const Params &prm, int n_prof, int max_n, cudaStream_t st)
{
    const int warps = (max_n + 31) / 32;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    for (int most = kOdeMaxCluster; most >= 8; most /= 2) {
        const int wpc = std::max(kOdeWarps, (warps + most - 1) / most);
        const int size = (warps + wpc - 1) / wpc;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[1];
        cfg.gridDim = dim3(n_prof * size);
        cfg.blockDim = dim3(32 * wpc);
        cfg.stream = st;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = size;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        if (size > 8) {
            int nc = 0;
            if (cudaOccupancyMaxActiveClusters(&nc, fn, &cfg) != cudaSuccess || nc < 1) {
                cudaGetLastError();
                continue;
            }
        }
        return cudaLaunchKernelEx(&cfg, fn, prm);
    }
    return cudaErrorInvalidConfiguration;
}

}  // namespace

cudaError_t launch_raman(const RamanParams &rp, int n_prof, int max_n, cudaStream_t st)
{
    return launch_clusters(k_raman_ode, rp, n_prof, max_n, st);
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
// with the stage powers e^Y kept by the forward run, the table sensitivities
// injected at the nodes z_m and L, and
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

// (J^T v) of the lane's channel at the stage power P = e^{Y_k}
__device__ __forceinline__ double ode_jt(cg::cluster_group &cl, OdeWindow &win, const OdeLane &L,
                                         const RamanParams &rp, int &buf, double P, double v)
{
    double2 up, dn;
    const double u = L.live ? L.sc * v : 0.0, w = L.f * u;
    ode_window(cl, win, L, buf, u, L.fr * u, w, L.fr * w, rp.photon ? 1 : 0, 0, up, dn);
    buf ^= 1;
    const double above = fma(L.fr, up.x, -up.y);
    const double g = fma(L.fr, dn.x, -dn.y) + (rp.photon ? above * L.invf : above);
    return rp.Cr * P * g;
}

}  // namespace

__global__ void __launch_bounds__(256) k_raman_adj(RamanAdjParams ap)
{
    __shared__ OdeWindow win;
    cg::cluster_group cl = cg::this_cluster();
    const RamanParams &rp = ap.r;
    const int n = ap.n, M = rp.n_steps;
    const OdeLane L = ode_lane(cl, win, rp, 0, 0, n);
    const int c = min(L.i, n - 1);
    double lam = L.live && ap.with_direct ? -ap.aase[c] : 0.0;             // dT/d ln rho(L)
    int buf = 0;
    size_t node = (size_t)ap.n_rk;
    const auto stage = [&](size_t k, int s) { return rp.stage_P[(4 * k + s) * n + c]; };
    // the stage powers of the next step back are fetched while this one runs
    double q1 = stage(node - 1, 0), q2 = stage(node - 1, 1), q3 = stage(node - 1, 2), q4 = stage(node - 1, 3);
    for (int m = M - 1; m >= 0; --m) {
        const int ns = rp.half_steps[m];
        const double h = 0.5 * rp.zs_d[m].y / ns;
        const double inj = L.live ? ap.gAt[(size_t)c * M + m] : 0.0;
        for (int half = 1; half >= 0; --half) {
            for (int t = 0; t < ns; ++t) {
                --node;
                const double P1 = q1, P2 = q2, P3 = q3, P4 = q4;
                const size_t nx = node > 0 ? node - 1 : 0;
                q1 = stage(nx, 0);
                q2 = stage(nx, 1);
                q3 = stage(nx, 2);
                q4 = stage(nx, 3);
                const double h6 = h / 6.0 * lam, h3 = h / 3.0 * lam;
                const double m4 = ode_jt(cl, win, L, rp, buf, P4, h6);
                const double m3 = ode_jt(cl, win, L, rp, buf, P3, fma(h, m4, h3));
                const double m2 = ode_jt(cl, win, L, rp, buf, P2, fma(0.5 * h, m3, h3));
                const double m1 = ode_jt(cl, win, L, rp, buf, P1, fma(0.5 * h, m2, h6));
                lam += ((m4 + m3) + m2) + m1;
            }
            if (half == 1) lam += inj;
        }
    }
    cl.sync();                       // no block leaves while others read its prefixes
    if (!L.live) return;
    // a = y - y(0): every table entry also depends on y(0) directly
    double direct = ap.with_direct ? ap.aase[c] : 0.0;             // - dT/d ln rho(L)
    for (int m = 0; m < M; ++m) direct -= ap.gAt[(size_t)c * M + m];
    const double P = rp.P[c];
    double g = (lam + direct + ap.gV[c]) / P;
    if (ap.with_direct) {                                          // the SNR numerator
        const double snr = ap.snr[c], B = ap.ch_B[c];
        const double N = ap.pnli[c] + ap.pase[c];
        const double dTds = 2.0 * B / (0.69314718055994530942 * (1.0 + snr));
        g += dTds * snr * snr * N / (P * P);
    }
    ap.dT_dP[c] = g;
}

cudaError_t launch_raman_adj(const RamanAdjParams &ap, cudaStream_t st)
{
    const int nm = ap.n * ap.r.n_steps;
    k_fold_slope<<<(nm + 255) / 256, 256, 0, st>>>(ap);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_clusters(k_raman_adj, ap, 1, ap.n, st);
}

// ---------------------------------------------------------------------------
// Quadratures with the tabulated profile.
// ---------------------------------------------------------------------------
constexpr int kTabSlots = 512;       // node slots of a chunk
constexpr int kTabCand = 2;          // F_c candidates swept together (most pieces have two)
using TabNodes = WarpNodes<kTabSlots>;

// Dynamic shared memory of k_quad_f32_tab: eB and zD (pair_tables), then per warp
// the nodes and the candidates' step rows.
__host__ __device__ constexpr size_t tab_warp_bytes(int n_steps)
{
    return sizeof(TabNodes) + ((size_t)24 * kTabCand * step_pairs(n_steps) + 15) / 16 * 16;
}

// As k_quad_f32 (quad_fwd.cu: one warp per tile, row sums from nodes), with the
// step rows of the tabulated profile.  148 channels at G = 256: 112.3 -> 2.57 ms, XU
// pipe 71 % busy.
#ifndef ISRS_TAB_MIN_BLOCKS
#define ISRS_TAB_MIN_BLOCKS 3   // resident blocks per SM the register budget is sized for
#endif

__global__ void __launch_bounds__(256, ISRS_TAB_MIN_BLOCKS) k_quad_f32_tab(QuadParams qp)
{
    extern __shared__ float4 smem_f4[];
    const int M = qp.n_steps, G = qp.G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int M2 = step_pairs(M);
    float4 *eB = smem_f4, *zD = eB + M2;
    unsigned char *mine = reinterpret_cast<unsigned char *>(zD + M2) + tab_warp_bytes(M) * warp;
    TabNodes &ns = *reinterpret_cast<TabNodes *>(mine);
    float4 *Qa = reinterpret_cast<float4 *>(mine + sizeof(TabNodes));  // [kTabCand][M2] {A, A', Sl, Sl'}
    float2 *Qb = reinterpret_cast<float2 *>(Qa + kTabCand * M2);       // [kTabCand][M2] {Sd, Sd'}

    pair_tables(qp, eB, zD);
    __syncthreads();
    const float phi_direct = 3.14159265f / qp.dz_max;
    const float phi_small = kSmallPhiL / (qp.L * (float)qp.n_spans);
    PathCount count;

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
            const PieceBlocks pb = row_blocks(ns, qp.gauss, G);
            if (lane == 0 && part == 0) count.small += pb.R1 * G;
            for (int ca = 0; ca < g.nc; ca += kTabCand) {
                const int cb = min(g.nc, ca + kTabCand);
                float tilt = 0.0f;
                for (int c = ca; c < cb; ++c) {
                    const double fc = qp.ch_frel[coff + pc.c_lo + c];
                    for (int k = lane; k < M2; k += 32) {
                        const float4 r = tab_row(tp, pc.c_lo + c, fc, 2 * k, M);
                        float4 u = make_float4(-1000.0f, 0.0f, 0.0f, 0.0f);
                        if (2 * k + 1 < M) u = tab_row(tp, pc.c_lo + c, fc, 2 * k + 1, M);
                        Qa[(c - ca) * M2 + k] = make_float4(r.x, u.x, r.y, u.y);
                        Qb[(c - ca) * M2 + k] = make_float2(r.z, u.z);
                        tilt = fmaxf(tilt, fmaxf(fmaxf(fabsf(r.y), fabsf(r.z)), fmaxf(fabsf(u.y), fabsf(u.z))));
                    }
                }
                // the largest slope of ln p bounds its swing along a row
                tilt = 0.69314718f * __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(tilt)));
                if (lane == 0) g.tilt = tilt;
                __syncwarp();
                piece_nodes(ns, pb, qp.gauss, G, ca, cb, [&](int c0, int nq) {
                    for (int q = lane + 32 * part; q < nq; q += 32 * parts) {
                        Node nd;
                        node_get(ns, qp.gauss, c0, q, nd);
                        const int ci = dbg_clamp(nd.ci, g.nc, kDbgCand, qp.dbg);
                        const float aphi = fabsf(nd.phi);
                        const f32x2 dl = dup2(tp.ol + nd.x), dd = dup2(tp.od + nd.y);
                        const float4 *qa = Qa + (ci - ca) * M2;
                        const float2 *qb = Qb + (ci - ca) * M2;
                        const auto lp = [&](int k) {
                            const float4 x = qa[k];
                            const float2 y = qb[k];
                            return fma2(pack2(y.x, y.y), dd, fma2(pack2(x.z, x.w), dl, pack2(x.x, x.y)));
                        };
                        const bool direct = aphi <= phi_direct;
                        const float S2 = direct ? zsum_direct_n(nd.phi, lp, zD, M2)
                                                : zsum_tele_n<0>(nd.phi, nd.phi_lo, lp, eB, M2);
                        count.points(aphi, phi_small, !direct, nd.N);
                        count.sums(!direct, 1);
                        const float y = nd.wq * g.pd[ci] * S2 * array_factor_f(nd.phi, qp, nd.phi_lo) - comp;
                        const float t = sum + y;
                        comp = (t - sum) - y;
                        sum = t;
                    }
                });
            }
            acc += (double)(g.mult * g.wab) * ((double)sum - (double)comp);
        }
        const double tot = warp_sum_d(acc);
        if (lane == 0) qp.partial[it] = tot;
    }
    if (qp.path_count) count.store(qp.path_count);
}

// Plain FP64 quadrature with the tabulated profile (direct form, libm).
__global__ void __launch_bounds__(256) k_quad_f64_tab(QuadParams qp)
{
    extern __shared__ double2 smem_d2[];
    const int M = qp.n_steps, G = qp.G;
    double2 *sz = smem_d2;                              // [M] {z_m, dz_m}
    double2 *sQ = sz + M;                               // [nc_max][M][2] {A, Sa}, {Sb, e^A}
    RowD *rows = reinterpret_cast<RowD *>(sQ + (size_t)2 * qp.nc_max * M);
    __shared__ PieceConst<double> kc;
    __shared__ double s_d0[2];
    __shared__ double scratch[32];
    __shared__ int s_item;

    for (int m = threadIdx.x; m < M; m += blockDim.x) sz[m] = qp.zs_d[m];
    const double phi_direct = kF64Direct / qp.dz_max;
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
                    const double A = 0.5 * (ta.x + tb.x + tc.x - ti.x + tc.y * D);
                    sQ[2 * t] = make_double2(A, 0.5 * (ta.y + tc.y));
                    sQ[2 * t + 1] = make_double2(0.5 * (tb.y + tc.y), exp(A));
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
                const double S2 = zsum_f64(phi, phi_direct, sz, M, [&](int m) {
                    const double2 q0 = Q[2 * m], q1 = Q[2 * m + 1];
                    return q1.y * exp_small(q0.y * da + q1.x * db);
                });
                sum += rw.w * W * S2 * array_factor_d(phi, qp);
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
        const auto bytes = [&](int b) { return sizeof(float4) * 2 * step_pairs(qp.n_steps) + tab_warp_bytes(qp.n_steps) * (b / 32); };
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
