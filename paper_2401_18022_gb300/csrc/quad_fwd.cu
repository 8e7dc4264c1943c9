// Forward kernels of the ISRS GN integral model (arXiv 2401.18022, App. A).
//
//  k_prep        per profile and z-step (FP64): P_tot, the ISRS
//                normalisation ln N(z_m) by log-sum-exp over channels, and the
//                per-step power tables of Eq. pk for the linear-slope
//                closed-form profile.
//  k_gauss       the Gauss rules of the discrete uniform measures (quad_nodes.cuh).
//  k_quad_f32    persistent quadrature: one warp per work tile (a range of
//                pieces of one CUT); G x G hyperbolic grid per piece
//                (Eqs. q1..q4), each row's sum taken from a few nodes
//                (quad_nodes.cuh), the z-sum of Eq. slow_vary per node in FP32
//                (quad_zsum.cuh) with a float-float phase; compensated
//                accumulation; one FP64 partial per tile.
//  k_quad_f64    the same quadrature in plain FP64 at every grid point, used as
//                the reference GPU path.
//  k_finish      per profile: deterministic FP64 sum of tile partials per CUT,
//                eta (Eq. gain_fin), P_NLI, SNR and throughput (Eq. loss).
#include <cuda_runtime.h>

#include <algorithm>

#include "isrs_internal.cuh"
#include "isrs_kernels.h"
#include "quad_common.cuh"
#include "quad_nodes.cuh"
#include "quad_zsum.cuh"

namespace isrs {

// ---------------------------------------------------------------------------
// k_prep: ISRS profile tables (FP64).  One block per (profile, z-step), the
// last step index standing for z = L:
//   rho(z,F) = e^{-alpha_c z} P_tot e^{-kappa(z)(F - f_ref)} / N(z)
//   kappa(z) = P_tot C_r L_eff(z),  N(z) = sum_k P_k e^{-kappa f_k'} sinhc(kappa B_k/2)
// so ln p_m (Eq. pk) = lnPtot - lnN_m - kappa_m (F_c - f_ref) - at z_m with
// at = (alpha_a + alpha_b + alpha_c - alpha_i)/2, because F_a + F_b + F_c - f
// = 2 F_c.  Writes, per step, {A2, K2} = log2(e) {lnPtot - lnN, -kappa} and
// {lnPtot - lnN, kappa}; per channel P/B (step 0's block) and ln rho(L, f_c)
// (the z = L block); where a gradient follows, the chain rule's step terms too
// (ln N, kappa, L_eff and the tilted mean frequency Fbar - f_ref).  ln N is a
// log-sum-exp over the channels with a block maximum and a block sum in fixed
// order.  A launch is one wave of short blocks, so it is bound by the latency of
// its FP64 chain: one exp per channel, log_sinhc by its series (two logs, two
// sinhs and a log more took 20 us at 5 channels).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_prep(PrepParams pp)
{
    __shared__ double scratch[32];
    const int p = blockIdx.x, m = blockIdx.y;
    const int plan = pp.prof_plan[p];
    const int n = pp.plan_n[plan];
    const int coff = pp.plan_ch_off[plan];
    const int poff = pp.prof_ch_off[p];
    const double *P = pp.P + poff;
    const double *fr = pp.ch_frel + coff;
    const double *B = pp.ch_B + coff;
    const int M = pp.n_steps;

    double part = 0.0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) part += P[c];
    const double Ptot = block_sum_d(part, scratch);
    const double lnPtot = log(Ptot);
    if (m == 0) {
        for (int c = threadIdx.x; c < n; c += blockDim.x) {
            double pd = P[c] / B[c];
            pp.pd_d[poff + c] = pd;
            pp.pd_f[poff + c] = (float)pd;
        }
    }
    const double z = (m < M) ? pp.zs_d[m].x : pp.L;
    const double leff = pp.alpha_R > 0.0 ? -expm1(-pp.alpha_R * z) / pp.alpha_R : z;
    const double kap = Ptot * pp.Cr * leff;
    const auto expo = [&](int c) { return log_sinhc(0.5 * kap * B[c]) - kap * fr[c]; };
    double mx = -1e300;
    for (int c = threadIdx.x; c < n; c += blockDim.x)
        if (P[c] > 0.0) mx = fmax(mx, expo(c));
    mx = block_max_d(mx, scratch);
    double s0 = 0.0, s1 = 0.0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        if (!(P[c] > 0.0)) continue;
        const double w = P[c] * exp(expo(c) - mx), hb = 0.5 * B[c];
        s0 += w;
        if (pp.cs) s1 += w * (fr[c] - hb * dlog_sinhc(kap * hb));
    }
    s0 = block_sum_d(s0, scratch);
    const double lnN = mx + log(s0);
    if (pp.cs) {
        s1 = block_sum_d(s1, scratch);
        if (threadIdx.x == 0) {
            const int st = M + 1;
            pp.cs[m] = lnN;
            pp.cs[st + m] = kap;
            pp.cs[2 * st + m] = leff;
            pp.cs[3 * st + m] = s1 / s0;
        }
    }
    if (m < M) {
        if (threadIdx.x == 0) {
            pp.step_d[(size_t)p * M + m] = make_double2(lnPtot - lnN, kap);
            pp.step_f[(size_t)p * M + m] = make_float2((float)((lnPtot - lnN) * kLog2e), (float)(-kap * kLog2e));
        }
        return;
    }
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        pp.lnrho_L[poff + c] = -pp.ch_alpha[coff + c] * pp.L + lnPtot - lnN - kap * fr[c];
    }
    if (threadIdx.x == 0) {
        pp.ptot[p] = Ptot;
        if (pp.kap_L) pp.kap_L[p] = kap;
    }
}

// ---------------------------------------------------------------------------
// k_gauss: nodes and weights of the n-node Gauss rules of the uniform measure
// on t_j = (2 j + 1 - N)/N, j < N, for every N <= kGaussMaxN.  The monic
// orthogonal polynomials (discrete Chebyshev, Gautschi 2004) satisfy
// p_{i+1} = t p_i - b_i p_{i-1} with b_i = i^2 (N^2 - i^2) / (N^2 (4 i^2 - 1)).
// One thread per node: the k-th smallest zero by bisection on the sign changes
// of the sequence p_0..p_n (Sturm), then Newton; weight N / sum of the squared
// orthonormal polynomials.  FP64, run once per device (4 ms).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_gauss(float2 *out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= kGaussEntries) {
        const int j = e - kGaussEntries;
        if (j >= kExp2Entries) return;
        const double v = exp2(-(double)j / kExp2Entries);
        out[e] = make_float2((float)v, (float)(v - (double)(float)v));
        return;
    }
    const int N = e / kGaussPerN + 1, o = e - (N - 1) * kGaussPerN;
    int m = 0;
    while (m + 1 < kGaussMenu && gauss_offset(m + 1) <= o) ++m;
    const int n = gauss_nodes(m), k = o - gauss_offset(m);
    if (n >= N) {                      // never used: a run takes its columns then
        out[e] = make_float2(0.0f, 0.0f);
        return;
    }
    const double N2 = (double)N * N;
    const auto b = [&](int i) { return (double)i * i * (N2 - (double)i * i) / (N2 * (4.0 * i * i - 1.0)); };
    // zeros below t, from the signs of the Sturm quotients p_{i+1}/p_i
    const auto below = [&](double t) {
        int cnt = 0;
        double q = -t;
        for (int i = 0;; ++i) {
            if (q < 0.0) ++cnt;
            if (i + 1 == n) break;
            if (q == 0.0) q = 1e-300;
            q = -t - b(i + 1) / q;
        }
        return cnt;
    };
    double lo = -1.0, hi = 1.0;
    for (int s = 0; s < 26; ++s) {
        const double mid = 0.5 * (lo + hi);
        if (below(mid) > k) hi = mid;
        else lo = mid;
    }
    double t = 0.5 * (lo + hi), sum = 0.0;
    for (int s = 0; s < 3; ++s) {
        double p0 = 1.0, p1 = t, d0 = 0.0, d1 = 1.0, h = 1.0;
        sum = 1.0;
        for (int i = 1; i < n; ++i) {
            const double bi = b(i);
            h *= bi;
            sum += p1 * p1 / h;
            const double p2 = t * p1 - bi * p0, d2 = p1 + t * d1 - bi * d0;
            p0 = p1;
            p1 = p2;
            d0 = d1;
            d1 = d2;
        }
        if (s < 2) t -= p1 / d1;
    }
    out[e] = make_float2((float)t, (float)(N / sum));
}

cudaError_t launch_gauss(float2 *out, cudaStream_t st)
{
    k_gauss<<<(kGaussEntries + kExp2Entries + 127) / 128, 128, 0, st>>>(out);
    return cudaGetLastError();
}

__device__ float2 g_isrs_gauss[kGaussEntries + kExp2Entries];

// ln(xhi / xlo), ln(yhi / ylo) and the row pitch of every piece, once per plan (the
// quadrature would otherwise take two FP64 logarithms and a division per piece and
// launch).
__global__ void __launch_bounds__(256) k_piece_logs(DevPiece *pieces, int n, int G, double ln_eps)
{
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        DevPiece &p = pieces[k];
        const double lx = p.xlo > 0.0 ? log(p.xhi / p.xlo) : 1e30, ly = p.ylo > 0.0 ? log(p.yhi / p.ylo) : 1e30;
        // upsilon1 runs from max(xlo ylo, eps xhi yhi) to xhi yhi
        const double ds2 = fmin(lx + ly, ln_eps) / G * kLog2e;
        p.lnx = (float)lx;
        p.lny = (float)ly;
        p.ds2 = make_float2((float)ds2, (float)(ds2 - (double)(float)ds2));
    }
}

cudaError_t launch_piece_logs(DevPiece *pieces, int n, int G, double ln_eps, cudaStream_t st)
{
    if (n > 0) k_piece_logs<<<std::min(2048, (n + 255) / 256), 256, 0, st>>>(pieces, n, G, ln_eps);
    return cudaGetLastError();
}

cudaError_t gauss_array(void **out) { return cudaGetSymbolAddress(out, g_isrs_gauss); }

// ---------------------------------------------------------------------------
// k_quad_f32: persistent FP32 quadrature.  Bound by the XU pipe (sin and cos at 16
// lanes a clock, ex2 at 32: 20 cycles per warp and z-step), 70 % busy on a 148-channel
// plan at G = 256 (2.41 ms; every grid point summed one by one: 74.4 ms).  589
// channels at G = 256: 1,129 -> 45.6 ms; 12 profiles at G = 64: 541 -> 81.8 ms, a
// quarter of it the pieces' set-up.  Three blocks of 80 registers an SM: two leave
// 5 % on the G = 256 case and 6 % on the G = 64 one, four spill (4 % and 9 %).
// ---------------------------------------------------------------------------
constexpr int kFwdSlots = 512;       // node slots of a chunk
using FwdNodes = WarpNodes<kFwdSlots>;

// The nodes a warp has yet to sum, by form of the z-sum (direct, telescoped).  A
// queue is drained 32 at a time, and what a tile leaves at its end shares the
// lanes, several to a node: a piece's ~250 nodes at G = 64 taken as they come
// filled 23 of 32 lanes, by the rows' tails and by rounds that held both forms and
// so took both.
struct FwdQueue {
    float4 a[2][64];            // {phi, phi_lo, F_c - f_i, attenuation part of log2 p}
    float w[2][64];             // weight
};

// Dynamic shared memory of k_quad_f32: eB and zD (pair_tables), then per warp the
// nodes, the queues and the step rows {A2, A2', K2, K2'} about the CUT's frequency.
__host__ __device__ constexpr size_t fwd_warp_bytes(int n_steps)
{
    return sizeof(FwdNodes) + sizeof(FwdQueue) + sizeof(float4) * (size_t)step_pairs(n_steps);
}
#ifndef ISRS_FWD_MIN_BLOCKS
#define ISRS_FWD_MIN_BLOCKS 3   // resident blocks per SM the register budget is sized for
#endif

__global__ void __launch_bounds__(256, ISRS_FWD_MIN_BLOCKS) k_quad_f32(QuadParams qp)
{
    extern __shared__ float4 smem_f4[];
    const int M = qp.n_steps, G = qp.G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int M2 = step_pairs(M);
    float4 *eB = smem_f4, *zD = eB + M2;
    unsigned char *mine = reinterpret_cast<unsigned char *>(zD + M2) + fwd_warp_bytes(M) * warp;
    FwdNodes &ns = *reinterpret_cast<FwdNodes *>(mine);
    FwdQueue &qu = *reinterpret_cast<FwdQueue *>(mine + sizeof(FwdNodes));
    float4 *sp = reinterpret_cast<float4 *>(mine + sizeof(FwdNodes) + sizeof(FwdQueue));

    pair_tables(qp, eB, zD);
    __syncthreads();
    const float phi_direct = 3.14159265f / qp.dz_max;
    const float phi_small = kSmallPhiL / (qp.L * (float)qp.n_spans);
    const float log2e = (float)kLog2e;
    PathCount count;
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(qp.counter, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= qp.n_items) break;
        const DevItem item = qp.items[it];
        const float tilt = (float)qp.kap_L[item.prof];
        const int part = item.part & 0xffff, parts = item.part >> 16;
        // log2 p at F_c = f_i: taken about f_ref, a plan tens of THz away from it would
        // lose the last digits to the difference of two large terms
        {
            const double fi = qp.ch_frel[qp.plan_ch_off[qp.prof_plan[item.prof]] + item.cut];
            const double2 *sd = qp.step_d + (size_t)item.prof * M;
            const float2 *st = qp.step_f + (size_t)item.prof * M;
            for (int k = lane; k < M2; k += 32) {
                const int k1 = min(2 * k + 1, M - 1);
                const double2 v = sd[2 * k], u = sd[k1];
                sp[k] = make_float4((float)(kLog2e * fma(-v.y, fi, v.x)),
                                    2 * k + 1 < M ? (float)(kLog2e * fma(-u.y, fi, u.x)) : -1000.0f,
                                    st[2 * k].y, st[k1].y);
            }
        }
        float sum = 0.0f, comp = 0.0f;
        int nd_q = 0, nt_q = 0;              // nodes in the queues
        // entries [first, first + n) of a queue, 32 / n lanes (a power of two) to a node
        const auto drain = [&](int form, int first, int n) {
            const int lg = n > 16 ? 0 : n > 8 ? 1 : n > 4 ? 2 : n > 2 ? 3 : n > 1 ? 4 : 5;
            const int node = lane >> lg, sub = lane - (node << lg);
            const int k0 = (M2 * sub) >> lg, k1 = (M2 * (sub + 1)) >> lg;
            const float4 a = qu.a[form][first + min(node, n - 1)];
            const float w = node < n && sub == 0 ? qu.w[form][first + node] : 0.0f;
            const f32x2 F2 = dup2(a.z), nat = dup2(-a.w);
            const auto lp = [&](int k) {
                const float4 x = sp[k], z = zD[k];
                return fma2(pack2(x.z, x.w), F2, fma2(nat, pack2(z.x, z.y), pack2(x.x, x.y)));
            };
            float2 S = form == 0 ? zsum_direct_part(a.x, lp, zD, k0, k1)
                                 : zsum_tele_part<0>(a.x, a.y, lp, eB, k0, k1);
            for (int o = (1 << lg) >> 1; o > 0; o >>= 1) {
                S.x += __shfl_xor_sync(0xffffffffu, S.x, o);
                S.y += __shfl_xor_sync(0xffffffffu, S.y, o);
            }
            if (lane == 0) count.sums(form, n);
            const float S2 = S.x * S.x + S.y * S.y;
            // compensated accumulation over this lane's nodes
            const float y = w * (form == 0 ? S2 : __fdividef(S2, a.x * a.x)) * array_factor_f(a.x, qp, a.y) - comp;
            const float t = sum + y;
            comp = (t - sum) - y;
            sum = t;
            __syncwarp();
        };
#pragma unroll 1
        for (int k = item.piece0; k < item.piece1; ++k) {
            const DevPiece &pc = qp.pieces[dbg_clamp(k, qp.n_pieces, kDbgPiece, qp.dbg)];
            __syncwarp();
            node_geo(qp, pc, item.prof, log2e, qp.pd_f, tilt, ns.geo);
            __syncwarp();
            const PieceGeo &g = ns.geo;
            const PieceBlocks pb = row_blocks(ns, qp.gauss, G);
            if (lane == 0 && part == 0) count.small += pb.R1 * G;
            const float wp = g.mult * g.wab;
            piece_nodes(ns, pb, qp.gauss, G, 0, g.nc, [&](int c0, int nq) {
#pragma unroll 1
                for (int q0 = 32 * part; q0 < nq; q0 += 32 * parts) {
                    const bool on = q0 + lane < nq;
                    Node nd;
                    node_get(ns, qp.gauss, c0, on ? q0 + lane : nq - 1, nd);
                    const int ci = dbg_clamp(nd.ci, g.nc, kDbgCand, qp.dbg);
                    const float aphi = fabsf(nd.phi);
                    const int form = aphi <= phi_direct ? 0 : 1;
                    const unsigned tele = __ballot_sync(0xffffffffu, on && form == 1);
                    const unsigned direct = __ballot_sync(0xffffffffu, on && form == 0);
                    const unsigned below = (1u << lane) - 1u;
                    if (on) {
                        const int d = (form ? nt_q : nd_q) + __popc((form ? tele : direct) & below);
                        qu.a[form][d] = make_float4(nd.phi, nd.phi_lo, g.Fi + (nd.x + nd.y), g.at_ab + g.hat[ci]);
                        qu.w[form][d] = wp * (nd.wq * g.pd[ci]) * zsum_gain(form);
                        count.points(aphi, phi_small, form, nd.N);
                    }
                    nd_q += __popc(direct);
                    nt_q += __popc(tele);
                    __syncwarp();
                    if (nd_q >= 32) drain(0, nd_q -= 32, 32);
                    if (nt_q >= 32) drain(1, nt_q -= 32, 32);
                }
            });
        }
        if (nd_q > 0) drain(0, 0, nd_q);
        if (nt_q > 0) drain(1, 0, nt_q);
        const double tot = warp_sum_d((double)sum - (double)comp);
        if (lane == 0) qp.partial[it] = tot;
    }
    if (qp.path_count) count.store(qp.path_count);
}

// ---------------------------------------------------------------------------
// k_quad_f64: the same quadrature in plain FP64, every grid point.
// ---------------------------------------------------------------------------
// F_c candidates with their powers at the channel centre in shared memory (0
// where a huge grid and z-grid leave no room)
__host__ __device__ constexpr int f64_cand(int n_steps, int G)
{
    return 64 * (size_t)n_steps + sizeof(RowD) * (size_t)G <= 200 * 1024 ? 4 : 0;
}

__global__ void __launch_bounds__(256) k_quad_f64(QuadParams qp)
{
    extern __shared__ double2 smem_d2[];
    const int M = qp.n_steps, G = qp.G;
    double2 *sz = smem_d2;                 // [M] {z_m, dz_m}
    double2 *st = sz + M;                  // [M] {lnPtot - lnN, kappa}
    RowD *rows = reinterpret_cast<RowD *>(st + M);
    double *sP = reinterpret_cast<double *>(rows + G);   // [f64_cand][M] p_m at the candidate's centre
    const int ncp = f64_cand(M, G);
    const double phi_direct = kF64Direct / qp.dz_max;
    __shared__ PieceConst<double> kc;
    __shared__ double scratch[32];
    __shared__ int s_item;

    for (int m = threadIdx.x; m < M; m += blockDim.x) sz[m] = qp.zs_d[m];
    const double c3 = kPi * qp.beta3;
    const double c4 = 2.0 * kPi * kPi / 3.0 * qp.beta4;
    int cur_prof = -1;

    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(qp.counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= qp.n_items) break;
        const DevItem item = qp.items[it];
        if (item.prof != cur_prof) {
            for (int m = threadIdx.x; m < M; m += blockDim.x) st[m] = qp.step_d[(size_t)item.prof * M + m];
            cur_prof = item.prof;
        }
        double acc = 0.0;
        for (int k = item.piece0; k < item.piece1; ++k) {
            const DevPiece pc = qp.pieces[dbg_clamp(k, qp.n_pieces, kDbgPiece, qp.dbg)];
            piece_rows<RowD>(pc, G, qp.eps_v1, rows);
            piece_consts<double>(qp, pc, item.prof, 1.0, qp.pd_d, kc);
            __syncthreads();
            const double fi = kc.fi;
            // powers at the channel centres of the first candidates
            for (int t = threadIdx.x; t < min(kc.nc, ncp) * M; t += blockDim.x) {
                const int c = t / M, m = t - c * M;
                sP[t] = exp(st[m].x - st[m].y * (fi + 0.5 * (kc.lo[c] + kc.hi[c])) - (kc.at_ab + kc.hat[c]) * sz[m].x);
            }
            __syncthreads();
            double sum = 0.0;
            const int npts = G * G;
            for (int q = threadIdx.x + (item.part & 0xffff) * blockDim.x; q < npts;
                 q += (item.part >> 16) * blockDim.x) {
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
                const double at = kc.at_ab + kc.hat[ci];
                const double Fc = fi + u;
                const double br = qp.beta2 + c3 * (u + 2.0 * fi) +
                                  c4 * (f1 * f1 + 1.5 * f1 * f2 + 3.0 * fi * u + f2 * f2 + 3.0 * fi * fi);
                const double phi = -4.0 * kPi * kPi * f1 * f2 * br;
                const double du = u - 0.5 * (kc.lo[ci] + kc.hi[ci]);
                const double *P = sP + (size_t)ci * M;
                const double S2 = zsum_f64(phi, phi_direct, sz, M, [&](int m) {
                    const double2 tt = st[m];
                    return ci < ncp ? P[m] * exp_small(-tt.y * du) : exp(tt.x - tt.y * Fc - at * sz[m].x);
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

// ---------------------------------------------------------------------------
// k_finish: per profile, Sigma_i = ordered sum of the CUT's tile partials;
// eta_i = (16/27) gamma_i^2 B_i Sigma_i / P_i^3 (Eq. gain_fin, P_NLI = G B);
// SNR_i = P_i / (P_NLI,i + P_ASE,i) with P_ASE,i = NF h f (1/rho(L,f) - 1) B
// and optional transceiver noise; T = 2 sum B log2(1 + SNR) (Eq. loss).  Eight
// lanes sum a CUT's tiles, then a thread per CUT takes the FP64 rest (one thread for
// both took 15 us at 5 channels).
// ---------------------------------------------------------------------------
constexpr int kFinishLanes = 8;

__global__ void __launch_bounds__(512) k_finish(FinishParams fp)
{
    __shared__ double scratch[32];
    const int p = blockIdx.x;
    const int plan = fp.prof_plan[p];
    const int coff = fp.plan_ch_off[plan];
    const int poff = fp.prof_ch_off[p];
    const int s0 = fp.prof_slot_off[p], s1 = fp.prof_slot_off[p + 1];
    double tpart = 0.0;
    const int sub = threadIdx.x % kFinishLanes, per = blockDim.x / kFinishLanes;
    __shared__ double sums[512];
    for (int cb = s0; cb < s1; cb += blockDim.x) {
        const int ce = min(cb + (int)blockDim.x, s1);
        for (int sb = cb; sb < ce; sb += per) {
            const int s = sb + threadIdx.x / kFinishLanes;
            double sig = 0.0;
            if (s < ce) {
                const int2 rg = fp.slot_items[s];
                for (int it = rg.x + sub; it < rg.y; it += kFinishLanes) sig += fp.partial[it];
                if (fp.slot_items2) {
                    const int2 r2 = fp.slot_items2[s];
                    for (int it = r2.x + sub; it < r2.y; it += kFinishLanes) sig += fp.partial2[it];
                }
            }
#pragma unroll
            for (int o = kFinishLanes / 2; o > 0; o >>= 1) sig += __shfl_xor_sync(0xffffffffu, sig, o);
            if (s < ce && sub == 0) sums[s - cb] = sig;
        }
        __syncthreads();
        const int s = cb + threadIdx.x;
        const double sig = s < ce ? sums[threadIdx.x] : 0.0;
        __syncthreads();
        if (s >= ce) continue;
        const int i = fp.slot_cut[s];
        const double g = fp.ch_gamma[coff + i];
        const double B = fp.ch_B[coff + i];
        const double P = fp.P[poff + i];
        const double pnli = 16.0 / 27.0 * g * g * B * sig;
        const double eta = P > 0.0 ? pnli / (P * P * P) : __longlong_as_double(0x7ff8000000000000LL);
        if (fp.sigma) fp.sigma[s] = sig;
        if (fp.pnli) fp.pnli[s] = pnli;
        if (fp.eta) fp.eta[s] = eta;
        if (fp.snr) {
            const double nf = fp.ch_nf ? fp.ch_nf[coff + i] : 1.0;
            const double f_abs = fp.ch_frel[coff + i] + fp.f_ref;
            const double gain = exp(-fp.lnrho_L[poff + i]);
            const double pase = fp.n_spans * nf * 6.62607015e-34 * (f_abs * 1e12) * (gain - 1.0) * (B * 1e12);
            const bool off = !(P > 0.0) || (fp.guard && fp.guard[coff + i]);
            double snr = 0.0;
            if (!off) {
                snr = P / (pnli + pase);
                if (fp.snr_trx_lin_inv > 0.0) snr = 1.0 / (1.0 / snr + fp.snr_trx_lin_inv);
                tpart += 2.0 * B * log2(1.0 + snr);
            }
            fp.snr[s] = snr;
            if (fp.pase) fp.pase[s] = pase;
        }
    }
    const double T = block_sum_d(tpart, scratch);
    if (threadIdx.x == 0 && fp.T) fp.T[p] = T;
}

// ---------------------------------------------------------------------------
// k_snr_from_eta: the Eq. loss part of k_finish for every channel, from a
// given eta (gathered from the shards of a split gradient): P_NLI = eta P^3,
// P_ASE, SNR and T.  One block.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_snr_from_eta(SnrFromEtaParams sp)
{
    __shared__ double scratch[32];
    double tpart = 0.0;
    for (int i = threadIdx.x; i < sp.n; i += blockDim.x) {
        const double B = sp.ch_B[i], P = sp.P[i];
        const double pnli = sp.eta[i] * P * P * P;
        const double nf = sp.ch_nf ? sp.ch_nf[i] : 1.0;
        const double f_abs = sp.ch_frel[i] + sp.f_ref;
        const double gain = exp(-sp.lnrho_L[i]);
        const double pase = sp.n_spans * nf * 6.62607015e-34 * (f_abs * 1e12) * (gain - 1.0) * (B * 1e12);
        const bool off = !(P > 0.0) || (sp.guard && sp.guard[i]);
        double snr = 0.0;
        if (!off) {
            snr = P / (pnli + pase);
            if (sp.snr_trx_lin_inv > 0.0) snr = 1.0 / (1.0 / snr + sp.snr_trx_lin_inv);
            tpart += 2.0 * B * log2(1.0 + snr);
        }
        sp.snr[i] = snr;
        sp.pnli[i] = pnli;
        sp.pase[i] = pase;
    }
    const double T = block_sum_d(tpart, scratch);
    if (threadIdx.x == 0 && sp.T) sp.T[0] = T;
}

cudaError_t launch_snr_from_eta(const SnrFromEtaParams &sp, cudaStream_t st)
{
    k_snr_from_eta<<<1, 256, 0, st>>>(sp);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_prep(const PrepParams &pp, int n_prof, cudaStream_t st)
{
    k_prep<<<dim3(n_prof, pp.n_steps + 1), 256, 0, st>>>(pp);
    return cudaGetLastError();
}

namespace {

size_t fwd_smem(int n_steps, int block)
{
    return sizeof(float4) * 2 * (size_t)step_pairs(n_steps) + fwd_warp_bytes(n_steps) * (size_t)(block / 32);
}

}  // namespace

// Persistent launch of the quadrature.  FP32: the warps of a block work alone,
// so a block is any number of them: as many as fit in shared memory (fewer than
// asked only past ~1,800 z-steps), one where there are too few tiles to give every
// SM a full block (a 5-channel plan's ~90 tiles then run on as many SMs).
cudaError_t launch_quad(const QuadParams &qp, int precision, int num_sms, int block, cudaStream_t st)
{
    int nb = 0, tiles = qp.n_items;
    size_t smem = (size_t)qp.n_steps * (2 * sizeof(double2) + f64_cand(qp.n_steps, qp.G) * sizeof(double)) +
                  (size_t)qp.G * sizeof(RowD);
    const void *fn = (const void *)k_quad_f64;
    if (precision == 0) {
        fn = (const void *)k_quad_f32;
        if (qp.n_items < num_sms * (block / 32)) block = 32;
        while (block > 32 && fwd_smem(qp.n_steps, block) > 200 * 1024) block -= 32;
        smem = fwd_smem(qp.n_steps, block);
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

cudaError_t launch_finish(const FinishParams &fp, int n_prof, cudaStream_t st)
{
    k_finish<<<n_prof, 512, 0, st>>>(fp);
    return cudaGetLastError();
}

}  // namespace isrs
