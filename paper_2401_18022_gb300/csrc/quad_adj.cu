// Adjoint of the FP32 quadrature: the gradient of the throughput T (Sec. IV,
// Eq. loss) with respect to every launch power P_j, through eta (App. A,
// Eqs. gain_fin, psi_fin, pk, slow_vary), the ASE gain and the SNR numerator.
//
// With the closed-form linear-slope profile, per grid point and step
//   ln p_m = A_m - kappa_m (F_c - f_ref) - at z_m,   A_m = ln P_tot - ln N(z_m),
// so the powers enter |S|^2 only through (A_m, kappa_m), shared by every point,
// and through the PSD product W = P_a P_b P_c / (B_a B_b B_c).  For CUT i:
//   dSigma_i/dP_j = V_ij / P_j + sum_m R_im dA_m/dP_j - sum_m R'_im dkappa_m/dP_j
// with the buckets
//   R_im  = sum_points w W d|S|^2/d ln p_m,
//   R'_im = sum_points w W (F_c - f_ref) d|S|^2/d ln p_m,
//   V_ij  = sum_points w W |S|^2 (number of j among the point's a, b, c).
//
// k_quad_adj evaluates the forward sum and these buckets in one pass over the
// nodes of the row sums (quad_nodes.cuh; the bucket terms have the band limit of
// |S|^2, so the nodes that sum a row sum its derivatives too), and every step
// term of Eq. slow_vary is evaluated once: a node is walked by a half-warp
// (quad_walk.cuh), each of the 16 lanes owning 2 K2 consecutive steps computes
// their terms t_m into registers, the half sums them with shuffles into S, and the
// same registers give d|S|^2/d ln p_m = 2 Re(conj(S) t_m) for the lane's own step
// buckets, which stay in registers between FP64 folds.  Those registers (128) leave
// 16 warps an SM, so the chain phase -> sin, cos -> term -> half sum -> bucket bounds
// it: issue 61 %, XU pipe 47 %.  557 channels at G = 128: 610 -> 42.6 ms.
#include <cuda_runtime.h>

#include "isrs_internal.cuh"
#include "isrs_kernels.h"
#include <algorithm>

#include "quad_common.cuh"
#include "quad_nodes.cuh"
#include "quad_walk.cuh"

namespace isrs {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kAdjSlots = 512;   // node slots of a chunk
constexpr int kAdjCand = 3;      // F_c candidates swept together (most pieces have two)
using AdjNodes = WarpNodes<kAdjSlots>;

// One warp's shared memory: nodes, the points to walk, step rows per
// candidate, FP64 step buckets.
template <int K2>
struct __align__(16) AdjWarp {
    AdjNodes ns;
    float4 L[32];                // {w W af, phi, phi_lo, u}
    int Lc[32];                  // candidate, from the sweep's first
    float4 ek[kAdjCand][K2 * 16];   // {log2 p at f_c (2), slope K2 (2)} of a pair, [k][lane of the half]
    double2 B[2 * K2 * 16];         // [step of the lane][lane]
};

}  // namespace

// ---------------------------------------------------------------------------
// k_quad_adj<K2>: fused forward + adjoint, persistent over work tiles of one
// profile; every warp takes its own tiles.  Per batch of 32 slots a warp sets up
// one node per lane, lists the direct ones from the front and the telescoped
// ones from the back, and walks them two at a time, one per half-warp (an odd
// one beside a zero-weight copy of itself).  Lane buckets accumulate in
// registers over a piece and are folded into the warp's FP64 buckets, which go
// to the tile's own row; PSD buckets are added to the tile's own row by one
// lane.  Every sum has a fixed order (k_adj_reduce sums a CUT's rows in tile
// order), so results are bit for bit reproducible.
// ---------------------------------------------------------------------------
#ifndef ISRS_ADJ_MIN_BLOCKS
#define ISRS_ADJ_MIN_BLOCKS 2   // resident blocks per SM the register budget is sized for (3 spill, 4 more so)
#endif

template <int K2>
__global__ void __launch_bounds__(256, ISRS_ADJ_MIN_BLOCKS) k_quad_adj(AdjParams ap)
{
    const QuadParams &qp = ap.q;
    extern __shared__ float4 smem_f4[];
    const int M = qp.n_steps, G = qp.G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l16 = lane & 15, half = lane >> 4;
    float4 *ze = smem_f4, *zd = ze + K2 * 16;          // walk_tables
    AdjWarp<K2> &w = reinterpret_cast<AdjWarp<K2> *>(zd + K2 * 16)[warp];
    AdjNodes &ns = w.ns;

    walk_tables<K2>(qp, ze, zd);
    __syncthreads();
    const float phi_direct = 3.14159265f / qp.dz_max;
    const float phi_small = kSmallPhiL / (qp.L * (float)qp.n_spans);
    const float log2e = (float)kLog2e;
    const unsigned lt_mask = (1u << lane) - 1u;
    PathCount count;

    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(qp.counter, 1);
        it = __shfl_sync(kFull, it, 0);
        if (it >= qp.n_items) break;
        const DevItem item = qp.items[it];
        const float2 *st = qp.step_f + (size_t)item.prof * M;
        const float tilt = (float)qp.kap_L[item.prof];
        const int part = item.part & 0xffff, parts = item.part >> 16;
        double *Vrow = ap.V + (size_t)it * ap.n_ch;     // this tile's PSD buckets
        for (int c = lane; c < ap.n_ch; c += 32) Vrow[c] = 0.0;
        for (int t = lane; t < 2 * K2 * 16; t += 32) w.B[t] = make_double2(0.0, 0.0);
        double acc = 0.0;                               // lane 0
        for (int kp = item.piece0; kp < item.piece1; ++kp) {
            const DevPiece &pc = qp.pieces[dbg_clamp(kp, qp.n_pieces, kDbgPiece, qp.dbg)];
            __syncwarp();
            node_geo(qp, pc, item.prof, log2e, qp.pd_f, tilt, ns.geo);
            __syncwarp();
            const PieceGeo &g = ns.geo;
            const float mult = g.mult;
            f32x2 R[K2], Rp[K2];
#pragma unroll
            for (int k = 0; k < K2; ++k) R[k] = Rp[k] = dup2(0.0f);
            double ptot = 0.0;
            const PieceBlocks pb = row_blocks(ns, qp.gauss, G);
            if (lane == 0 && part == 0) count.small += pb.R1 * G;
            for (int ca = 0; ca < g.nc; ca += kAdjCand) {
                const int cb = min(g.nc, ca + kAdjCand);
                for (int c = ca; c < cb; ++c) {
                    const float at = g.at_ab + g.hat[c], F = g.Fc0 + (0.5f * (g.lo[c] + g.hi[c]) - g.Fi);
                    for (int t = lane; t < K2 * 16; t += 32) {
                        const int m = walk_step<K2>(t >> 4, t & 15, 0);
                        float4 e = make_float4(kPadLog2, kPadLog2, 0.0f, 0.0f);
                        if (m < M) {
                            const float2 v = st[m];
                            e.x = fmaf(v.y, F, fmaf(-at, zd[t].x, v.x));
                            e.z = v.y;
                        }
                        if (m + 1 < M) {
                            const float2 v = st[m + 1];
                            e.y = fmaf(v.y, F, fmaf(-at, zd[t].y, v.x));
                            e.w = v.y;
                        }
                        w.ek[c - ca][t] = e;
                    }
                }
                __syncwarp();
                // forward sum (compensated) and PSD buckets of the candidates, on
                // lane 0 of each half
                float sum = 0.0f, comp = 0.0f, v0 = 0.0f, v1 = 0.0f, v2 = 0.0f;
                const auto add = [&](float val, int c) {
                    const float y = val - comp;
                    const float t = sum + y;
                    comp = (t - sum) - y;
                    sum = t;
                    v0 += c == 0 ? val : 0.0f;
                    v1 += c == 1 ? val : 0.0f;
                    v2 += c == 2 ? val : 0.0f;
                };
                piece_nodes(ns, pb, qp.gauss, G, ca, cb, [&](int c0, int nq) {
                    for (int q0 = 32 * part; q0 < nq; q0 += 32 * parts) {
                        Node nd;
                        int cls = -1;
                        if (q0 + lane < nq) {
                            node_get(ns, qp.gauss, c0, q0 + lane, nd);
                            const float aphi = fabsf(nd.phi);
                            cls = aphi <= phi_direct ? 0 : 1;
                            count.points(aphi, phi_small, cls == 1, nd.N);
                        }
                        const unsigned bd = __ballot_sync(kFull, cls == 0), bt = __ballot_sync(kFull, cls == 1);
                        if (cls >= 0) {
                            const int ci = dbg_clamp(nd.ci, g.nc, kDbgCand, qp.dbg);
                            const int at = cls == 0 ? __popc(bd & lt_mask) : 31 - __popc(bt & lt_mask);
                            w.L[at] = make_float4(nd.wq * g.wab * g.pd[ci] * array_factor_f(nd.phi, qp, nd.phi_lo),
                                                  nd.phi, nd.phi_lo, nd.x + nd.y);
                            w.Lc[at] = ci - ca;
                        }
                        __syncwarp();
                        const int nd0 = __popc(bd), nt0 = __popc(bt);
                        for (int f = 0; f < 2; ++f) {
                            const int cnt = f ? nt0 : nd0;
                            if (lane == 0) count.sums(f, cnt);
                            for (int p = 0; p < cnt; p += 2) {
                                const int e = min(p + half, cnt - 1), at = f ? 31 - e : e;
                                const float4 v = w.L[at];
                                const int c = w.Lc[at];
                                const float wq = p + half < cnt ? v.x : 0.0f;
                                const f32x2 dF = dup2(v.w - (0.5f * (g.lo[ca + c] + g.hi[ca + c]) - g.Fi));
                                const float4 *ek = w.ek[c] + l16;
                                const auto lp = [&](int k) {
                                    const float4 x = ek[k * 16];
                                    return fma2(pack2(x.z, x.w), dF, pack2(x.x, x.y));
                                };
                                f32x2 tr[K2], ti[K2];
                                float sr, si, sq = wq;
                                if (f) {
                                    walk_tele<K2, false>(ze + l16, l16, v.y, v.z, lp, tr, ti, sr, si);
                                    sq *= __fdividef(zsum_gain(true), v.y * v.y);
                                } else {
                                    walk_direct<K2>(zd + l16, v.y, lp, tr, ti, sr, si);
                                    sq *= zsum_gain(false);
                                }
                                const f32x2 c2 = dup2(2.0f * mult * sq), cF = dup2(2.0f * mult * sq * (g.Fc0 + v.w));
                                const f32x2 sr2 = dup2(sr), si2 = dup2(si);
#pragma unroll
                                for (int k = 0; k < K2; ++k) {
                                    const f32x2 rr = walk_term<K2>(tr, ti, k, sr2, si2);
                                    R[k] = fma2(c2, rr, R[k]);
                                    Rp[k] = fma2(cF, rr, Rp[k]);
                                }
                                add(l16 == 0 ? sq * fmaf(sr, sr, si * si) : 0.0f, c);
                            }
                        }
                        __syncwarp();
                    }
                });
                // sweep totals: the two halves' lane 0 meet on lane 0
                const double s = (double)sum - (double)comp;
                const double sw = (double)mult * (s + __shfl_down_sync(kFull, s, 16));
                const float w0 = __shfl_down_sync(kFull, v0, 16), w1 = __shfl_down_sync(kFull, v1, 16),
                            w2 = __shfl_down_sync(kFull, v2, 16);
                if (lane == 0) {
                    ptot += sw;
                    // one lane, in order; the row is this tile's
                    for (int c = ca; c < cb; ++c) {
                        const double vc = c == ca ? (double)v0 + (double)w0
                                        : c == ca + 1 ? (double)v1 + (double)w1 : (double)v2 + (double)w2;
                        atomicAdd(&Vrow[dbg_clamp(pc.c_lo + c, ap.n_ch, kDbgVrow, qp.dbg)], (double)mult * vc);
                    }
                }
                __syncwarp();
            }
            if (lane == 0) {
                acc += ptot;
                atomicAdd(&Vrow[dbg_clamp(pc.a, ap.n_ch, kDbgVrow, qp.dbg)], ptot);
                atomicAdd(&Vrow[dbg_clamp(pc.b, ap.n_ch, kDbgVrow, qp.dbg)], ptot);
            }
#pragma unroll
            for (int k = 0; k < K2; ++k) {
                float x0, x1, y0, y1;
                unpack2(R[k], x0, x1);
                unpack2(Rp[k], y0, y1);
                x0 += __shfl_xor_sync(kFull, x0, 16);
                x1 += __shfl_xor_sync(kFull, x1, 16);
                y0 += __shfl_xor_sync(kFull, y0, 16);
                y1 += __shfl_xor_sync(kFull, y1, 16);
                // each half folds one place of the pair
                double2 &d = w.B[(2 * k + half) * 16 + l16];
                d.x += (double)(half ? x1 : x0);
                d.y += (double)(half ? y1 : y0);
            }
        }
        // tile outputs: the forward partial and the step buckets
        if (lane == 0) qp.partial[it] = acc;
        __syncwarp();
        for (int m = lane; m < M; m += 32) {
            const int ln = m / (2 * K2), kk = m - ln * 2 * K2;
            ap.item_R[(size_t)it * M + m] = w.B[kk * 16 + ln];
        }
        __syncwarp();
    }
    if (qp.path_count) count.store(qp.path_count);
}

// ---------------------------------------------------------------------------
// Chain rule (FP64).  Notation: s_i = SNR_i = P_i / N_i (optionally with
// 1/SNR += t), N_i = P_NLI,i + P_ASE,i, P_NLI,i = K_i Sigma_i with
// K_i = (16/27) gamma_i^2 B_i, P_ASE,i = NF h f B (G_i - 1), G_i = 1/rho(L,f_i),
// T = 2 sum_i B_i log2(1 + s_i).  Then ds/dN = -s^2/P and ds/dP|_N = s^2 N/P^2.
// For the closed-form profile at any z (kappa = P_tot C_r L_eff(z)):
//   d ln rho(z,F)/dP_j = 1/P_tot - h_j(kappa)/N(z) - C_r L_eff(z) (F - Fbar(z)),
//   h_j(kappa) = e^{-kappa f_j'} sinhc(kappa B_j/2),  Fbar = tilted mean frequency.
// ---------------------------------------------------------------------------
constexpr int kMaxAdjSteps = 128;
constexpr double kHPlanck = 6.62607015e-34;

__global__ void __launch_bounds__(256) k_ybar(ChainParams cp)
{
    for (int i = threadIdx.x + blockIdx.x * blockDim.x; i < cp.n_ch; i += blockDim.x * gridDim.x) {
        const double P = cp.P[i], B = cp.ch_B[i], g = cp.ch_gamma[i], snr = cp.snr[i];
        const double dTds = 2.0 * B / (0.69314718055994530942 * (1.0 + snr));
        const double dsdN = -snr * snr / P;
        const double nf = cp.ch_nf ? cp.ch_nf[i] : 1.0;
        const double hfb = cp.n_spans * nf * kHPlanck * ((cp.ch_frel[i] + cp.f_ref) * 1e12) * (B * 1e12);
        cp.ybar[i] = dTds * dsdN * (16.0 / 27.0) * g * g * B;
        cp.aase[i] = dTds * dsdN * (cp.pase[i] + hfb);    // dT/dASE * dASE/d ln G
    }
}

// The tiles' buckets, every sum in a fixed order.  Blocks [0, n_steps): Rb[m] =
// sum over tiles of ybar(channel of tile) {R_m, R'_m}.  Block n_steps + s: V[s][j]
// = the PSD buckets of slot s's tiles (regular, then MCI): lane = channel, each of
// the eight warps an eighth of the tiles in tile order, the eighths in order (a
// thread per channel over all 144 tiles took 24 us at 5 channels).
__global__ void __launch_bounds__(256) k_adj_reduce(ChainParams cp)
{
    __shared__ double scratch[32];
    if ((int)blockIdx.x < cp.n_steps) {
        const int m = blockIdx.x;
        double rx = 0.0, ry = 0.0;
        for (int it = threadIdx.x; it < cp.n_items; it += blockDim.x) {
            const double y = cp.ybar[cp.slot_cut[cp.item_slot[it]]];
            const double2 v = cp.item_R[(size_t)it * cp.n_steps + m];
            rx += y * v.x;
            ry += y * v.y;
        }
        rx = block_sum_d(rx, scratch);
        ry = block_sum_d(ry, scratch);
        if (threadIdx.x == 0) cp.Rb[m] = make_double2(rx, ry);
        return;
    }
    const int s = blockIdx.x - cp.n_steps, n = cp.n_ch;
    const int2 r1 = cp.slot_items[s];
    const int2 r2 = cp.slot_items2 ? cp.slot_items2[s] : make_int2(0, 0);
    __shared__ double part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, t1 = r1.y - r1.x, tn = t1 + r2.y - r2.x;
    for (int j0 = 0; j0 < n; j0 += 32) {
        double v = 0.0;
        if (j0 + lane < n)
            for (int t = tn * warp / 8; t < tn * (warp + 1) / 8; ++t)
                v += cp.Vt[(size_t)(t < t1 ? r1.x + t : cp.n_items_reg + r2.x + t - t1) * n + j0 + lane];
        __syncthreads();
        part[warp][lane] = v;
        __syncthreads();
        if (warp == 0 && j0 + lane < n) {
            v = 0.0;
            for (int w = 0; w < 8; ++w) v += part[w][lane];
            cp.Vs[(size_t)s * n + j0 + lane] = v;
        }
    }
}

// The chain rule from the buckets, one warp per channel j: its lanes split the
// steps and the output slots, a warp tree sums them.  The step terms cs = [lnN |
// kappa | L_eff | Fbar - f_ref] (M + 1 each) come from the forward's k_prep; the
// sums over all channels and steps that every channel needs are a few hundred
// terms, so each block takes them itself, in the same order (as launches of their
// own the step terms took 17 us and the sums 5 us of a 5-channel gradient).
__global__ void __launch_bounds__(256) k_chain_ch(ChainParams cp)
{
    __shared__ double scratch[32];
    const int n = cp.n_ch, M = cp.n_steps, st = M + 1;
    const int lane = threadIdx.x & 31;
    const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const double *lnN = cp.cs, *kap = cp.cs + st, *Le = cp.cs + 2 * st, *Fb = cp.cs + 3 * st;
    double pt = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
    for (int m = threadIdx.x; m < M; m += blockDim.x) a1 += cp.Rb[m].y * Le[m];
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        pt += cp.P[i];
        a2 += cp.aase[i];
        a3 += cp.aase[i] * (cp.ch_frel[i] - Fb[M]);
    }
    a1 = block_sum_d(a1, scratch);
    pt = block_sum_d(pt, scratch);
    a2 = block_sum_d(a2, scratch);
    a3 = block_sum_d(a3, scratch);
    if (j >= n) return;                  // warp-uniform
    const double k0 = -cp.Cr * a1, k2 = cp.Cr * Le[M] * a3;      // R' term, ASE tilt term
    const double invPt = 1.0 / pt;
    const double fj = cp.ch_frel[j], hB = 0.5 * cp.ch_B[j];
    double gm = 0.0;
    for (int m = lane; m < M; m += 32) {
        const double hN = exp(log_sinhc(kap[m] * hB) - kap[m] * fj - lnN[m]);
        gm += cp.Rb[m].x * (invPt - hN + cp.Cr * Le[m] * Fb[m]);
    }
    double v = 0.0;
    for (int s = lane; s < cp.n_slots; s += 32) v += cp.ybar[cp.slot_cut[s]] * cp.V[(size_t)s * n + j];
    gm = warp_sum_d(gm);
    v = warp_sum_d(v);
    if (lane == 0) {
        double g = k0 + gm + v / cp.P[j];
        if (cp.with_direct) {
            // through the ASE gain of every channel, and the SNR numerator
            const double hNL = exp(log_sinhc(kap[M] * hB) - kap[M] * fj - lnN[M]);
            g += -a2 * (invPt - hNL) + k2;
            const double snr = cp.snr[j], P = cp.P[j], B = cp.ch_B[j];
            const double N = cp.pnli[j] + cp.pase[j];
            const double dTds = 2.0 * B / (0.69314718055994530942 * (1.0 + snr));
            g += dTds * snr * snr * N / (P * P);
        }
        cp.dT_dP[j] = g;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
namespace {

template <int K2>
cudaError_t launch_adj_k(const AdjParams &ap, int num_sms, int block, cudaStream_t st)
{
    if (ap.q.n_items < num_sms * (block / 32)) block = 32;      // too few tiles for full blocks on every SM
    const int nw = block / 32;
    const size_t smem = sizeof(float4) * 2 * K2 * 16 + sizeof(AdjWarp<K2>) * nw;
    cudaError_t e = cudaFuncSetAttribute(k_quad_adj<K2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_quad_adj<K2>, block, smem);
    if (e != cudaSuccess) return e;
    const int grid = std::max(1, std::min((ap.q.n_items + nw - 1) / nw, num_sms * std::max(1, nb)));
    k_quad_adj<K2><<<grid, block, smem, st>>>(ap);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_adjoint(const AdjParams &ap, int num_sms, int block, cudaStream_t st)
{
    switch ((ap.q.n_steps + 31) / 32) {
    case 1: return launch_adj_k<1>(ap, num_sms, block, st);
    case 2: return launch_adj_k<2>(ap, num_sms, block, st);
    case 3: return launch_adj_k<3>(ap, num_sms, block, st);
    case 4: return launch_adj_k<4>(ap, num_sms, block, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_ybar(const ChainParams &cp, cudaStream_t st)
{
    k_ybar<<<(cp.n_ch + 127) / 128, 128, 0, st>>>(cp);
    return cudaGetLastError();
}

cudaError_t launch_chain(const ChainParams &cp, cudaStream_t st)
{
    if (cp.n_steps > kMaxAdjSteps) return cudaErrorInvalidValue;
    cudaError_t e = launch_ybar(cp, st);
    if (e != cudaSuccess) return e;
    k_adj_reduce<<<cp.n_steps + cp.n_slots, 256, 0, st>>>(cp);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_chain_ch<<<(cp.n_ch + 7) / 8, 256, 0, st>>>(cp);
    return cudaGetLastError();
}

}  // namespace isrs
