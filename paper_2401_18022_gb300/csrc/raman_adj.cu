// Adjoint of the FP32 quadrature with the tabulated (Raman-ODE) profile: the
// sensitivities of the throughput T (Sec. IV, Eq. loss) to the profile tables
// {a_c(m), b_c(m)} and to the PSD products, given dT/dSigma_i of every CUT.
//
// For a grid point of piece (a, b) of CUT i with F_c in candidate channel c,
//   ln p_m = A(m) + Sa(m) da + Sb(m) db,
//   A = (a_a + a_b + a_c - a_i + b_c D) / 2,  Sa = (b_a + b_c)/2,  Sb = (b_b + b_c)/2,
// with da = F_a - f_a, db = F_b - f_b, D = f_a + f_b - f_i - f_c.  With the
// per-(piece, candidate) buckets
//   R(m)  = sum_points ybar_i w W d|S|^2/d ln p_m,   Ra(m) = same * da,   Rb(m) = same * db,
// the chain rule gives
//   dT/da_a, dT/da_b, dT/da_c += R/2,   dT/da_i -= R/2,
//   dT/db_a += Ra/2,  dT/db_b += Rb/2,  dT/db_c += (D R + Ra + Rb)/2,
// and the PSD products W = P_a P_b P_c / (B_a B_b B_c) add
//   dT/d ln P_x += ybar_i w W |S|^2 for x = a, b, c.
//
// k_quad_adj_tab takes the nodes of every piece's row sums (quad_nodes.cuh) once
// per candidate channel, so a warp's buckets stay in registers, and evaluates
// every step term once: a node is walked by a half-warp (quad_walk.cuh), whose
// lanes keep their steps' terms t_m in registers; the half sums them into S with
// shuffles, and the same registers give d|S|^2/d ln p_m = 2 Re(conj(S) t_m).  The
// 557-channel launch at G = 64 took 377 ms with every point walked, about 28 ms with
// the nodes.  The same pass sums the forward
// value w W |S|^2 (the tile's partial of Sigma_i), so no separate forward runs.
// The buckets are not yet weighted by dT/dSigma_i (unknown until every tile
// of CUT i is done): at the end of a candidate the warp adds them, in
// order, into the rows of its own tile (one row per plan channel the tile
// touches, owned by this warp alone), and k_tab_gather applies dT/dSigma_i and
// sums each channel's rows in tile order, so the gradient is reproducible bit
// for bit.
#include <cuda_runtime.h>

#include <algorithm>

#include "isrs_internal.cuh"
#include "isrs_kernels.h"
#include "quad_common.cuh"
#include "quad_nodes.cuh"
#include "quad_tab.cuh"
#include "quad_walk.cuh"

namespace isrs {

namespace {

constexpr unsigned kFullT = 0xffffffffu;
constexpr int kTabAdjSlots = 512;   // node slots of a chunk
// One warp's shared memory: nodes, the points to walk, the candidate's rows.
template <int K2>
struct __align__(16) AdjTabWarp {
    WarpNodes<kTabAdjSlots> ns;
    float4 L[32];                // {mult w W af, phi, phi_lo, dl}
    float Ld[32];                // dd
    float4 qa[K2 * 16];          // {A, A', Sl, Sl'} of a pair, [k][lane of the half]
    float2 qb[K2 * 16];          // {Sd, Sd'}
};

}  // namespace

#ifndef ISRS_ADJ_TAB_MIN_BLOCKS
#define ISRS_ADJ_TAB_MIN_BLOCKS 2   // resident blocks per SM the register budget is sized for (3 spill, 4 more so)
#endif

template <int K2>
__global__ void __launch_bounds__(256, ISRS_ADJ_TAB_MIN_BLOCKS) k_quad_adj_tab(AdjTabParams ap)
{
    const QuadParams &qp = ap.q;
    extern __shared__ float4 smem_f4[];
    const int M = qp.n_steps, G = qp.G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l16 = lane & 15, half = lane >> 4;
    float4 *ze = smem_f4, *zd = ze + K2 * 16;          // walk_tables
    AdjTabWarp<K2> &w = reinterpret_cast<AdjTabWarp<K2> *>(zd + K2 * 16)[warp];
    auto &ns = w.ns;
    walk_tables<K2>(qp, ze, zd);
    __syncthreads();
    const float phi_direct = 3.14159265f / qp.dz_max;
    const unsigned lt_mask = (1u << lane) - 1u;

    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(qp.counter, 1);
        it = __shfl_sync(kFullT, it, 0);
        if (it >= qp.n_items) break;
        const DevItem item = qp.items[it];
        const int part = item.part & 0xffff, parts = item.part >> 16;
        // this tile's rows start at zero
        const int row0 = ap.row_off[it];
        const int nrow = ap.row_off[it + 1] - row0;
        double2 *trows = ap.rows + (size_t)row0 * M;
        double *trowsV = ap.rowsV + row0;
        for (int t = lane; t < nrow * M; t += 32) trows[t] = make_double2(0.0, 0.0);
        for (int t = lane; t < nrow; t += 32) trowsV[t] = 0.0;
        double acc = 0.0;           // the tile's partial of Sigma_i (lane 0)
        for (int kp = item.piece0; kp < item.piece1; ++kp) {
            const DevPiece &pc = qp.pieces[dbg_clamp(kp, qp.n_pieces, kDbgPiece, qp.dbg)];
            __syncwarp();
            const bool sw = node_geo(qp, pc, item.prof, 0.0f, qp.pd_f, 0.0f, ns.geo);
            const TabPiece tp = tab_piece(qp, pc, item.prof, sw);
            const int coff = qp.plan_ch_off[pc.plan];
            const int4 pr = ap.prow[kp];
            __syncwarp();
            PieceGeo &g = ns.geo;
            const PieceBlocks pb = row_blocks(ns, qp.gauss, G);
            for (int cc = 0; cc < g.nc; ++cc) {
                const double fc = qp.ch_frel[coff + pc.c_lo + cc];
                float tilt = 0.0f;
                for (int t = lane; t < K2 * 16; t += 32) {
                    const int m = walk_step<K2>(t >> 4, t & 15, 0);
                    const float4 none = make_float4(kPadLog2, 0.0f, 0.0f, 0.0f);
                    const float4 r = m < M ? tab_row(tp, pc.c_lo + cc, fc, m, M) : none;
                    const float4 u = m + 1 < M ? tab_row(tp, pc.c_lo + cc, fc, m + 1, M) : none;
                    w.qa[t] = make_float4(r.x, u.x, r.y, u.y);
                    w.qb[t] = make_float2(r.z, u.z);
                    tilt = fmaxf(tilt, fmaxf(fmaxf(fabsf(r.y), fabsf(r.z)), fmaxf(fabsf(u.y), fabsf(u.z))));
                }
                tilt = 0.69314718f * __uint_as_float(__reduce_max_sync(kFullT, __float_as_uint(tilt)));
                if (lane == 0) g.tilt = tilt;
                __syncwarp();
                f32x2 R[K2], Rl[K2], Rd[K2];
#pragma unroll
                for (int k = 0; k < K2; ++k) R[k] = Rl[k] = Rd[k] = dup2(0.0f);
                float sum = 0.0f, comp = 0.0f;
                const auto add = [&](float val) {
                    const float y = val - comp;
                    const float t = sum + y;
                    comp = (t - sum) - y;
                    sum = t;
                };
                piece_nodes(ns, pb, qp.gauss, G, cc, cc + 1, [&](int c0, int nq) {
                    for (int q0 = 32 * part; q0 < nq; q0 += 32 * parts) {
                        Node nd;
                        int cls = -1;
                        if (q0 + lane < nq) {
                            node_get(ns, qp.gauss, c0, q0 + lane, nd);
                            cls = fabsf(nd.phi) <= phi_direct ? 0 : 1;
                        }
                        const unsigned bd = __ballot_sync(kFullT, cls == 0), bt = __ballot_sync(kFullT, cls == 1);
                        if (cls >= 0) {
                            const int at = cls == 0 ? __popc(bd & lt_mask) : 31 - __popc(bt & lt_mask);
                            w.L[at] = make_float4(g.mult * nd.wq * g.wab * g.pd[cc] *
                                                      array_factor_f(nd.phi, qp, nd.phi_lo),
                                                  nd.phi, nd.phi_lo, tp.ol + nd.x);
                            w.Ld[at] = tp.od + nd.y;
                        }
                        __syncwarp();
                        const int nd0 = __popc(bd), nt0 = __popc(bt);
                        for (int f = 0; f < 2; ++f) {
                            const int cnt = f ? nt0 : nd0;
                            for (int p = 0; p < cnt; p += 2) {
                                const int e = min(p + half, cnt - 1), at = f ? 31 - e : e;
                                const float4 v = w.L[at];
                                const float dd = w.Ld[at];
                                const f32x2 dl2 = dup2(v.w), dd2 = dup2(dd);
                                const float4 *qa = w.qa + l16;
                                const float2 *qb = w.qb + l16;
                                const auto lp = [&](int k) {
                                    const float4 x = qa[k * 16];
                                    const float2 y = qb[k * 16];
                                    return fma2(pack2(y.x, y.y), dd2, fma2(pack2(x.z, x.w), dl2, pack2(x.x, x.y)));
                                };
                                f32x2 tr[K2], ti[K2];
                                float sr, si, cp = p + half < cnt ? v.x : 0.0f;
                                if (f) {
                                    walk_tele<K2, false>(ze + l16, l16, v.y, v.z, lp, tr, ti, sr, si);
                                    cp *= __fdividef(zsum_gain(true), v.y * v.y);
                                } else {
                                    walk_direct<K2>(zd + l16, v.y, lp, tr, ti, sr, si);
                                    cp *= zsum_gain(false);
                                }
                                const f32x2 c2 = dup2(2.0f * cp), cl = dup2(2.0f * cp * v.w), cd = dup2(2.0f * cp * dd);
                                const f32x2 sr2 = dup2(sr), si2 = dup2(si);
#pragma unroll
                                for (int k = 0; k < K2; ++k) {
                                    const f32x2 rr = walk_term<K2>(tr, ti, k, sr2, si2);
                                    R[k] = fma2(c2, rr, R[k]);
                                    Rl[k] = fma2(cl, rr, Rl[k]);
                                    Rd[k] = fma2(cd, rr, Rd[k]);
                                }
                                add(l16 == 0 ? cp * fmaf(sr, sr, si * si) : 0.0f);
                            }
                        }
                        __syncwarp();
                    }
                });
                double vtot = (double)sum - (double)comp;
                vtot += __shfl_down_sync(kFullT, vtot, 16);
                const double D = tp.Dl - fc;
                // the tile's rows, written by this warp alone: one lane per step, in
                // program order, so rows that coincide (a = CUT, c = b) add in a
                // fixed order; reductions without a result, so no lane waits
                double2 *ra = trows + (size_t)pr.x * M, *rb = trows + (size_t)pr.y * M;
                double2 *ri = trows + (size_t)pr.z * M, *rc = trows + (size_t)(pr.w + cc) * M;
#pragma unroll
                for (int k = 0; k < K2; ++k) {
                    float v[6];
                    unpack2(R[k], v[0], v[1]);
                    unpack2(Rl[k], v[2], v[3]);
                    unpack2(Rd[k], v[4], v[5]);
#pragma unroll
                    for (int t = 0; t < 6; ++t) v[t] += __shfl_xor_sync(kFullT, v[t], 16);
                    // each half adds one place of the pair
                    const int m = walk_step<K2>(k, l16, half);
                    if (m < M) {
                        const double r0 = 0.5 * (double)(half ? v[1] : v[0]);
                        const double f1 = 0.5 * (double)(half ? v[3] : v[2]), f2 = 0.5 * (double)(half ? v[5] : v[4]);
                        const double r1 = sw ? f2 : f1, r2 = sw ? f1 : f2;
                        if (pr.x != pr.z) {              // a = CUT: the two terms cancel
                            atomicAdd(&ra[m].x, r0);
                            atomicAdd(&ri[m].x, -r0);
                        }
                        atomicAdd(&rb[m].x, r0);
                        atomicAdd(&rc[m].x, r0);
                        atomicAdd(&ra[m].y, r1);
                        atomicAdd(&rb[m].y, r2);
                        atomicAdd(&rc[m].y, fma(D, r0, r1 + r2));
                    }
                }
                if (lane == 0) {
                    acc += vtot;
                    atomicAdd(&trowsV[pr.x], vtot);
                    atomicAdd(&trowsV[pr.y], vtot);
                    atomicAdd(&trowsV[pr.w + cc], vtot);
                }
                __syncwarp();
            }
        }
        if (lane == 0) qp.partial[it] = acc;
    }
}

// dT/d{a_c, b_c}(m) and dT/d ln P_c (PSD): the rows of channel c from every
// tile that touches it, weighted by dT/dSigma of the tile's CUT.  One block per
// plan channel and 32 steps (lane = step); its warps take equal shares of the
// rows in tile order and are summed in warp order.  Bound by reading the rows
// (16 M bytes each); one block per channel in one
// chain over its rows left a 41-channel plan on 41 SMs (1.95 ms).
constexpr int kGatherWarps = 16;

__global__ void __launch_bounds__(32 * kGatherWarps) k_tab_gather(TabGatherParams gp)
{
    __shared__ double2 part[kGatherWarps][32];
    __shared__ double partV[kGatherWarps];
    const int c = blockIdx.x, M = gp.n_steps, m = blockIdx.y * 32 + (threadIdx.x & 31);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e0 = gp.gath_off[c], len = gp.gath_off[c + 1] - e0;
    const int ea = e0 + (int)((long long)len * warp / kGatherWarps);
    const int eb = e0 + (int)((long long)len * (warp + 1) / kGatherWarps);
    double ga = 0.0, gb = 0.0, gv = 0.0;
    for (int e = ea; e < eb; e += 32) {
        int row = 0;
        double y = 0.0;
        if (e + lane < eb) {
            const int2 rs = gp.gath[e + lane];
            row = rs.x;
            y = gp.ybar[gp.slot_cut[rs.y]];
            if (blockIdx.y == 0) gv += y * gp.rowsV[row];
        }
        const int n = min(32, eb - e);
#pragma unroll 8
        for (int i = 0; i < n; ++i) {
            const int r = __shfl_sync(kFullT, row, i);
            const double yi = __shfl_sync(kFullT, y, i);
            if (m < M) {
                const double2 v = gp.rows[(size_t)r * M + m];
                ga += yi * v.x;
                gb += yi * v.y;
            }
        }
    }
    gv = warp_sum_d(gv);
    part[warp][lane] = make_double2(ga, gb);
    if (lane == 0) partV[warp] = gv;
    __syncthreads();
    if (warp != 0) return;
    ga = gb = gv = 0.0;
    for (int w = 0; w < kGatherWarps; ++w) {
        ga += part[w][lane].x;
        gb += part[w][lane].y;
        gv += partV[w];
    }
    if (m < M) gp.gAB[(size_t)c * M + m] = make_double2(ga, gb);
    if (blockIdx.y == 0 && lane == 0) gp.gV[c] = gv;
}

cudaError_t launch_tab_gather(const TabGatherParams &gp, cudaStream_t st)
{
    k_tab_gather<<<dim3(gp.n_ch, (gp.n_steps + 31) / 32), 32 * kGatherWarps, 0, st>>>(gp);
    return cudaGetLastError();
}

namespace {

template <int K2>
cudaError_t launch_adj_tab_k(const AdjTabParams &ap, int num_sms, int block, cudaStream_t st)
{
    if (ap.q.n_items < num_sms * (block / 32)) block = 32;      // too few tiles for full blocks on every SM
    const int nw = block / 32;
    const size_t smem = sizeof(float4) * 2 * K2 * 16 + sizeof(AdjTabWarp<K2>) * nw;
    cudaError_t e = cudaFuncSetAttribute(k_quad_adj_tab<K2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_quad_adj_tab<K2>, block, smem);
    if (e != cudaSuccess) return e;
    const int grid = std::max(1, std::min((ap.q.n_items + nw - 1) / nw, num_sms * std::max(1, nb)));
    k_quad_adj_tab<K2><<<grid, block, smem, st>>>(ap);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_adjoint_tab(const AdjTabParams &ap, int num_sms, int block, cudaStream_t st)
{
    switch ((ap.q.n_steps + 31) / 32) {
    case 1: return launch_adj_tab_k<1>(ap, num_sms, block, st);
    case 2: return launch_adj_tab_k<2>(ap, num_sms, block, st);
    case 3: return launch_adj_tab_k<3>(ap, num_sms, block, st);
    case 4: return launch_adj_tab_k<4>(ap, num_sms, block, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace isrs
