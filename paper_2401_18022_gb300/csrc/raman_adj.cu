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
// every step term once: a node is walked by a half-warp, each of the 16 lanes
// owning K = ceil(M/16) consecutive steps, which keeps their terms t_m in
// registers; the half sums them into S with shuffles, and the same registers
// give d|S|^2/d ln p_m = 2 Re(conj(S) t_m).  The same pass sums the forward
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
constexpr float kPadLog2T = -1000.0f;

// Half-warp walks of a node (weight cp = mult w W af, phi float-float, in-channel
// offsets dl, dd of the longer and the shorter axis).  Lane l16 owns steps [K
// l16, K l16 + K) with zt[k][16] = {edge/2pi hi, lo, z, dz} and the candidate's
// q[k][16] = {A, Sl, Sd} (offset by l16; padding steps carry log2 weight -1000).
// Each walk adds the lane's bucket terms R += cp d|S|^2/d ln p_m, Rl += dl
// (same), Rd += dd (same) and returns |S|^2.
template <int K>
__device__ __forceinline__ float walk_direct_t(const float4 *zt, const float4 *q, float cp, float ph, float dl,
                                               float dd, float (&R)[K], float (&Rl)[K], float (&Rd)[K])
{
    const float hph = 0.5f * ph;
    const float phr = ph * 0.15915494309189535f;
    float tr[K], ti[K];
    float sr = 0.0f, si = 0.0f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float4 e = q[k * 16];
        const float4 z = zt[k * 16];
        float sn, cs;
        sincos_rev(phr, z.z, sn, cs);
        const float amp = ex2_approx(fmaf(e.z, dd, fmaf(e.y, dl, e.x))) * (sinc_poly(hph * z.w) * z.w);
        tr[k] = amp * cs;
        ti[k] = amp * sn;
        sr += tr[k];
        si += ti[k];
    }
    sr = half_sum(sr);
    si = half_sum(si);
    const float c2 = 2.0f * cp, ca = c2 * dl, cb = c2 * dd;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float rr = fmaf(sr, tr[k], si * ti[k]);
        R[k] = fmaf(c2, rr, R[k]);
        Rl[k] = fmaf(ca, rr, Rl[k]);
        Rd[k] = fmaf(cb, rr, Rd[k]);
    }
    return fmaf(sr, sr, si * si);
}

template <int K>
__device__ __forceinline__ float walk_tele_t(const float4 *zt, const float4 *q, int l16, float cp, float ph,
                                             float ph_lo, float dl, float dd, float (&R)[K], float (&Rl)[K],
                                             float (&Rd)[K])
{
    float tr[K], ti[K];
    float Er = 1.0f, Ei = 0.0f, p0 = 0.0f, e1r = 1.0f, e1i = 0.0f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float4 e = q[k * 16];
        const float4 z = zt[k * 16];
        float sn, cs;
        phasor_rev_ff(ph, z.x, z.y, sn, cs, ph_lo);
        const float pm = ex2_approx(fmaf(e.z, dd, fmaf(e.y, dl, e.x)));
        if (k == 0) {
            p0 = pm;
            e1r = cs;
            e1i = sn;
            tr[0] = 0.0f;
            ti[0] = 0.0f;
        } else {
            tr[k] = pm * (cs - Er);
            ti[k] = pm * (sn - Ei);
        }
        Er = cs;
        Ei = sn;
    }
    // the lower edge of this lane's first step is the previous lane's last edge
    float elr = __shfl_up_sync(kFullT, Er, 1, 16);
    float eli = __shfl_up_sync(kFullT, Ei, 1, 16);
    elr = l16 == 0 ? 1.0f : elr;
    eli = l16 == 0 ? 0.0f : eli;
    tr[0] = p0 * (e1r - elr);
    ti[0] = p0 * (e1i - eli);
    float ur = 0.0f, ui = 0.0f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        ur += tr[k];
        ui += ti[k];
    }
    ur = half_sum(ur);
    ui = half_sum(ui);
    const float iph2 = __fdividef(1.0f, ph * ph);
    const float c2 = 2.0f * cp * iph2, ca = c2 * dl, cb = c2 * dd;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float rr = fmaf(ur, tr[k], ui * ti[k]);
        R[k] = fmaf(c2, rr, R[k]);
        Rl[k] = fmaf(ca, rr, Rl[k]);
        Rd[k] = fmaf(cb, rr, Rd[k]);
    }
    return fmaf(ur, ur, ui * ui) * iph2;
}

// One warp's shared memory: nodes, the points to walk, the candidate's rows.
template <int K>
struct __align__(16) AdjTabWarp {
    WarpNodes<kTabAdjSlots> ns;
    float4 L[32];                // {mult w W af, phi, phi_lo, dl}
    float Ld[32];                // dd
    float4 q[K * 16];            // {A, Sl, Sd}, [k][lane of the half]
};

}  // namespace

#ifndef ISRS_ADJ_TAB_MIN_BLOCKS
#define ISRS_ADJ_TAB_MIN_BLOCKS 3   // resident blocks per SM the register budget is sized for
#endif

template <int K>
__global__ void __launch_bounds__(256, ISRS_ADJ_TAB_MIN_BLOCKS) k_quad_adj_tab(AdjTabParams ap)
{
    const QuadParams &qp = ap.q;
    extern __shared__ float4 smem_f4[];
    const int M = qp.n_steps, G = qp.G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l16 = lane & 15, half = lane >> 4;
    float4 *zt = smem_f4;                              // [K][16] {edge/2pi hi, lo, z, dz}
    AdjTabWarp<K> &w = reinterpret_cast<AdjTabWarp<K> *>(zt + K * 16)[warp];
    auto &ns = w.ns;
    // padding steps past M repeat the last edge
    for (int t = threadIdx.x; t < K * 16; t += blockDim.x) {
        const int m = min((t & 15) * K + (t >> 4), M - 1);
        const float4 za = qp.zs_a[m], zb = qp.zs_b[m];
        zt[t] = make_float4(zb.x, zb.y, za.x, za.w);
    }
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
            for (int cc = 0; cc < g.nc; ++cc) {
                const double fc = qp.ch_frel[coff + pc.c_lo + cc];
                float tilt = 0.0f;
                for (int t = lane; t < K * 16; t += 32) {
                    const int m = (t & 15) * K + (t >> 4);
                    float4 r = make_float4(kPadLog2T, 0.0f, 0.0f, 0.0f);
                    if (m < M) r = tab_row(tp, pc.c_lo + cc, fc, m, M);
                    w.q[t] = r;
                    tilt = fmaxf(tilt, fmaxf(fabsf(r.y), fabsf(r.z)));
                }
                tilt = 0.69314718f * __uint_as_float(__reduce_max_sync(kFullT, __float_as_uint(tilt)));
                if (lane == 0) g.tilt = tilt;
                __syncwarp();
                float R[K], Rl[K], Rd[K];
#pragma unroll
                for (int k = 0; k < K; ++k) R[k] = Rl[k] = Rd[k] = 0.0f;
                float sum = 0.0f, comp = 0.0f;
                const auto add = [&](float val) {
                    const float y = val - comp;
                    const float t = sum + y;
                    comp = (t - sum) - y;
                    sum = t;
                };
                int small;
                piece_nodes(ns, qp.gauss, G, cc, cc + 1, small, [&](int c0, int nq) {
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
                        for (int p = 0; p < nd0; p += 2) {
                            const int at = min(p + half, nd0 - 1);
                            const float4 v = w.L[at];
                            const float cp = p + half < nd0 ? v.x : 0.0f;
                            const float s2 = walk_direct_t<K>(zt + l16, w.q + l16, cp, v.y, v.w, w.Ld[at], R, Rl, Rd);
                            add(l16 == 0 ? cp * s2 : 0.0f);
                        }
                        for (int p = 0; p < nt0; p += 2) {
                            const int at = 31 - min(p + half, nt0 - 1);
                            const float4 v = w.L[at];
                            const float cp = p + half < nt0 ? v.x : 0.0f;
                            const float s2 = walk_tele_t<K>(zt + l16, w.q + l16, l16, cp, v.y, v.z, v.w, w.Ld[at], R,
                                                            Rl, Rd);
                            add(l16 == 0 ? cp * s2 : 0.0f);
                        }
                        __syncwarp();
                    }
                });
                double vtot = (double)sum - (double)comp;
                vtot += __shfl_down_sync(kFullT, vtot, 16);
                const int c = pc.c_lo + cc;
                const double D = tp.Dl - fc;
                // the tile's rows, written by this warp alone: one lane per step, in
                // program order, so rows that coincide (a = CUT, c = b) add in a
                // fixed order; reductions without a result, so no lane waits
                double2 *ra = trows + (size_t)pr.x * M, *rb = trows + (size_t)pr.y * M;
                double2 *ri = trows + (size_t)pr.z * M, *rc = trows + (size_t)(pr.w + cc) * M;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const float f0 = R[k] + __shfl_xor_sync(kFullT, R[k], 16);
                    const float f1 = Rl[k] + __shfl_xor_sync(kFullT, Rl[k], 16);
                    const float f2 = Rd[k] + __shfl_xor_sync(kFullT, Rd[k], 16);
                    const int m = l16 * K + k;
                    if (half == 0 && m < M) {
                        const double r0 = 0.5 * (double)f0, r1 = 0.5 * (double)(sw ? f2 : f1),
                                     r2 = 0.5 * (double)(sw ? f1 : f2);
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
// tile that touches it, weighted by dT/dSigma of the tile's CUT, in tile
// order.  One block per plan channel.
__global__ void __launch_bounds__(128) k_tab_gather(TabGatherParams gp)
{
    const int c = blockIdx.x, M = gp.n_steps;
    const int e0 = gp.gath_off[c], e1 = gp.gath_off[c + 1];
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
        double ga = 0.0, gb = 0.0;
        for (int e = e0; e < e1; ++e) {
            const int2 rs = gp.gath[e];
            const double y = gp.ybar[gp.slot_cut[rs.y]];
            const double2 v = gp.rows[(size_t)rs.x * M + m];
            ga += y * v.x;
            gb += y * v.y;
        }
        gp.gAB[(size_t)c * M + m] = make_double2(ga, gb);
    }
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int e = e0; e < e1; ++e) {
            const int2 rs = gp.gath[e];
            v += gp.ybar[gp.slot_cut[rs.y]] * gp.rowsV[rs.x];
        }
        gp.gV[c] = v;
    }
}

cudaError_t launch_tab_gather(const TabGatherParams &gp, cudaStream_t st)
{
    k_tab_gather<<<gp.n_ch, 128, 0, st>>>(gp);
    return cudaGetLastError();
}

namespace {

template <int K>
cudaError_t launch_adj_tab_k(const AdjTabParams &ap, int num_sms, int block, cudaStream_t st)
{
    if (ap.q.n_items < num_sms * (block / 32)) block = 32;      // too few tiles for full blocks on every SM
    const int nw = block / 32;
    const size_t smem = sizeof(float4) * K * 16 + sizeof(AdjTabWarp<K>) * nw;
    cudaError_t e = cudaFuncSetAttribute(k_quad_adj_tab<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_quad_adj_tab<K>, block, smem);
    if (e != cudaSuccess) return e;
    const int grid = std::max(1, std::min((ap.q.n_items + nw - 1) / nw, num_sms * std::max(1, nb)));
    k_quad_adj_tab<K><<<grid, block, smem, st>>>(ap);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_adjoint_tab(const AdjTabParams &ap, int num_sms, int block, cudaStream_t st)
{
    switch ((ap.q.n_steps + 15) / 16) {
    case 1: return launch_adj_tab_k<1>(ap, num_sms, block, st);
    case 2: return launch_adj_tab_k<2>(ap, num_sms, block, st);
    case 3: return launch_adj_tab_k<3>(ap, num_sms, block, st);
    case 4: return launch_adj_tab_k<4>(ap, num_sms, block, st);
    case 5: return launch_adj_tab_k<5>(ap, num_sms, block, st);
    case 6: return launch_adj_tab_k<6>(ap, num_sms, block, st);
    case 7: return launch_adj_tab_k<7>(ap, num_sms, block, st);
    case 8: return launch_adj_tab_k<8>(ap, num_sms, block, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace isrs
