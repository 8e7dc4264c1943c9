// Adjoint over the multi-channel-interference (MCI) cells on their own grid
// (App. A: the frequency integral of Eq. gain_fin over the whole band; the
// cells (a, b) with neither F_a nor F_b in the CUT's channel, each on a
// G_mci x G_mci hyperbolic grid as in the MCI quadrature).  With the
// closed-form profile it fills, for its work items, the same quantities as
// the fused adjoint of the SCI/XCI pieces:
//   R_im  = sum_points w W d|S|^2/d ln p_m,   R'_im = same * (F_c - f_ref),
//   V_ij += w W |S|^2 for each of the point's channels a, b, c,
// and the forward partial of each item, so the chain rule (k_chain_ch) takes the
// MCI items as further tiles of their CUTs.
//
// A block takes an item: a round compacts the next cells whose F_c can fall in a
// channel and deals them to the warps.  A warp takes their points 32 at a time
// (the row set-up is per point), lists them by z-sum form, and
// walks a full list two points at a time on half-warps (quad_walk.cuh), every step
// term evaluated once and reused for the bucket terms.  Far cells reach phases
// of ~1e8 revolutions, so the telescoped walk uses the wide phase reduction.
// The PSD buckets go to one shared row per warp over the plan's channels, a
// warp sum for each channel that occurs among a list's points (few: consecutive
// cells share a and neighbour in b and c), in a fixed order; the rows are summed
// over the warps in order.
#include <cuda_runtime.h>

#include <algorithm>

#include "isrs_internal.cuh"
#include "isrs_kernels.h"
#include "quad_cells.cuh"
#include "quad_common.cuh"
#include "quad_walk.cuh"

namespace isrs {

namespace {

constexpr int kMciList = 96;       // points waiting: telescoped from the front, direct from the back (31 + 31 + 32)
constexpr int kFoldLists = 128;    // lists walked between FP64 folds of the register buckets (2,048 terms a lane)

// One warp's shared memory; its PSD buckets [n] follow.
template <int K2>
struct __align__(16) AdjMciWarp {
    float4 L[kMciList];          // {w W af, phi, F_c - f_ref, attenuation}
    int2 ch[kMciList];           // {a | b << 16, c}
    float val[32];
    double2 B[2 * K2 * 16];      // FP64 step buckets, [step of the lane][lane]
};

// row[ch] += the sum of val over the lanes with channel ch, for every ch that
// occurs (ch < 0: none); ascending in the lane that first holds it.
__device__ __forceinline__ void v_add(float *row, int ch, float val, int lane)
{
    unsigned todo = __ballot_sync(kWarpAll, ch >= 0);
    while (todo) {
        const int c = __shfl_sync(kWarpAll, ch, __ffs(todo) - 1);
        float v = ch == c ? val : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kWarpAll, v, o);
        if (lane == 0) row[c] += v;
        todo &= ~__ballot_sync(kWarpAll, ch == c);
    }
}

}  // namespace

#ifndef ISRS_ADJ_MCI_MIN_BLOCKS
#define ISRS_ADJ_MCI_MIN_BLOCKS 3   // resident blocks per SM the register budget is sized for
#endif

template <int K2>
__global__ void __launch_bounds__(256, ISRS_ADJ_MCI_MIN_BLOCKS) k_quad_adj_mci(AdjParams ap)
{
    const QuadParams &qp = ap.q;
    extern __shared__ float4 smem_f4[];
    const int M = qp.n_steps, G = qp.G;
    const int G2 = G * G;
    const int nw = blockDim.x >> 5;
    const int nmax = (qp.mci_n_max + 3) & ~3;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l16 = lane & 15, half = lane >> 4;
    float4 *ze = smem_f4, *zd = ze + K2 * 16;                 // walk_tables
    float4 *wk = zd + K2 * 16;                                // [K2][16] {A2, A2', K2, K2'} of the profile
    AdjMciWarp<K2> *ws = reinterpret_cast<AdjMciWarp<K2> *>(wk + K2 * 16);   // [nw]
    AdjMciWarp<K2> &w = ws[warp];
    float *rel = reinterpret_cast<float *>(ws + nw);          // [nmax] channel centre - f_i
    float *hb = rel + nmax;                                   // [nmax] B/2
    float *pd = hb + nmax;                                    // [nmax] P/B
    float *ha = pd + nmax;                                    // [nmax] alpha/2 log2 e
    float *sV = ha + nmax;                                    // [nw][nmax] PSD buckets of the item
    __shared__ CellRound cr;
    __shared__ double scratch[32];
    __shared__ int s_item;

    walk_tables<K2>(qp, ze, zd);
    for (int t = lane; t < 2 * K2 * 16; t += 32) w.B[t] = make_double2(0.0, 0.0);
    const float phi_direct = 3.14159265f / qp.dz_max;
    const float phi_small = kSmallPhiL / (qp.L * (float)qp.n_spans);
    const float eps = (float)qp.eps_v1;
    const unsigned lt_mask = (1u << lane) - 1u;
    PathCount count;
    int cur_prof = -1, cur_cut = -1;

    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(qp.counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= qp.n_items) break;
        const DevItem item = qp.items[it];
        const int plan = qp.prof_plan[item.prof];
        const int coff = qp.plan_ch_off[plan];
        const int poff = qp.prof_ch_off[item.prof];
        const int n = qp.plan_n[plan];
        const int i = item.cut;
        if (item.prof != cur_prof) {
            const float2 *st = qp.step_f + (size_t)item.prof * M;
            for (int t = threadIdx.x; t < K2 * 16; t += blockDim.x) {
                const int m = walk_step<K2>(t >> 4, t & 15, 0);
                const float2 v = m < M ? st[m] : make_float2(kPadLog2, 0.0f);
                const float2 u = m + 1 < M ? st[m + 1] : make_float2(kPadLog2, 0.0f);
                wk[t] = make_float4(v.x, u.x, v.y, u.y);
            }
        }
        if (item.prof != cur_prof || i != cur_cut) {
            const double fi = qp.ch_frel[coff + i];
            for (int c = threadIdx.x; c < n; c += blockDim.x) {
                rel[c] = (float)(qp.ch_frel[coff + c] - fi);
                hb[c] = (float)(0.5 * qp.ch_B[coff + c]);
                pd[c] = qp.pd_f[poff + c];
                ha[c] = (float)(0.5 * qp.ch_alpha[coff + c] * kLog2e);
            }
            cur_prof = item.prof;
            cur_cut = i;
        }
        for (int t = threadIdx.x; t < nw * nmax; t += blockDim.x) sV[t] = 0.0f;
        __syncthreads();
        float *myV = sV + warp * nmax;
        const float fi = (float)qp.ch_frel[coff + i];
        const MciPhase ph = {(float)qp.beta2, (float)qp.c3, (float)qp.c4, fi};
        const float ha_i = ha[i];
        float sum = 0.0f, comp = 0.0f;
        f32x2 R[K2], Rp[K2];
#pragma unroll
        for (int k = 0; k < K2; ++k) R[k] = Rp[k] = dup2(0.0f);
        int nd = 0, nt = 0, lists = 0;      // list lengths (warp-uniform)
        const auto fold = [&]() {
#pragma unroll
            for (int k = 0; k < K2; ++k) {
                float x0, x1, y0, y1;
                unpack2(R[k], x0, x1);
                unpack2(Rp[k], y0, y1);
                x0 += __shfl_xor_sync(kWarpAll, x0, 16);
                x1 += __shfl_xor_sync(kWarpAll, x1, 16);
                y0 += __shfl_xor_sync(kWarpAll, y0, 16);
                y1 += __shfl_xor_sync(kWarpAll, y1, 16);
                // each half folds one place of the pair
                double2 &d = w.B[(2 * k + half) * 16 + l16];
                d.x += (double)(half ? x1 : x0);
                d.y += (double)(half ? y1 : y0);
                R[k] = Rp[k] = dup2(0.0f);
            }
            lists = 0;
        };
        // walks a list's first 32 points (or what is left)
        const auto flush = [&](bool tele) {
            const int len = tele ? nt : nd, cnt = min(len, 32);
            if (lane == 0) count.sums(tele, cnt);
            __syncwarp();
            for (int p = 0; p < cnt; p += 2) {
                const int e = min(p + half, cnt - 1), at = tele ? e : kMciList - 1 - e;
                const float4 v = w.L[at];
                const f32x2 F2 = dup2(v.z), nat = dup2(-v.w);
                const auto lp = [&](int k) {
                    const float4 x = wk[k * 16 + l16], z = zd[k * 16 + l16];
                    return fma2(nat, pack2(z.x, z.y), fma2(pack2(x.z, x.w), F2, pack2(x.x, x.y)));
                };
                f32x2 tr[K2], ti[K2];
                float sr, si, sq = p + half < cnt ? v.x : 0.0f;
                if (tele) {
                    walk_tele<K2, true>(ze + l16, l16, v.y, 0.0f, lp, tr, ti, sr, si, turn_magic(v.y * qp.Lrev_hi));
                    sq *= __fdividef(zsum_gain(true), v.y * v.y);
                } else {
                    walk_direct<K2>(zd + l16, v.y, lp, tr, ti, sr, si);
                    sq *= zsum_gain(false);
                }
                const f32x2 c2 = dup2(2.0f * sq), cF = dup2(2.0f * sq * v.z), sr2 = dup2(sr), si2 = dup2(si);
#pragma unroll
                for (int k = 0; k < K2; ++k) {
                    const f32x2 rr = walk_term<K2>(tr, ti, k, sr2, si2);
                    R[k] = fma2(c2, rr, R[k]);
                    Rp[k] = fma2(cF, rr, Rp[k]);
                }
                if (l16 == 0 && p + half < cnt) w.val[p + half] = sq * fmaf(sr, sr, si * si);
            }
            __syncwarp();
            const int at = tele ? lane : kMciList - 1 - lane, step = tele ? cnt : -cnt;
            const bool live = lane < cnt;
            const float val = live ? w.val[lane] : 0.0f;
            const int2 ch = live ? w.ch[at] : make_int2(0, 0);
            const float y = val - comp, t = sum + y;
            comp = (t - sum) - y;
            sum = t;
            v_add(myV, live ? ch.x & 0xffff : -1, val, lane);
            v_add(myV, live ? ch.x >> 16 : -1, val, lane);
            v_add(myV, live ? ch.y : -1, val, lane);
            if (lane < len - cnt) {                      // at most 31 stay
                w.L[at] = w.L[at + step];
                w.ch[at] = w.ch[at + step];
            }
            if (tele) nt = len - cnt;
            else nd = len - cnt;
            __syncwarp();
            if (++lists == kFoldLists) fold();
        };
        for (int t0 = item.piece0; t0 < item.piece1; t0 += blockDim.x) {
            const int nv = cell_round(cr, t0, item.piece1, n, i, rel, hb, pd, qp.dbg);
            const int v0 = nv * warp / nw, npts = (nv * (warp + 1) / nw - v0) * G2;   // this warp's cells
            for (int q0 = 0; q0 < npts; q0 += 32) {
                // this lane's grid point: cell, row and column from its index
                const int q = q0 + lane;
                float phi = 0.0f, Fc = 0.0f, at = 0.0f, wwa = 0.0f;
                int cls = -1, a = 0, b = 0, c = -1;
                if (q < npts) {
                    const int tl = q / G2, rem = q - tl * G2;
                    const int r = rem / G, j = rem - r * G;
                    const int4 cl = cr.cell[v0 + tl];
                    a = cl.x;
                    b = cl.y;
                    const float ra = rel[a], rb = rel[b];
                    const float4 row = mci_row(fabsf(ra), fabsf(rb), hb[a], hb[b], eps, G, r, a == b ? 1.0f : 2.0f);
                    if (row.w != 0.0f) {
                        const float2 f = mci_point(row, ra, rb, j, G);
                        const float u = f.x + f.y;
                        for (int x = cl.z; x <= cl.w; ++x)
                            if (rel[x] - hb[x] <= u && u < rel[x] + hb[x]) c = x;
                        if (c >= 0) {
                            const float W = pd[a] * pd[b] * pd[c];
                            if (W != 0.0f) {
                                at = ha[a] + ha[b] - ha_i + ha[c];
                                Fc = fi + u;
                                phi = ph.at<true>(f.x, f.y);
                                wwa = row.w * W * array_factor_f<true>(phi, qp);
                                cls = fabsf(phi) <= phi_direct ? 0 : 1;
                            }
                        }
                    }
                }
                const unsigned bd = __ballot_sync(kWarpAll, cls == 0), bt = __ballot_sync(kWarpAll, cls == 1);
                if (cls >= 0) {
                    const int pos = cls ? nt + __popc(bt & lt_mask) : kMciList - 1 - (nd + __popc(bd & lt_mask));
                    w.L[pos] = make_float4(wwa, phi, Fc, at);
                    w.ch[pos] = make_int2(a | b << 16, c);
                    count.points(fabsf(phi), phi_small, cls, 1);
                }
                nd += __popc(bd);
                nt += __popc(bt);
                if (nt >= 32) flush(true);
                if (nd >= 32) flush(false);
            }
        }
        if (nt > 0) flush(true);
        if (nd > 0) flush(false);
        fold();
        // item outputs: the forward partial, the PSD buckets and the step buckets
        const double tot = block_sum_d((double)sum - (double)comp, scratch);   // syncs the block
        if (threadIdx.x == 0) qp.partial[it] = tot;
        double *Vrow = ap.V + (size_t)it * ap.n_ch;     // this tile's own row (k_adj_reduce sums them)
        for (int c = threadIdx.x; c < n; c += blockDim.x) {
            double v = 0.0;
            for (int x = 0; x < nw; ++x) v += (double)sV[x * nmax + c];
            Vrow[c] = v;
        }
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
            const int ln = m / (2 * K2), kk = m - ln * 2 * K2;
            double rx = 0.0, ry = 0.0;
            for (int x = 0; x < nw; ++x) {
                const double2 bb = ws[x].B[kk * 16 + ln];
                rx += bb.x;
                ry += bb.y;
            }
            ap.item_R[(size_t)it * M + m] = make_double2(rx, ry);
        }
        __syncthreads();
        for (int t = lane; t < 2 * K2 * 16; t += 32) w.B[t] = make_double2(0.0, 0.0);
    }
    if (qp.path_count) count.store(qp.path_count);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
namespace {

template <int K2>
cudaError_t launch_adj_mci_k(const AdjParams &ap, int num_sms, int block, cudaStream_t st)
{
    const auto bytes = [&](int b) {
        const int nw = b / 32;
        return sizeof(float4) * 3 * K2 * 16 + sizeof(AdjMciWarp<K2>) * nw +
               sizeof(float) * (size_t)(4 + nw) * ((ap.q.mci_n_max + 3) & ~3);
    };
    while (block > 32 && bytes(block) > 200 * 1024) block -= 32;
    const size_t smem = bytes(block);
    cudaError_t e = cudaFuncSetAttribute(k_quad_adj_mci<K2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int nb = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_quad_adj_mci<K2>, block, smem);
    if (e != cudaSuccess) return e;
    const int grid = std::max(1, std::min(ap.q.n_items, num_sms * std::max(1, nb)));
    k_quad_adj_mci<K2><<<grid, block, smem, st>>>(ap);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_adjoint_mci(const AdjParams &ap, int num_sms, int block, cudaStream_t st)
{
    switch ((ap.q.n_steps + 31) / 32) {
    case 1: return launch_adj_mci_k<1>(ap, num_sms, block, st);
    case 2: return launch_adj_mci_k<2>(ap, num_sms, block, st);
    case 3: return launch_adj_mci_k<3>(ap, num_sms, block, st);
    case 4: return launch_adj_mci_k<4>(ap, num_sms, block, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace isrs
