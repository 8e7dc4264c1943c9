// Multi-channel-interference (MCI) cells of the ISRS GN integral (App. A:
// the frequency integral of Eq. gain_fin runs over the whole band, so besides
// the CUT's own row and column of channel-pair cells (SCI, XCI) it contains
// every cell (a, b) with neither F_a nor F_b in the CUT's channel).
//
// For N channels there are (N-1) N / 2 such cells per CUT after folding the
// mirror cell (b, a) onto (a, b) (the integrand is symmetric in f1, f2), so
// no piece list is built: a work item is a range of cells of one CUT in the
// triangular order of the pairs (a', b'), a' <= b', of the N - 1 channels
// other than the CUT (a = a' + [a' >= i], likewise b), decoded from the index.
// Each cell lies in one
// quadrant (channel a does not straddle f_i) and gets its own G_mci x G_mci
// hyperbolic grid: rows uniform in ln(upsilon1), columns uniform in upsilon2,
// exactly as the per-piece grids of the SCI/XCI cells.  The z-sum and the
// closed-form profile are those of k_quad_f32 / k_quad_f64; far cells reach
// phases of ~1e8 revolutions, so the FP32 kernel's telescoped form uses the
// wide phase reduction.
#include <cuda_runtime.h>

#include "isrs_internal.cuh"
#include "isrs_kernels.h"
#include "quad_common.cuh"
#include "quad_zsum.cuh"
#include "quad_cells.cuh"

namespace isrs {

namespace {

constexpr int kMciRows = 32;       // grid rows (and so cells) of a group at most
constexpr int kMciList = 96;       // points waiting: telescoped from the front, direct from the back (31 + 31 + 32)

struct __align__(16) MciWarpC {
    float4 row[kMciRows];           // mci_row
    float4 Lp[kMciList];            // {phi, F_c - f_i, attenuation part of log2 p, weight}
    int4 cell[kMciRows];            // {a, b, first F_c channel, last}
};

}  // namespace

// ---------------------------------------------------------------------------
// k_quad_mci_f32: persistent over MCI work items (cell ranges of one CUT), one
// block per item.  A round compacts the next cells whose F_c can fall in a channel
// and deals them to the warps; a warp takes up to 32 grid rows at a time, appends
// their points to a list per z-sum form and sums 32 at a time, one per lane, two
// steps at a time.  The profile depends on a point only through F_c and the
// attenuation, so the lists last for the whole item and only its end leaves lanes
// idle.  Bound by the XU pipe (20 cycles per warp and step).  (A thread per grid
// row, its points in turn, took both forms in most warps and idled the lanes whose
// cells have no F_c in a channel: 77 ms for every cell of 295 channels at G_mci 8, now
// 24 ms.)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 3) k_quad_mci_f32(QuadParams qp)
{
    extern __shared__ float4 smem_f4[];
    const int M = qp.n_steps, G = qp.G, M2 = step_pairs(M), GC = kMciRows / G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float4 *eB = smem_f4;                              // [M2] {edge/2pi hi, hi', lo, lo'}
    float4 *zD = eB + M2;                              // [M2] {z, z', dz, dz'}
    float4 *sp = zD + M2;                              // [M2] {A2, A2', K2, K2'} about the CUT
    MciWarpC &w = reinterpret_cast<MciWarpC *>(sp + M2)[warp];
    float *rel = reinterpret_cast<float *>(reinterpret_cast<MciWarpC *>(sp + M2) + nw);    // [n] channel centre - f_i
    float *hb = rel + qp.mci_n_max;                    // [n] B/2
    float *ha = hb + qp.mci_n_max;                     // [n] alpha/2 log2 e
    __shared__ CellRound cr;
    __shared__ double scratch[32];
    __shared__ int s_item;

    pair_tables(qp, eB, zD);
    const float phi_direct = 3.14159265f / qp.dz_max;
    const float phi_wide = 6.28318531f * 1048576.0f / qp.L;     // 2^20 revolutions over the span: one rounding does
    const float eps = (float)qp.eps_v1;
    const unsigned lt_mask = (1u << lane) - 1u;
    const float inv_G = 1.0f / (float)G;               // (q + 1/2) inv_G floors to q / G: q <= 1,024
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
        const int n = qp.plan_n[plan];
        const int i = item.cut;
        if (item.prof != cur_prof || i != cur_cut) {
            const double fi = qp.ch_frel[coff + i];
            for (int c = threadIdx.x; c < n; c += blockDim.x) {
                rel[c] = (float)(qp.ch_frel[coff + c] - fi);
                hb[c] = (float)(0.5 * qp.ch_B[coff + c]);
                ha[c] = (float)(0.5 * qp.ch_alpha[coff + c] * kLog2e);
            }
            const double2 *sd = qp.step_d + (size_t)item.prof * M;
            for (int k = threadIdx.x; k < M2; k += blockDim.x) {
                const double2 v = sd[2 * k], u = sd[min(2 * k + 1, M - 1)];
                sp[k] = make_float4((float)(kLog2e * fma(-v.y, fi, v.x)),
                                    2 * k + 1 < M ? (float)(kLog2e * fma(-u.y, fi, u.x)) : -1000.0f,
                                    (float)(-kLog2e * v.y), (float)(-kLog2e * u.y));
            }
            cur_prof = item.prof;
            cur_cut = i;
        }
        __syncthreads();
        const float *pd = qp.pd_f + qp.prof_ch_off[item.prof];     // [n] P/B
        const float fi = (float)qp.ch_frel[coff + i], ha_i = ha[i];
        const MciPhase ph = {(float)qp.beta2, (float)qp.c3, (float)qp.c4, fi};
        float sum = 0.0f, comp = 0.0f;
        int nl[2] = {0, 0};                              // list lengths (direct, telescoped)
        // one list's first 32 points, one per lane; of what is left at the item's end,
        // 32 / cnt lanes (a power of two) share a point's steps
        const auto flush = [&](int f) {
            const int cnt = min(nl[f], 32);
            const int lg = cnt > 16 ? 0 : cnt > 8 ? 1 : cnt > 4 ? 2 : cnt > 2 ? 3 : cnt > 1 ? 4 : 5;
            const int pt = lane >> lg, sub = lane - (pt << lg);
            const int k0 = (M2 * sub) >> lg, k1 = (M2 * (sub + 1)) >> lg;
            __syncwarp();
            {
                const int e = min(pt, cnt - 1);
                const float4 v = w.Lp[f ? e : kMciList - 1 - e];
                const f32x2 F2 = dup2(v.y), nat = dup2(-v.z);
                const auto lp = [&](int k) {
                    const float4 x = sp[k], z = zD[k];
                    return fma2(pack2(x.z, x.w), F2, fma2(nat, pack2(z.x, z.y), pack2(x.x, x.y)));
                };
                float2 S;
                if (f == 0) S = zsum_direct_part(v.x, lp, zD, k0, k1);
                else if (__any_sync(0xffffffffu, fabsf(v.x) > phi_wide))
                    S = zsum_tele_part<1>(v.x, 0.0f, lp, eB, k0, k1, turn_magic(v.x * qp.Lrev_hi));
                else S = zsum_tele_part<2>(v.x, 0.0f, lp, eB, k0, k1);
                for (int o = (1 << lg) >> 1; o > 0; o >>= 1) {
                    S.x += __shfl_xor_sync(0xffffffffu, S.x, o);
                    S.y += __shfl_xor_sync(0xffffffffu, S.y, o);
                }
                const float S2 = S.x * S.x + S.y * S.y, wt = pt < cnt && sub == 0 ? v.w * zsum_gain(f) : 0.0f;
                const float y = wt * (f ? __fdividef(S2, v.x * v.x) : S2) * array_factor_f<true>(v.x, qp) - comp;
                const float t = sum + y;
                comp = (t - sum) - y;
                sum = t;
            }
            __syncwarp();
            nl[f] -= cnt;
            const int at = f ? lane : kMciList - 1 - lane, step = f ? cnt : -cnt;
            if (lane < nl[f]) w.Lp[at] = w.Lp[at + step];          // at most 31 stay
            __syncwarp();
        };
        for (int t0 = item.piece0; t0 < item.piece1; t0 += blockDim.x) {
            const int nv = cell_round(cr, t0, item.piece1, n, i, rel, hb, pd, qp.dbg);
            const int v1 = nv * (warp + 1) / nw;
            const bool end = t0 + (int)blockDim.x >= item.piece1;
            // the item's last turn, without points, sums what is left
            for (int v = nv * warp / nw, more = 1; more; v += GC) {
                const int ncc = max(0, min(GC, v1 - v)), np = ncc * G * G;
                more = ncc > 0;
                if (!more && !end) break;
                if (lane < ncc) w.cell[lane] = cr.cell[v + lane];
                __syncwarp();
                if (lane < ncc * G) {
                    const int cc = (int)(((float)lane + 0.5f) * inv_G);
                    const int4 cl = w.cell[cc];
                    w.row[lane] = mci_row(fabsf(rel[cl.x]), fabsf(rel[cl.y]), hb[cl.x], hb[cl.y], eps, G,
                                          lane - cc * G, (cl.x == cl.y ? 1.0f : 2.0f) * (pd[cl.x] * pd[cl.y]));
                }
                __syncwarp();
#pragma unroll 1
                for (int q0 = 0; q0 < np || !more; q0 += 32) {
                    const int q = q0 + lane;
                    int cls = -1;
                    float4 pt = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (q < np) {
                        const int rr = (int)(((float)q + 0.5f) * inv_G);
                        const float4 o = w.row[rr];
                        if (o.w != 0.0f) {
                            const int4 cl = w.cell[(int)(((float)rr + 0.5f) * inv_G)];
                            const float2 f = mci_point(o, rel[cl.x], rel[cl.y], q - rr * G, G);
                            pt.y = f.x + f.y;
                            int ci = -1;
                            for (int c = cl.z; c <= cl.w; ++c)
                                if (rel[c] - hb[c] <= pt.y && pt.y < rel[c] + hb[c]) ci = c;
                            if (ci >= 0) {
                                pt.x = ph.at<true>(f.x, f.y);
                                pt.z = (ha[cl.x] + ha[cl.y] - ha_i) + ha[ci];
                                pt.w = o.w * pd[ci];
                                if (pt.w != 0.0f) cls = fabsf(pt.x) <= phi_direct ? 0 : 1;
                            }
                        }
                    }
#pragma unroll
                    for (int f = 0; f < 2; ++f) {
                        const unsigned m = __ballot_sync(0xffffffffu, cls == f);
                        const int e = nl[f] + __popc(m & lt_mask);
                        if (cls == f) w.Lp[f ? e : kMciList - 1 - e] = pt;
                        nl[f] += __popc(m);
                        if (nl[f] >= (more ? 32 : 1)) flush(f);
                    }
                    if (!more) break;
                }
                __syncwarp();
            }
        }
        const double tot = block_sum_d((double)sum - (double)comp, scratch);
        if (threadIdx.x == 0) qp.partial[it] = tot;
    }
}

__global__ void __launch_bounds__(256) k_quad_mci_f64(QuadParams qp)
{
    extern __shared__ double2 smem_d2[];
    const int M = qp.n_steps, G = qp.G;
    double2 *sz = smem_d2;                 // [M] {z_m, dz_m}
    double2 *st = sz + M;                  // [M] {lnPtot - lnN, kappa}
    __shared__ double scratch[32];
    __shared__ int s_item;

    for (int m = threadIdx.x; m < M; m += blockDim.x) sz[m] = qp.zs_d[m];
    const double phi_f64 = kF64Direct / qp.dz_max;
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
        __syncthreads();
        const int plan = qp.prof_plan[item.prof];
        const int coff = qp.plan_ch_off[plan];
        const int poff = qp.prof_ch_off[item.prof];
        const int n = qp.plan_n[plan];
        const int i = item.cut;
        const double *fr = qp.ch_frel + coff;
        const double *Bc = qp.ch_B + coff;
        const double *al = qp.ch_alpha + coff;
        const double *pdv = qp.pd_d + poff;
        const double fi = fr[i];
        const int n2 = n - 1;
        double sum = 0.0;
        const int nrows = (item.piece1 - item.piece0) * G;
        for (int q = threadIdx.x; q < nrows; q += blockDim.x) {
            const int tl = q / G, r = q - tl * G;
            int ap, bp;
            tri_decode(item.piece0 + tl, n2, ap, bp);
            const int a = dbg_clamp(ap + (ap >= i), n, kDbgCell, qp.dbg), b = dbg_clamp(bp + (bp >= i), n, kDbgCell, qp.dbg);
            const double mult = a == b ? 1.0 : 2.0;
            const double ra = fr[a] - fi, rb = fr[b] - fi;
            const double s1 = ra > 0.0 ? 1.0 : -1.0, s2 = rb > 0.0 ? 1.0 : -1.0;
            const double xlo = fabs(ra) - 0.5 * Bc[a], xhi = fabs(ra) + 0.5 * Bc[a];
            const double ylo = fabs(rb) - 0.5 * Bc[b], yhi = fabs(rb) + 0.5 * Bc[b];
            const double u1hi = xhi * yhi;
            const double llo = log(fmax(xlo * ylo, qp.eps_v1 * u1hi));
            const double ds = (log(u1hi) - llo) / G;
            const double u1 = exp(llo + (r + 0.5) * ds);
            const double ymin = fmax(ylo, u1 / xhi), ymax = fmin(yhi, u1 / xlo);
            if (!(ymax > ymin)) continue;
            const double du2 = log1p((ymax - ymin) / ymin) / G;
            const double yc = sqrt(ymin * ymax), xc = u1 / yc;
            const double w = u1 * ds * du2 * mult;
            for (int j = 0; j < G; ++j) {
                const double d = ((double)j + 0.5 - 0.5 * (double)G) * du2;
                const double f1 = s1 * (xc * exp(d)), f2 = s2 * (yc * exp(-d));
                const double u = f1 + f2;
                // channel of F_c = f_i + u
                int lo = 0, hi = n - 1, c = -1;
                while (lo <= hi) {
                    const int mid = (lo + hi) >> 1;
                    if (fr[mid] - fi - 0.5 * Bc[mid] <= u) {
                        c = mid;
                        lo = mid + 1;
                    } else {
                        hi = mid - 1;
                    }
                }
                if (c < 0 || !(u < fr[c] - fi + 0.5 * Bc[c])) continue;
                const double W = pdv[a] * pdv[b] * pdv[c];
                if (W == 0.0) continue;
                const double at = 0.5 * (al[a] + al[b] + al[c] - al[i]);
                const double Fc = fi + u;
                const double br = qp.beta2 + c3 * (u + 2.0 * fi) +
                                  c4 * (f1 * f1 + 1.5 * f1 * f2 + 3.0 * fi * u + f2 * f2 + 3.0 * fi * fi);
                const double phi = -4.0 * kPi * kPi * f1 * f2 * br;
                const double S2 = zsum_f64(phi, phi_f64, sz, M, [&](int m) {
                    const double2 tt = st[m];
                    return exp(tt.x - tt.y * Fc - at * sz[m].x);
                });
                sum += w * W * S2 * array_factor_d(phi, qp);
            }
        }
        const double tot = block_sum_d(sum, scratch);
        if (threadIdx.x == 0) qp.partial[it] = tot;
    }
}

size_t quad_mci_smem_bytes(int precision, int n_steps, int n_max, int block)
{
    if (precision == 0)
        return (size_t)step_pairs(n_steps) * 3 * sizeof(float4) + sizeof(MciWarpC) * (block / 32) +
               (size_t)n_max * 3 * sizeof(float);
    return (size_t)n_steps * 2 * sizeof(double2);
}

int quad_mci_blocks_per_sm(int precision, int n_steps, int n_max, int block)
{
    int nb = 0;
    const size_t smem = quad_mci_smem_bytes(precision, n_steps, n_max, block);
    void *fn = precision == 0 ? (void *)k_quad_mci_f32 : (void *)k_quad_mci_f64;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, block, smem);
    return nb > 0 ? nb : 1;
}

cudaError_t launch_quad_mci(const QuadParams &qp, int precision, int grid, int block, cudaStream_t st)
{
    const size_t smem = quad_mci_smem_bytes(precision, qp.n_steps, qp.mci_n_max, block);
    void *fn = precision == 0 ? (void *)k_quad_mci_f32 : (void *)k_quad_mci_f64;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    QuadParams q = qp;
    void *args[] = {&q};
    return cudaLaunchKernel(fn, dim3(grid), dim3(block), args, smem, st);
}

}  // namespace isrs
