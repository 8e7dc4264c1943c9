// Multi-channel-interference (MCI) cells on their own grid with the
// tabulated (Raman-ODE) power profile (Sec. III, App. A: the integral of
// Eq. gain_fin over the whole band, with rho(z, f) from the Raman
// power-evolution ODEs).
//
// The cells, their triangular enumeration and their G_mci x G_mci hyperbolic
// grids are those of quad_mci.cu.  Only the profile term of Eq. pk changes:
// inside channel c, ln rho(z_m, F) = a_c(m) + b_c(m) (F - f_c), so for a point
// of cell (a, b) with F_c in channel c and in-channel offsets
// da = F_a - f_a, db = F_b - f_b, dc = F_c - f_c,
//   ln p_m = 1/2 [a_a + a_b - a_i + a_c + b_a da + b_b db + b_c dc](m).
// For the few cells a warp takes together the FP32 kernel tabulates, per cell, F_c
// channel and pair of steps, {A, S_a, S_b} (log2 units; A at da = db = 0, S_a = (b_a +
// b_c)/2, S_b = (b_b + b_c)/2) in shared memory from an FP32 copy of the profile
// tables, so a step costs two FMAs for ln p.  The z-sum forms are those of
// quad_zsum.cuh.
#include <cuda_runtime.h>

#include <algorithm>

#include "f32x2.cuh"
#include "isrs_internal.cuh"
#include "isrs_kernels.h"
#include "quad_cells.cuh"
#include "quad_common.cuh"
#include "quad_zsum.cuh"

namespace isrs {

namespace {

constexpr int kMciCells = 6;       // cells of a group at most
constexpr int kMciUnits = 4;       // step rows of a group: one per cell and F_c channel
constexpr int kMciList = 96;       // points waiting: telescoped from the front, direct from the back (31 + 31 + 32)
constexpr int kMciRows = 32;       // rows of a group

// Cells a warp takes together: at most 32 grid rows (and kMciUnits step rows).
__host__ __device__ constexpr int mci_group(int G) { return G >= 32 ? 1 : (32 / G < kMciCells ? 32 / G : kMciCells); }

// {1/2 log2(e) a_c, 1/2 log2(e) b_c} in FP32: float4 {a, a', b, b'} of channel c and
// pair k at (prof_ch_off[p] + c) pairs + k, the order in which a warp reads them for
// its step rows.  One block row per profile.
__global__ void __launch_bounds__(256) k_tab_half_log2(TabHalfParams hp)
{
    const int p = blockIdx.y, n = hp.plan_n[hp.prof_plan[p]], M = hp.n_steps, M2 = step_pairs(M);
    const double2 *ab = hp.ab + (size_t)hp.prof_ch_off[p] * M;
    float4 *out = hp.abf + (size_t)hp.prof_ch_off[p] * M2;
    for (int t = threadIdx.x + blockIdx.x * blockDim.x; t < n * M2; t += blockDim.x * gridDim.x) {
        const int c = t / M2, k = t - c * M2;
        const double2 v = ab[(size_t)c * M + 2 * k], w = ab[(size_t)c * M + min(2 * k + 1, M - 1)];
        const double h = 0.5 * kLog2e;
        out[t] = make_float4((float)(h * v.x), (float)(h * w.x), (float)(h * v.y), (float)(h * w.y));
    }
}

// One warp's shared memory; the step rows of the group's cells follow it.
struct __align__(16) MciWarp {
    float4 row[kMciRows];            // {xc, yc, du2, w P_a P_b / (B_a B_b)}
    float4 Lp[kMciList];             // {phi, da, db, w W}
    int Lu[kMciList];                // step row
    int4 cell[kMciCells];            // {a | b << 16, first F_c channel, last, step row of the first}
    int2 unit[kMciUnits];            // {cell, F_c channel} of each step row
};

__host__ __device__ constexpr size_t mci_warp_bytes(int n_steps)
{
    // per step row float4 {A, A', Sa, Sa'} and float2 {Sb, Sb'} of every pair, the
    // pitches odd so that the rows of a warp's points sit in different banks
    return sizeof(MciWarp) + ((size_t)kMciUnits * (step_pairs(n_steps) | 1) * 24 + 15) / 16 * 16;
}

}  // namespace

// ---------------------------------------------------------------------------
// k_quad_mci_f32_tab: persistent over MCI work items (cell ranges of one CUT),
// one block per item.  A round compacts the next cells whose F_c can fall in a
// channel and deals them to the warps, which take them in groups of about 32
// grid rows: a step row for every cell and F_c channel (reading the F_c rows at
// every step instead left the loop waiting on L2: the block's shared memory leaves
// the L1 28 KB), then grid rows, then points, which go to a list per z-sum form and
// are summed 32 at a time, one per lane.  Bound by the XU pipe (20 cycles per warp
// and step; 74 % busy on 147 adjacent channels) and the issue of the rest (70 %).
// 557 channels, G_mci 8: 518 ms with the F_c rows read at every step, now 278 ms.
// ---------------------------------------------------------------------------
#ifndef ISRS_MCI_TAB_MIN_BLOCKS
#define ISRS_MCI_TAB_MIN_BLOCKS 3   // resident blocks per SM the register budget is sized for
#endif

__global__ void __launch_bounds__(256, ISRS_MCI_TAB_MIN_BLOCKS) k_quad_mci_f32_tab(QuadParams qp)
{
    extern __shared__ float4 smem_f4[];
    const int M = qp.n_steps, G = qp.G, M2 = step_pairs(M), MS = M2 | 1, GC = mci_group(G);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float4 *eB = smem_f4;                              // [M2] {edge/2pi hi, hi', lo, lo'}
    float4 *zD = eB + M2;                              // [M2] {z, z', dz, dz'}
    unsigned char *mine = reinterpret_cast<unsigned char *>(zD + M2) + mci_warp_bytes(M) * warp;
    MciWarp &w = *reinterpret_cast<MciWarp *>(mine);
    float4 *Qa = reinterpret_cast<float4 *>(mine + sizeof(MciWarp));       // [kMciUnits][MS]
    float2 *Qb = reinterpret_cast<float2 *>(Qa + (size_t)kMciUnits * MS);  // [kMciUnits][MS]
    float *rel = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(zD + M2) +
                                           mci_warp_bytes(M) * nw);     // [n] channel centre - f_i
    float *hb = rel + qp.mci_n_max;                    // [n] B/2
    __shared__ CellRound cr;
    __shared__ double scratch[32];
    __shared__ int s_item;

    pair_tables(qp, eB, zD);
    const float phi_direct = 3.14159265f / qp.dz_max;
    const float phi_wide = 6.28318531f * 1048576.0f / qp.L;     // 2^20 revolutions over the span: one rounding does
    const float eps = (float)qp.eps_v1;
    const unsigned lt_mask = (1u << lane) - 1u;
    const float inv_G = 1.0f / (float)G;               // (q + 1/2) inv_G floors to q / G: q < 1,024
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
        if (item.prof != cur_prof || i != cur_cut) {
            const double fi = qp.ch_frel[coff + i];
            for (int c = threadIdx.x; c < n; c += blockDim.x) {
                rel[c] = (float)(qp.ch_frel[coff + c] - fi);
                hb[c] = (float)(0.5 * qp.ch_B[coff + c]);
            }
            cur_prof = item.prof;
            cur_cut = i;
        }
        __syncthreads();
        const float4 *T = qp.ab_f + (size_t)poff * M2;   // this profile's channel rows
        const float *pd = qp.pd_f + poff;                // [n] P/B
        const float fi = (float)qp.ch_frel[coff + i];
        const MciPhase ph = {(float)qp.beta2, (float)qp.c3, (float)qp.c4, fi};
        float sum = 0.0f, comp = 0.0f;
        int nl[2] = {0, 0};                              // list lengths (direct, telescoped)
        // one list's first 32 points, one per lane; of what is left at a group's end, 32 /
        // cnt lanes (a power of two) share a point's steps
        const auto flush = [&](int f) {
            const int cnt = min(nl[f], 32);
            const int lg = cnt > 16 ? 0 : cnt > 8 ? 1 : cnt > 4 ? 2 : cnt > 2 ? 3 : cnt > 1 ? 4 : 5;
            const int pt = lane >> lg, sub = lane - (pt << lg);
            const int k0 = (M2 * sub) >> lg, k1 = (M2 * (sub + 1)) >> lg;
            __syncwarp();
            {
                const int e = min(pt, cnt - 1), at = f ? e : kMciList - 1 - e;
                const float4 v = w.Lp[at];
                const int u = w.Lu[at] * MS;
                const f32x2 da = dup2(v.y), db = dup2(v.z);
                const auto lp = [&](int k) {
                    const float4 x = Qa[u + k];
                    const float2 y = Qb[u + k];
                    return fma2(pack2(y.x, y.y), db, fma2(pack2(x.z, x.w), da, pack2(x.x, x.y)));
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
            if (lane < nl[f]) {                          // at most 31 stay
                w.Lp[at] = w.Lp[at + step];
                w.Lu[at] = w.Lu[at + step];
            }
            __syncwarp();
        };
        for (int t0 = item.piece0; t0 < item.piece1; t0 += blockDim.x) {
            const int nv = cell_round(cr, t0, item.piece1, n, i, rel, hb, pd, qp.dbg);
            int v = nv * warp / nw, cs = -1;                     // this warp's cells; next F_c channel of v
            const int v1 = nv * (warp + 1) / nw;
            while (v < v1) {
                // the next cells and F_c channels, in order
                int ncc = 0, nu = 0;
                while (v < v1 && ncc < GC && nu < kMciUnits) {
                    const int4 cl = cr.cell[v];
                    const int c0 = cs < 0 ? cl.z : cs, c1 = min(cl.w, c0 + kMciUnits - nu - 1);
                    if (nu > 0 && c1 < cl.w) break;              // whole cells while they fit
                    if (lane == 0) w.cell[ncc] = make_int4(cl.x | cl.y << 16, c0, c1, nu);
                    if (lane <= c1 - c0) w.unit[nu + lane] = make_int2(ncc, c0 + lane);
                    nu += c1 - c0 + 1;
                    ++ncc;
                    cs = c1 < cl.w ? c1 + 1 : -1;
                    v += c1 < cl.w ? 0 : 1;
                }
                __syncwarp();
                // step rows: ln p at da = db = 0 of the cell with F_c in channel c, dc
                // = da + db + D
#pragma unroll 1
                for (int u = 0; u < nu; ++u) {
                    const int2 un = w.unit[u];
                    const int ab = w.cell[un.x].x, a = ab & 0xffff, b = ab >> 16;
                    const float D = (rel[a] + rel[b]) - rel[un.y];
                    const float4 *Ta = T + a * M2, *Tb = T + b * M2, *Tc = T + un.y * M2, *Ti = T + i * M2;
                    for (int k = lane; k < M2; k += 32) {
                        const float4 ta = Ta[k], tb = Tb[k], ti = Ti[k], tc = Tc[k];
                        float4 q = make_float4(fmaf(tc.z, D, (ta.x + tb.x) + (tc.x - ti.x)),
                                               fmaf(tc.w, D, (ta.y + tb.y) + (tc.y - ti.y)), ta.z + tc.z, ta.w + tc.w);
                        if (2 * k + 1 >= M) q.y = -1000.0f;
                        Qa[u * MS + k] = q;
                        Qb[u * MS + k] = make_float2(tb.z + tc.z, tb.w + tc.w);
                    }
                }
                // grid rows
                for (int e = lane; e < ncc * G; e += 32) {
                    const int cc = (int)(((float)e + 0.5f) * inv_G), r = e - cc * G;
                    const int4 cl = w.cell[cc];
                    const int a = cl.x & 0xffff, b = cl.x >> 16;
                    w.row[e] = mci_row(fabsf(rel[a]), fabsf(rel[b]), hb[a], hb[b], eps, G, r,
                                       (a == b ? 1.0f : 2.0f) * (pd[a] * pd[b]));
                }
                __syncwarp();
                // the last turn, without points, sums what is left: the next group
                // replaces the step rows
#pragma unroll 1
                for (int q0 = 0, more = 1; more; q0 += 32) {
                    const int q = q0 + lane;
                    more = q0 < ncc * G * G;
                    int cls = -1, ci = -1, un = 0;
                    float phi = 0.0f, da = 0.0f, db = 0.0f, W = 0.0f;
                    if (q < ncc * G * G) {
                        const int rr = (int)(((float)q + 0.5f) * inv_G), j = q - rr * G;
                        const float4 o = w.row[rr];
                        if (o.w != 0.0f) {
                            const int4 cl = w.cell[(int)(((float)rr + 0.5f) * inv_G)];
                            const float ra = rel[cl.x & 0xffff], rb = rel[cl.x >> 16];
                            const float2 f = mci_point(o, ra, rb, j, G);
                            const float u = f.x + f.y;
                            for (int c = cl.y; c <= cl.z; ++c)
                                if (rel[c] - hb[c] <= u && u < rel[c] + hb[c]) ci = c;
                            if (ci >= 0) {
                                W = o.w * pd[ci];
                                da = f.x - ra;
                                db = f.y - rb;
                                un = cl.w + (ci - cl.y);
                                phi = ph.at<false>(f.x, f.y);
                                if (W != 0.0f) cls = fabsf(phi) <= phi_direct ? 0 : 1;
                            }
                        }
                    }
#pragma unroll
                    for (int f = 0; f < 2; ++f) {
                        const unsigned m = __ballot_sync(0xffffffffu, cls == f);
                        if (cls == f) {
                            const int e = nl[f] + __popc(m & lt_mask), at = f ? e : kMciList - 1 - e;
                            w.Lp[at] = make_float4(phi, da, db, W);
                            w.Lu[at] = un;
                        }
                        nl[f] += __popc(m);
                        if (nl[f] >= (more ? 32 : 1)) flush(f);
                    }
                }
            }
        }
        const double tot = block_sum_d((double)sum - (double)comp, scratch);
        if (threadIdx.x == 0) qp.partial[it] = tot;
    }
}

// Plain FP64 reference kernel: every step reads the profile rows of a, b, c
// and the CUT from the FP64 tables; the z-sum by zsum_f64.
__global__ void __launch_bounds__(256) k_quad_mci_f64_tab(QuadParams qp)
{
    extern __shared__ double2 smem_d2[];
    const int M = qp.n_steps, G = qp.G;
    double2 *sz = smem_d2;                 // [M] {z_m, dz_m}
    double *sti = reinterpret_cast<double *>(sz + M);   // [M] a_i(m) of the item's CUT
    __shared__ double scratch[32];
    __shared__ int s_item;

    for (int m = threadIdx.x; m < M; m += blockDim.x) sz[m] = qp.zs_d[m];
    const double phi_f64 = kF64Direct / qp.dz_max;
    const double c3 = kPi * qp.beta3;
    const double c4 = 2.0 * kPi * kPi / 3.0 * qp.beta4;

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
        const double2 *T = qp.ab + (size_t)poff * M;
        for (int m = threadIdx.x; m < M; m += blockDim.x) sti[m] = T[(size_t)i * M + m].x;
        __syncthreads();
        const double *fr = qp.ch_frel + coff;
        const double *Bc = qp.ch_B + coff;
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
            const double2 *Ta = T + (size_t)a * M, *Tb = T + (size_t)b * M;
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
                const double da = f1 - ra, db = f2 - rb, dc = u - (fr[c] - fi);
                const double br = qp.beta2 + c3 * (u + 2.0 * fi) +
                                  c4 * (f1 * f1 + 1.5 * f1 * f2 + 3.0 * fi * u + f2 * f2 + 3.0 * fi * fi);
                const double phi = -4.0 * kPi * kPi * f1 * f2 * br;
                const double2 *Tc = T + (size_t)c * M;
                const double S2 = zsum_f64(phi, phi_f64, sz, M, [&](int m) {
                    const double2 ta = Ta[m], tb = Tb[m], tc = Tc[m];
                    return exp(0.5 * (ta.x + tb.x + tc.x - sti[m] + ta.y * da + tb.y * db + tc.y * dc));
                });
                sum += w * W * S2 * array_factor_d(phi, qp);
            }
        }
        const double tot = block_sum_d(sum, scratch);
        if (threadIdx.x == 0) qp.partial[it] = tot;
    }
}

size_t quad_mci_tab_smem_bytes(int precision, int n_steps, int n_max, int G, int block)
{
    if (precision == 0)
        return (size_t)step_pairs(n_steps) * 32 + mci_warp_bytes(n_steps) * (block / 32) +
               (size_t)n_max * 2 * sizeof(float);
    return (size_t)n_steps * (sizeof(double2) + sizeof(double));
}

// Warps of a block: as many of the asked ones as shared memory holds (0: none)
int quad_mci_tab_block(int n_steps, int n_max, int G, int block)
{
    while (block > 0 && quad_mci_tab_smem_bytes(0, n_steps, n_max, G, block) > 200 * 1024) block -= 32;
    return block;
}

static void *mci_tab_fn(int precision)
{
    return precision == 0 ? (void *)k_quad_mci_f32_tab : (void *)k_quad_mci_f64_tab;
}

int quad_mci_tab_blocks_per_sm(int precision, int n_steps, int n_max, int G, int block)
{
    int nb = 0;
    const size_t smem = quad_mci_tab_smem_bytes(precision, n_steps, n_max, G, block);
    void *fn = mci_tab_fn(precision);
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, block, smem);
    return nb > 0 ? nb : 1;
}

cudaError_t launch_tab_half_log2(const TabHalfParams &hp, int n_prof, int max_n, int n_sms, cudaStream_t st)
{
    const int grid = std::max(1, std::min((max_n * step_pairs(hp.n_steps) + 255) / 256, 4 * n_sms));
    k_tab_half_log2<<<dim3(grid, n_prof), 256, 0, st>>>(hp);
    return cudaGetLastError();
}

cudaError_t launch_quad_mci_tab(const QuadParams &qp, int precision, int grid, int block, cudaStream_t st)
{
    const size_t smem = quad_mci_tab_smem_bytes(precision, qp.n_steps, qp.mci_n_max, qp.G, block);
    void *fn = mci_tab_fn(precision);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    QuadParams q = qp;
    void *args[] = {&q};
    return cudaLaunchKernel(fn, dim3(grid), dim3(block), args, smem, st);
}

}  // namespace isrs
