// Cells and grid points of the multi-channel-interference (MCI) grid: a work item is a range of cells (a, b),
// a <= b, a, b != CUT, in triangular order over the other N - 1 channels.
#pragma once
#include <cuda_runtime.h>

#include "isrs_debug.cuh"

namespace isrs {

// (a', b') of triangular index t over n2 channels: rows a' hold n2 - a'
// pairs starting at S(a') = a' (2 n2 - a' + 1) / 2.
__device__ __forceinline__ void tri_decode(int t, int n2, int &ap, int &bp)
{
    const float q = 2.0f * n2 + 1.0f;
    int a = (int)floorf(0.5f * (q - sqrtf(fmaxf(q * q - 8.0f * (float)t, 0.0f))));
    a = max(0, min(a, n2 - 1));
    while (a > 0 && a * (2 * n2 - a + 1) / 2 > t) --a;
    while (a + 1 < n2 && (a + 1) * (2 * n2 - a) / 2 <= t) ++a;
    ap = a;
    bp = a + (t - a * (2 * n2 - a + 1) / 2);
}

// The cells of one round of a block (blockDim cells from t0, one per thread) whose
// F_c can fall in a channel, compacted in order: {a, b, first and last channel}.
struct CellRound {
    int4 cell[256];
    int cnt[8];
};

// Called by every thread; ends with a barrier.  Returns the number of cells.  The
// test is a little wider than the cell, its points decide; 42 % of the cells of
// the 557-ch plan (68 % of a random 295-slot subset) drop out here, and dealing the
// rest to the warps in equal runs keeps them level.
__device__ __forceinline__ int cell_round(CellRound &cr, int t0, int t1, int n, int i, const float *rel,
                                          const float *hb, const float *pd, unsigned *dbg)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int a = 0, b = 0, c0 = 0, c1 = -1;
    if (t0 + (int)threadIdx.x < t1) {
        tri_decode(t0 + threadIdx.x, n - 1, a, b);
        a = dbg_clamp(a + (a >= i), n, kDbgCell, dbg);
        b = dbg_clamp(b + (b >= i), n, kDbgCell, dbg);
        if (pd[a] * pd[b] != 0.0f) {
            const float uc = rel[a] + rel[b], r = 1.0001f * (hb[a] + hb[b]) + 1e-5f * fabsf(uc) + 1e-6f;
            int hi = n;                                  // first channel ending above uc - r
            while (c0 < hi) {
                const int m = (c0 + hi) >> 1;
                if (rel[m] + hb[m] > uc - r) hi = m;
                else c0 = m + 1;
            }
            c1 = c0 - 1;
            while (c1 + 1 < n && rel[c1 + 1] - hb[c1 + 1] <= uc + r) ++c1;
        }
    }
    const unsigned m = __ballot_sync(0xffffffffu, c1 >= c0);
    __syncthreads();                                     // the previous round's cells are no longer read
    if (lane == 0) cr.cnt[warp] = __popc(m);
    __syncthreads();
    int off = 0, tot = 0;
    for (int w = 0; w < nw; ++w) {
        off += w < warp ? cr.cnt[w] : 0;
        tot += cr.cnt[w];
    }
    if (c1 >= c0) cr.cell[off + __popc(m & ((1u << lane) - 1u))] = make_int4(a, b, c0, c1);
    __syncthreads();
    return tot;
}

// Row r of a cell's hyperbolic grid (ra, rb: |f_a - f_i|, |f_b - f_i|; P: the
// powers' product with the mirror weight): {xc, yc, du2, weight}, 0 if empty.
__device__ __forceinline__ float4 mci_row(float ra, float rb, float hba, float hbb, float eps, int G, int r, float P)
{
    const float xlo = ra - hba, xhi = ra + hba;
    const float ylo = rb - hbb, yhi = rb + hbb;
    const float u1hi = xhi * yhi;
    const float llo = logf(fmaxf(xlo * ylo, eps * u1hi));
    const float ds = (logf(u1hi) - llo) / (float)G;
    const float u1 = expf(fmaf((float)r + 0.5f, ds, llo));
    const float ymin = fmaxf(ylo, u1 / xhi), ymax = fminf(yhi, u1 / xlo);
    float4 o = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (ymax > ymin) {
        o.z = log1pf((ymax - ymin) / ymin) / (float)G;
        o.y = sqrtf(ymin * ymax);
        o.x = u1 / o.y;
        o.w = u1 * ds * o.z * P;
    }
    return o;
}

// f1 and f2 at column j of a row (sa, sb: f_a - f_i, f_b - f_i)
__device__ __forceinline__ float2 mci_point(const float4 &o, float sa, float sb, int j, int G)
{
    const float d = ((float)j + 0.5f - 0.5f * (float)G) * o.z;
    const float ex = expf(d);
    const float s1 = sa > 0.0f ? 1.0f : -1.0f, s2 = sb > 0.0f ? 1.0f : -1.0f;
    return make_float2(s1 * (o.x * ex), s2 * (o.y * __frcp_rn(ex)));
}

// phi (Eq. phi) of a point from its FP32 f1 and f2.  The bracket is a small
// difference of large terms near the zero-dispersion wavelength: the rounding of a far
// cell's phi there is radians of |phi| L, the phase is a sample of its rounding, and a
// multiply-add fused elsewhere moved eta by up to 2.1e-4 (404 channels, 10 spans) and
// by 7e-5 between the forward and the adjoint of one plan.  So every operation is
// written with its rounding, in one place for all kernels; what a compiler makes of the
// code around it no longer shows in the result.  Fused: the last term of the sum as a
// multiply-add (closed-form profile) or rounded by itself (Raman ODE): the orders these
// results have always had.
struct MciPhase {
    float b2, c3, c4, fi;
    template <bool Fused>
    __device__ __forceinline__ float at(float f1, float f2) const
    {
        const float u = __fadd_rn(f1, f2), fi3 = __fmul_rn(3.0f, fi);
        float q = __fmaf_rn(f1, f1, __fmul_rn(__fmul_rn(1.5f, f1), f2));
        q = __fmaf_rn(f2, f2, __fmaf_rn(fi3, u, q));
        q = Fused ? __fmaf_rn(fi3, fi, q) : __fadd_rn(q, __fmul_rn(fi3, fi));
        const float br = __fmaf_rn(c4, q, __fmaf_rn(c3, __fmaf_rn(2.0f, fi, u), b2));
        return __fmul_rn(__fmul_rn(__fmul_rn(-39.4784176f, f1), f2), br);     // -4 pi^2 f1 f2
    }
};

}  // namespace isrs
