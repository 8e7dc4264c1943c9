// Cell decoding of the multi-channel-interference (MCI) grid, shared by the
// MCI quadrature and its adjoint: a work item is a range of cells (a, b),
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

// index of the channel containing offset u from the CUT, or -1
// (lo[c] = rel[c] - hb[c] ascending, channels disjoint)
template <typename T>
__device__ __forceinline__ int channel_of(const T *rel, const T *hb, int n, T u)
{
    int lo = 0, hi = n - 1, c = -1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        if (rel[mid] - hb[mid] <= u) {
            c = mid;
            lo = mid + 1;
        } else {
            hi = mid - 1;
        }
    }
    return (c >= 0 && u < rel[c] + hb[c]) ? c : -1;
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

}  // namespace isrs
