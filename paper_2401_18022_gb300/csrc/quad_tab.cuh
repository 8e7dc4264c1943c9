// Step rows of the tabulated (Raman-ODE) profile for the warp-per-piece
// quadratures.  Inside piece (a, b) of CUT i with F_c in candidate c,
//   log2 p_m = A(m) + Sl(m) dl + Sd(m) dd,
//   A = (a_a + a_b + a_c - a_i + b_c D) / 2,  D = f_a + f_b - f_i - f_c,
//   S = (b_a + b_c) / 2 or (b_b + b_c) / 2 (log2 units),
// dl, dd the offsets of F_a, F_b inside their channels, the longer axis of the
// piece first (quad_nodes.cuh may swap a and b).
#pragma once
#include <cuda_runtime.h>

#include "quad_nodes.cuh"

namespace isrs {

struct TabPiece {
    const double2 *Tl, *Td, *Ti;    // {a, b} of the longer axis's channel, the other, the CUT
    const double2 *T;               // ... of channel 0
    double Dl;                      // f_a + f_b - f_i - f_ref ... minus f_c gives D
    float ol, od;                   // dl, dd at the piece's corner
};

__device__ __forceinline__ TabPiece tab_piece(const QuadParams &qp, const DevPiece &pc, int prof, bool sw)
{
    TabPiece t;
    const int coff = qp.plan_ch_off[pc.plan], M = qp.n_steps;
    t.T = qp.ab + (size_t)qp.prof_ch_off[prof] * M;
    const int cl = sw ? pc.b : pc.a, cd = sw ? pc.a : pc.b;
    t.Tl = t.T + (size_t)cl * M;
    t.Td = t.T + (size_t)cd * M;
    t.Ti = t.T + (size_t)pc.cut * M;
    const double fi = qp.ch_frel[coff + pc.cut], fl = qp.ch_frel[coff + cl], fd = qp.ch_frel[coff + cd];
    const double sl = pc.flags & (sw ? 2 : 1) ? -1.0 : 1.0, sd = pc.flags & (sw ? 1 : 2) ? -1.0 : 1.0;
    t.Dl = (fl + fd) - fi;
    t.ol = (float)((fi - fl) + sl * (sw ? pc.yhi : pc.xhi));
    t.od = (float)((fi - fd) + sd * (sw ? pc.xhi : pc.yhi));
    return t;
}

// Row of step m for candidate channel c (f_c - f_ref = fc)
__device__ __forceinline__ float4 tab_row(const TabPiece &t, int c, double fc, int m, int M)
{
    const double2 l = t.Tl[m], d = t.Td[m], i = t.Ti[m], k = t.T[(size_t)c * M + m];
    const double A = (0.5 * kLog2e) * fma(k.y, t.Dl - fc, (l.x + d.x) + (k.x - i.x));
    const float h = (float)(0.5 * kLog2e), kb = (float)k.y;
    return make_float4((float)A, h * ((float)l.y + kb), h * ((float)d.y + kb), 0.0f);
}

}  // namespace isrs
