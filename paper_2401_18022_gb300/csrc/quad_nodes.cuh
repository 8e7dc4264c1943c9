// Row sums of the hyperbolic grid from a few nodes (App. A, Eqs. q1..q4).
//
// Along one grid row upsilon1 = |f1||f2| is constant, so the phase of Eq. phi,
// F_c and the power profile of Eq. pk depend on the point only through
// u = F_c - f_i, a smooth function of the column index j.  Inside one F_c
// channel the row's points are a run of N consecutive columns, and their sum
//   sum_{j = j0}^{j0 + N - 1} f(j)
// is the integral of f against the discrete uniform measure on N points.  The
// Gauss rule of that measure (its orthogonal polynomials are the discrete
// Chebyshev polynomials, Gautschi, "Orthogonal Polynomials: Computation and
// Approximation", 2004, Sec. 1.5) with n nodes reproduces the sum exactly for
// every polynomial of degree 2 n - 1.  |S|^2 is band limited along the row
// (|d phi| L per half run, A below), so its Chebyshev coefficients vanish
// faster than exponentially past degree ~A and n a little above A / 2 gives
// the same Riemann sum: it is a regrouping of the sum over the G points, not
// another grid.  In 64 bits Sigma is within 1e-8 on the plans of this repository
// and within 6e-8 on random plans around the zero-dispersion wavelength (up to 100
// spans, 16 to 300 rows, eps_v1 up to 0.05); the FP32 z-sums carry 2e-7.  The rule
// holds for the adjoint's bucket terms too, which have the same band limit.
//
// The rows are uniform in ln upsilon1, so the row sums of a block of low rows
// (one F_c channel, |phi| L small) are smooth in the row index as well, and the
// same rules take the block's sum from a few rows at real-valued indices.
//
// Why: the quadratures are bound by the z-sums (112 steps per point).  A piece
// of the 589-channel plan has 65,536 points at G = 256 (4,096 at G = 64) and
// takes about 1,000 (250) nodes.
//
// Coordinates are carried relative to a corner of the piece, U = s1 xhi +
// s2 yhi, so that an FP32 point is located to ~1e-8 THz also where F_c - f_i
// is tens of THz, and phi is split per row into its value at the row's centre
// (a float-float pair) and an increment quadratic in u.
//
// FP64 is used once per piece (node_geo, one warp instruction for several values
// where that goes): an SM takes 16 clocks for an FP64 warp instruction, and with
// ~30 of them per row and row test the set-up was bound by that pipe (half of a
// 589-channel call at G = 64).
//
// One warp works on one piece: lane = row while rows are set up and their runs
// listed, lane = node (or half-warp = node) afterwards.  Blocks working on one
// piece together spent a third of their issue slots at barriers, because the
// set-up is a chain of short FP64 steps.
#pragma once
#include <cuda_runtime.h>

#include "quad_common.cuh"

namespace isrs {

// Node counts of the rules: 2..8, 10, 12 .. 20, 24, 28, 32, 40, 48.  One table
// of {t, weight} per run length N <= kGaussMaxN and node count; node k lies at
// column centre + t N / 2.
constexpr int kGaussMaxN = 256;
constexpr int kGaussMaxNodes = 48;
constexpr int kGaussMenu = 18;
constexpr int kGaussPerN = 297;                        // nodes of all rules of one N
constexpr int kGaussEntries = kGaussMaxN * kGaussPerN;
constexpr int kRowRuns = 4;                            // runs of a row listed at a time
// behind the rules: 2^(-j / kExp2Entries) as float-float pairs (node_row)
constexpr int kExp2Entries = 256;

__host__ __device__ constexpr int gauss_nodes(int k)
{
    return k <= 6 ? 2 + k : k <= 12 ? 2 * (k - 2) : k <= 15 ? 20 + 4 * (k - 12) : 32 + 8 * (k - 15);
}

__host__ __device__ constexpr int gauss_offset(int k)
{
    return k <= 6 ? 2 * k + k * (k - 1) / 2 : k <= 12 ? k * (k - 5) + 21
         : k <= 15 ? 125 + 24 * (k - 13) + 2 * (k - 13) * (k - 14) : 209 + 40 * (k - 16);
}

// smallest rule with at least `need` nodes (need <= kGaussMaxNodes)
__host__ __device__ inline int gauss_pick(int need)
{
    return need <= 2 ? 0 : need <= 8 ? need - 2 : need <= 20 ? 6 + (need - 7) / 2
         : need <= 32 ? 12 + (need - 17) / 4 : 15 + (need - 25) / 8;
}

// Nodes that give a run's sum: A bounds the phase swing of |S|^2 over half the
// run, D its half-length in upsilon2 (the map from column to u is exp-like).
// Measured need over the runs of the 589-ch, O-band and 10-span plans (A up to
// 670, D up to 11.5): to 3e-8 of the run's sum, or of the piece's where the run
// is a fast row (|S|^2 falls as 1/phi^2, so a row at |phi| L = 6 t weighs 1/t),
// 2 n - A stays below 4 at A < 0.05, 8 at 0.3, 9.3 at 3, 12.5 at 30, 13.7 at 100.
// A fast row by itself may be further off (1e-5 of its own sum at A = 10 to 20 and 10
// spans); what counts is Sigma.
__host__ __device__ inline int gauss_need(float A, float D)
{
    const float two_n = A + 4.0f + 4.2f * A / (A + 0.35f) + 0.6f * sqrtf(A) + 1.4f * D;
    return two_n < 8192.0f ? (int)ceilf(0.5f * two_n) : 4096;
}

// Nodes for the sum of a block of rows (row_blocks).  Along a row only |S|^2 varies;
// over a block the rows' weight is exp-like, e^{D t}, and wants 4 + 6 sqrt(D) = 2 n by
// itself (e^{D t} and e^{D t} (c - t) to 1e-8, D up to 20, N from 16 to 256).  With
// gauss_need a block of every row (three 32 GBaud channels at 1310 nm, eps_v1 1e-3, D
// 3.4) was off by 3.6e-5 of Sigma.  part: rows up to kBlkPhiLow below others, a few per
// cent of the piece, where the weight alone counts.  Over 640 random plans (16 to 200
// rows, 1 to 100 spans, either cell set) Sigma is within 6e-8 now, all of it the rows'
// part, for 2 % more nodes and of the time (589 channels, G 256: 43.9 -> 44.9 ms; 12
// profiles, G 64: 77.1 -> 79.0; 45.8 and 82.0 if the low part follows the swing too).
__host__ __device__ inline int block_need(float A, float D, bool part)
{
    const float two_n = 4.0f + 6.0f * sqrtf(D) + (part ? 0.0f : A + 4.2f * A / (A + 0.35f) + 0.6f * sqrtf(A));
    return two_n < 8192.0f ? (int)ceilf(0.5f * two_n) : 4096;
}

constexpr int kBlkMax = 18;              // row blocks of a piece at most (kMaxG / 256 + 2)
constexpr float kBlkPhiL = kSmallPhiL;   // |phi| n_spans L up to which rows join a block ...
constexpr float kBlkPhiLow = 0.15f;      // ... and up to which they join the low ones

// One piece's geometry, |f1| the longer axis (f1 and f2 enter symmetrically,
// so swapping them only reverses the columns).
struct PieceGeo {
    float2 vC;                  // -4 pi^2 f1 f2 at the corner, float-float
    float2 br0;                 // bracket of Eq. phi: br0 + br1 u + c4 u^2 - c4/2 f1 f2, u from the corner
    float2 ds2;                 // row pitch in log2 upsilon1
    float2 u1hi;                // xhi yhi, float-float
    float2 k[3];                // of a row's centre, float-float: yhi / xhi, ylo / xlo and the root of
                                // xlo xhi (R < Rb) or ylo yhi
    float br1, c4;
    float ds;                   // row pitch in ln upsilon1
    float xhi, yhi;             // corner of the piece
    float s1, s2;               // signs of f1, f2
    float R, Rb;                // ln(xhi / xlo), ln(yhi / ylo) (1e30 where the lower limit is 0)
    float off;                  // bound of |row_u - point_u|
    float band;                 // n_spans L: phase swing per |d phi|
    float tilt;                 // bound of |d ln p / dF|
    float Fc0, Fi;              // F_c - f_ref and F_c - f_i at the corner
    float wab, at_ab, mult;     // P_a P_b / (B_a B_b), attenuation part of ln p, mirror weight
    bool sw;                    // the longer axis belongs to F_b
    int nc;                     // F_c candidates: edges from the CUT, P/B, half attenuation
    float lo[kMaxCand], hi[kMaxCand], pd[kMaxCand], hat[kMaxCand];
};

// One grid row: centre, column pitch, weight; f1 - s1 xhi and f2 - s2 yhi at
// the centre, and phi there as a float-float pair: |S|^2 turns through hundreds
// of radians of phi L that the rows sample far apart, so an FP32 relative error
// of a whole row's phase would show in the sum (errors of single points
// average out along the row).
struct __align__(16) NodeRow {
    float xc, yc, du2, w;
    float x0, y0, phi0, phi0_lo;
};

// A run of N columns of one row inside one F_c candidate, with its rule.
struct __align__(16) NodeRun {
    float jc;                   // centre column, from the row's centre
    float half;                 // N / 2
    int toff;                   // first entry of the rule; -1: the N columns themselves
    unsigned id;                // first slot of the warp's rows | candidate << 16 | nodes << 24
};

struct RowBlock {
    int unit0, r0, N, toff;     // first unit, first row, rows, rule (-1: every row)
};

template <int Cap>
struct WarpNodes {
    NodeRow row[32];
    NodeRun run[32 * kRowRuns];         // [row][run]
    unsigned char of[Cap];              // run of each slot of the chunk
    RowBlock blk[kBlkMax];
    PieceGeo geo;
};

// float-float product, quotient and square root (~2^-45; a, b > 0)
__device__ __forceinline__ float2 ff_sum(float a, float b)            // |a| >= |b|
{
    const float h = __fadd_rn(a, b);
    return make_float2(h, __fadd_rn(b, -__fadd_rn(h, -a)));
}

__device__ __forceinline__ float2 ff_mul(float2 a, float2 b)
{
    const float h = __fmul_rn(a.x, b.x);
    return ff_sum(h, fmaf(a.x, b.x, -h) + fmaf(a.x, b.y, a.y * b.x));
}

__device__ __forceinline__ float2 ff_div(float2 a, float2 b)
{
    const float r = __fdividef(1.0f, b.x), q = __fmul_rn(a.x, r);
    return ff_sum(q, (fmaf(-q, b.x, a.x) + fmaf(-q, b.y, a.y)) * r);
}

__device__ __forceinline__ float2 ff_sqrt(float2 a)
{
    const float r = rsqrtf(a.x), q = __fmul_rn(a.x, r);
    return ff_sum(q, (fmaf(-q, q, a.x) + a.y) * (0.5f * r));
}

// The piece's geometry (whole warp; the caller syncs the warp).  sw: the
// longer axis belongs to F_b.
__device__ __forceinline__ bool node_geo(const QuadParams &qp, const DevPiece &pc, int prof, float at_scale,
                                         const float *pdv, float tilt, PieceGeo &g)
{
    const int lane = threadIdx.x & 31;
    const bool sw = pc.yhi > pc.xhi;
    const double xhi = sw ? pc.yhi : pc.xhi, yhi = sw ? pc.xhi : pc.yhi;
    const bool n1 = pc.flags & (sw ? 2 : 1), n2 = pc.flags & (sw ? 1 : 2);
    const int coff = qp.plan_ch_off[pc.plan], poff = qp.prof_ch_off[prof];
    const double fi = qp.ch_frel[coff + pc.cut];
    const double U = (n1 ? -xhi : xhi) + (n2 ? -yhi : yhi);
    const int nc = min(pc.c_hi - pc.c_lo + 1, kMaxCand);
    if (lane < nc) {
        const double fc = qp.ch_frel[coff + pc.c_lo + lane], hb = 0.5 * qp.ch_B[coff + pc.c_lo + lane];
        g.lo[lane] = (float)((fc - hb) - fi);
        g.hi[lane] = (float)((fc + hb) - fi);
        g.pd[lane] = pdv[poff + pc.c_lo + lane];
        g.hat[lane] = 0.5f * (float)qp.ch_alpha[coff + pc.c_lo + lane] * at_scale;
    }
    // lane k takes the k-th value apart
    const double t = 3.0 * qp.c4 * fi, b1 = qp.c3 + t;
    const double b0 = fma(fi, qp.c3 + b1, qp.beta2), u1 = xhi * yhi;
    double v = u1;
    if (lane == 1) v = (n1 == n2 ? -4.0 : 4.0) * kPi * kPi * u1;
    if (lane == 2) v = fma(U, fma(qp.c4, U, b1), b0);
    if (lane == 3) v = fma(2.0 * qp.c4, U, b1);
    if (lane == 4) v = fi + U;
    if (lane == 8) v = U;
    if (lane == 5) v = xhi;
    if (lane == 6) v = yhi;
    if (lane == 9) v = sw ? pc.ylo : pc.xlo;
    if (lane == 10) v = sw ? pc.xlo : pc.ylo;
    if (lane == 7)
        v = 0.5 * (qp.ch_alpha[coff + pc.a] + qp.ch_alpha[coff + pc.b] - qp.ch_alpha[coff + pc.cut]);
    const float vh = (float)v, vl = (float)(v - (double)vh);
    if (lane == 1) g.vC = make_float2(vh, vl);
    if (lane == 2) g.br0 = make_float2(vh, vl);
    if (lane == 3) g.br1 = vh;
    if (lane == 4) g.Fc0 = vh;
    if (lane == 8) g.Fi = vh;
    if (lane == 5) g.xhi = vh;
    if (lane == 6) g.yhi = vh;
    if (lane == 7) g.at_ab = vh * at_scale;
    // lanes 0..2: yhi / xhi, ylo / xlo, the mean of the limits of the shorter range (what
    // a lower limit of 0 leaves undefined no row takes)
    const bool cx = (sw ? pc.lny : pc.lnx) < (sw ? pc.lnx : pc.lny);
    const int la = lane == 0 ? 6 : lane == 1 ? 10 : cx ? 5 : 6, lb = lane == 0 ? 5 : lane == 1 || cx ? 9 : 10;
    const float2 ka = make_float2(__shfl_sync(0xffffffffu, vh, la), __shfl_sync(0xffffffffu, vl, la));
    const float2 kb = make_float2(__shfl_sync(0xffffffffu, vh, lb), __shfl_sync(0xffffffffu, vl, lb));
    if (lane < 3) g.k[lane] = lane == 2 ? ff_sqrt(ff_mul(ka, kb)) : ff_div(ka, kb);
    if (lane == 0) {
        const float2 ds2 = pc.ds2;
        g.u1hi = make_float2(vh, vl);
        g.sw = sw;
        g.c4 = (float)qp.c4;
        g.ds2 = ds2;
        g.ds = fmaf(ds2.x, 0.693147182f, fmaf(ds2.x, -1.90465421e-9f, ds2.y * 0.693147182f));   // times ln 2
        g.s1 = n1 ? -1.0f : 1.0f;
        g.s2 = n2 ? -1.0f : 1.0f;
        g.R = sw ? pc.lny : pc.lnx;
        g.Rb = sw ? pc.lnx : pc.lny;
        // 2.4e-7 of |f1| and 3e-7 of |f2| by point_u's rounding, 6e-8 |d| by d's (|d| is at
        // most half the shorter range, 20 for any epsilon), as much again by row_u's
        g.off = 8e-7f * (float)(xhi + yhi) * (1.0f + fminf(20.0f, fminf(pc.lnx, pc.lny)));
        g.band = qp.L * (float)qp.n_spans;
        g.tilt = tilt;
        g.wab = pdv[poff + pc.a] * pdv[poff + pc.b];
        g.mult = pc.mult;
        g.nc = nc;
    }
    return sw;
}

// The row k + k_lo = G - 1/2 - r pitches below the corner (r real-valued in a
// block).  upsilon1 / (xhi yhi) = 2^-t, t = k ds2, is taken in FP32 pairs to ~1e-10
// relative: t = n + j / 256 + rest, a table of 2^(-j/256) and the Taylor series of
// 2^-rest - 1 (|rest| <= 1/512; to the third power, remainder below 2e-13).  In logarithms relative to the corner, l = ln(upsilon1 / (xhi yhi)), |f2| runs
// over [max(-Rb, l), min(0, l + R)] and the row's centre lies at ln(xc / xhi) =
// gx, ln(yc / yhi) = gy.  Returns which limits hold: bit 0 the one set by xhi,
// bit 1 by xlo (else by ylo, yhi); -1 for an empty row.
__device__ __forceinline__ int node_row(const PieceGeo &g, const float2 *gauss, int G, float k, float k_lo,
                                        NodeRow &o)
{
    const float t = k * g.ds2.x, tl = fmaf(k, g.ds2.x, -t) + fmaf(k, g.ds2.y, k_lo * g.ds2.x);
    const float mf = __fadd_rn(fmaf(t, (float)kExp2Entries, 12582912.0f), -12582912.0f);
    const float y = (fmaf(mf, -1.0f / kExp2Entries, t) + tl) * -0.6931471806f;
    const float q = fmaf(y * y, fmaf(y, 1.0f / 6.0f, 0.5f), y);
    const int mi = (int)mf, n = mi / kExp2Entries;
    const float2 T = __ldg(gauss + kGaussEntries + (mi & (kExp2Entries - 1)));
    const float eh = fmaf(T.x, q, T.x), el = fmaf(T.x, q, __fadd_rn(T.x, -eh)) + fmaf(T.y, q, T.y);
    const float sc = n < 127 ? __int_as_float((127 - n) << 23) : 0.0f;
    const float uh = __fmul_rn(g.u1hi.x, eh);
    const float ul = fmaf(g.u1hi.x, eh, -uh) + fmaf(g.u1hi.x, el, g.u1hi.y * eh);
    const float u1 = (uh + ul) * sc;
    const float l = -k * g.ds;
    const bool a = l > -g.Rb, b = l + g.R < 0.0f;
    const float D = a ? (b ? g.R : -l) : (b ? l + g.R + g.Rb : g.Rb);
    const float gx = a ? (b ? -0.5f * g.R : 0.5f * l) : (b ? 0.5f * (l + g.Rb - g.R) : l + 0.5f * g.Rb);
    const float gy = a ? (b ? l + 0.5f * g.R : 0.5f * l) : (b ? 0.5f * (l + g.R - g.Rb) : -0.5f * g.Rb);
    if (!(D > 0.0f) || u1 < 1e-37f) {
        o.xc = o.yc = o.du2 = o.w = o.x0 = o.y0 = o.phi0 = o.phi0_lo = 0.0f;
        return -1;
    }
    // The centre lies at |f2| = sqrt(ymin ymax): sqrt(u1 yhi / xhi), sqrt(u1 ylo / xlo), or
    // one of f1 and f2 is the mean of its limits.  Rounded once, for point_u.
    const bool mid = a == b;
    const float2 U = make_float2(uh * sc, ul * sc);
    const float2 p = mid ? g.k[2] : ff_sqrt(ff_mul(U, a ? g.k[0] : g.k[1]));
    const float qc = ff_div(U, p).x;
    o.xc = mid && a ? p.x : qc;
    o.yc = mid && a ? qc : p.x;
    const float rG = __fdividef(1.0f, (float)G), du2 = D * rG;
    o.du2 = fmaf(fmaf(-du2, (float)G, D), rG, du2);
    o.w = u1 * g.ds * o.du2;
    o.x0 = g.s1 * g.xhi * expm1f(gx);
    o.y0 = g.s2 * g.yhi * expm1f(gy);
    const float u0 = o.x0 + o.y0;
    const float db = fmaf(-0.5f * g.c4 * g.s1 * g.s2, u1, u0 * fmaf(g.c4, u0, g.br1));
    const float bh = __fadd_rn(g.br0.x, db), bb = __fadd_rn(bh, -g.br0.x);        // two-sum
    const float bl = __fadd_rn(__fadd_rn(g.br0.x, -__fadd_rn(bh, -bb)), __fadd_rn(db, -bb)) + g.br0.y;
    const float vh = g.vC.x * eh, vl = fmaf(g.vC.x, eh, -vh) + fmaf(g.vC.x, el, g.vC.y * eh);
    const float ph = vh * bh;
    o.phi0 = ph * sc;
    o.phi0_lo = (fmaf(vh, bh, -ph) + fmaf(vh, bl, vl * bh)) * sc;
    return (a ? 1 : 0) | (b ? 2 : 0);
}

// phi = phi0 + du (p1 + p2 du) along a row, du = u - u0
__device__ __forceinline__ void row_slopes(const PieceGeo &g, const NodeRow &o, float &p1, float &p2)
{
    const float cv = -39.47841760435743f * g.s1 * g.s2 * (o.xc * o.yc);      // -4 pi^2 f1 f2
    p1 = cv * fmaf(2.0f * g.c4, o.x0 + o.y0, g.br1);
    p2 = cv * g.c4;
}

// e^d - 1 and e^{-d} - 1, both to FP32 relative accuracy: cosh d - 1 +- sinh d
// by their Taylor series for |d| <= 0.6 (remainders below 2e-11), which covers all
// rows but those of the CUT's own cell.
__device__ __forceinline__ void expm1_pair(float d, float &ep, float &em)
{
    if (fabsf(d) <= 0.6f) {
        const float x = d * d;
        const float sh = d * fmaf(x, fmaf(x, fmaf(x, fmaf(x, 1.0f / 362880.0f, 1.0f / 5040.0f), 1.0f / 120.0f),
                                          1.0f / 6.0f), 1.0f);
        const float ch = x * fmaf(x, fmaf(x, fmaf(x, fmaf(x, 1.0f / 3628800.0f, 1.0f / 40320.0f), 1.0f / 720.0f),
                                          1.0f / 24.0f), 0.5f);
        ep = ch + sh;
        em = ch - sh;
        return;
    }
    const float E = expm1f(fabsf(d));
    const float En = __fdividef(-E, 1.0f + E);
    ep = d >= 0.0f ? E : En;
    em = d >= 0.0f ? En : E;
}

// u from the corner at d = upsilon2 - (row centre)
__device__ __forceinline__ float row_u(const PieceGeo &g, const NodeRow &o, float d)
{
    float ep, em;
    expm1_pair(d, ep, em);
    return (o.x0 + o.y0) + fmaf(g.s1 * o.xc, ep, g.s2 * o.yc * em);
}

// F_c - f_i at column j of a grid row, as the sum of the point's FP32 f1 and f2: what
// decides its F_c channel.  A point next to a channel's edge falls on the side where this
// rounding puts it (a few 1e-6 THz in the far cells).  From the corner's coordinates,
// which are finer, others fall otherwise, each worth up to 1e-3 of a channel's eta on a
// coarse grid: 148 neighbouring channels around the zero-dispersion wavelength at G 40
// came out 5.3e-5 (2-norm of eta) from the sum over single points, 8.3e-7 now.  So every
// factor is rounded as that sum rounds it: the row's centre and pitch once to FP32, e^d,
// its reciprocal, the products.  Costs 1 to 5 % of the time (589 channels, G 256: 44.9 ->
// 45.5 ms; 12 profiles, G 64: 79.7 -> 83.8, 81.8 with row_whole's ends in a loop); taking
// it only within g.off of an edge costs more (46.9 and 93.7), some row of a warp nearly
// always is.
__device__ __forceinline__ float point_u(const PieceGeo &g, const NodeRow &o, int G, int j)
{
    const float d = __fmul_rn((float)j + 0.5f - 0.5f * (float)G, o.du2);
    const float e = expf(g.sw ? -d : d), er = __frcp_rn(e);
    return __fadd_rn(g.s1 * __fmul_rn(o.xc, g.sw ? er : e), g.s2 * __fmul_rn(o.yc, g.sw ? e : er));
}

// first column of the row past |f1| = |f2|, where u turns if both have one sign
__device__ __forceinline__ int row_turn(const PieceGeo &g, const NodeRow &o, int G)
{
    if (g.s1 != g.s2) return 0;
    const float x = __fdividef(0.5f * __logf(__fdividef(o.yc, o.xc)), o.du2) + 0.5f * (float)G - 0.5f;
    return x > 0.0f ? (x < (float)G ? (int)ceilf(x) : G) : 0;
}

// The runs of one row in column order: f(candidate, j0, N).  On one half-open
// interval of columns u is monotone, so a candidate's columns are a run found
// by bisection.  whole: the one candidate that holds every column, or -1.
// (The loops of the set-up stay rolled: unrolled, a kernel's code is 94 KB and
// the warps, each at its own place in it, wait for instructions.)
template <typename F>
__device__ __forceinline__ void row_runs(const PieceGeo &g, const NodeRow &o, int G, int ca, int cb, int whole,
                                         const F &f)
{
    const auto u_at = [&](int j) { return point_u(g, o, G, j); };
    const int jm = whole >= 0 ? 0 : row_turn(g, o, G);
    if (whole >= 0) {
        ca = whole;
        cb = whole + 1;
    }
#pragma unroll 1
    for (int part = 0; part < 2; ++part) {
        const int ja = part == 0 ? 0 : jm, jb = part == 0 ? jm : G;
        if (jb <= ja) continue;
        const bool up = (g.s1 > 0.0f) == (part == 1 || g.s1 != g.s2);
        float ua = 0.0f, ub = 0.0f;
        if (whole < 0)
#pragma unroll 1
            for (int side = 0; side < 2; ++side) {
                ua = ub;
                ub = u_at(side == 0 ? ja : jb - 1);
            }
        // first column of [ja, jb) at or past edge e in the direction of travel (ja
        // is before it, jb - 1 at or past it or nothing is): the column a straight
        // line between the ends gives and a neighbour of it usually bracket it (u
        // is nearly linear on most rows), bisection does the rest
        const float slope = __fdividef((float)(jb - 1 - ja), ub - ua);
        const auto first = [&](float e) {
            int lo = ja + 1, hi = jb;
            int m = (int)fminf(fmaxf(ceilf((e - ua) * slope), 1.0f), (float)(jb - 1 - ja)) + ja;
#pragma unroll 1
            for (int it = 0; lo < hi; ++it) {
                const float u = m == jb - 1 ? ub : u_at(m);
                const bool past = up ? u >= e : u < e;
                if (past) hi = m;
                else lo = m + 1;
                m = it > 0 ? (lo + hi) >> 1 : past ? m - 1 : m + 1;
                m = max(lo, min(m, hi - 1));
            }
            return lo;
        };
#pragma unroll 1
        for (int q = ca; q < cb; ++q) {
            const int c = up ? q : ca + cb - 1 - q;
            const float lo = g.lo[c], hi = g.hi[c];
            int j0 = ja, j1 = jb;
            if (whole < 0) {
                if ((up ? ub : ua) < lo || (up ? ua : ub) >= hi) continue;
#pragma unroll 1
                for (int side = 0; side < 2; ++side) {            // entering edge, leaving edge
                    const float e = up == (side == 0) ? lo : hi;
                    const bool in = side == 0 ? (up ? ua >= e : ua < e) : (up ? ub < e : ub >= e);
                    const int j = in ? (side == 0 ? ja : jb) : first(e);
                    if (side == 0) j0 = j;
                    else j1 = j;
                }
            }
            if (j1 > j0) f(c, j0, j1 - j0);
        }
    }
}

// Bound of |du/dt| per column of a run's half-length, t in [-1, 1], and the
// phase swing it brings: du/dupsilon2 = f1 - f2 is monotone along the row, so it
// is largest at one of the ends.
__device__ __forceinline__ float row_swing(const PieceGeo &g, const NodeRow &o, int G)
{
    float p1, p2;
    row_slopes(g, o, p1, p2);
    const float E = expf(0.5f * (float)G * o.du2), Ei = __fdividef(1.0f, E);
    const float x = g.s1 * o.xc, y = g.s2 * o.yc;
    const float e = fmaxf(fabsf(x * E - y * Ei), fabsf(x * Ei - y * E)) * 0.5f * o.du2;
    return e * (g.band * (fabsf(p1) + 2.0f * fabsf(p2) * e * (float)G)) + (fabsf(x) + fabsf(y)) * E * o.du2 * g.tilt;
}

// A run cut into the parts one rule each covers: f(j0, N, n), n = N where the
// columns themselves are no more than the rule needs.  n <= kGaussMaxNodes: a
// part of a run that needs n > 48 nodes has (A + 1.4 D) / parts <= 48 and so
// needs at most 31, and a part of <= 48 columns takes at most its columns.
template <typename F>
__device__ __forceinline__ void run_parts(const PieceGeo &g, const NodeRow &o, int G, int j0, int N, const F &f)
{
    const float per = row_swing(g, o, G), hd = 0.5f * o.du2;
    int n = gauss_need(per * (float)N, hd * (float)N);
    int parts = 1;
    if (N > kGaussMaxNodes && (n > kGaussMaxNodes || N > kGaussMaxN)) {
        parts = max((N + kGaussMaxN - 1) / kGaussMaxN, (n + 23) / 24);
        parts = min(parts, (N + kGaussMaxNodes - 1) / kGaussMaxNodes);
    }
    int b = 0;
#pragma unroll 1
    for (int s = 0; s < parts; ++s) {
        const int a = b;
        b = parts == 1 ? N : N * (s + 1) / parts;
        const int Ns = b - a;
        if (parts > 1) n = gauss_need(per * (float)Ns, hd * (float)Ns);
        const int nn = n <= kGaussMaxNodes ? gauss_nodes(gauss_pick(n)) : Ns;
        f(j0 + a, Ns, nn < Ns ? nn : Ns);
    }
}

// The F_c candidate that holds every column of the row with room for point_u's rounding,
// or -1; ph: bound of |phi| band over the row's columns.
__device__ __forceinline__ int row_whole(const PieceGeo &g, const NodeRow &o, int G, float &ph)
{
    const float c0 = 0.5f - 0.5f * (float)G;
    const int jm = row_turn(g, o, G);
    float mn = 1e30f, mx = -1e30f;
    const int n = jm > 0 && jm < G ? 4 : 2;
#pragma unroll 1
    for (int k = 0; k < n; ++k) {                         // both ends, both sides of the turn
        const int j = k == 0 ? 0 : k == 1 ? G - 1 : jm + k - 3;
        const float u = row_u(g, o, ((float)j + c0) * o.du2);
        mn = fminf(mn, u);
        mx = fmaxf(mx, u);
    }
    float p1, p2;
    row_slopes(g, o, p1, p2);
    const float r = mx - mn;
    ph = g.band * (fabsf(o.phi0) + r * (fabsf(p1) + fabsf(p2) * r));
    mn = (mn + g.Fi) - g.off;
    mx = (mx + g.Fi) + g.off;
    int c = -1;
#pragma unroll 1
    for (int q = 0; q < g.nc; ++q)
        if (mn >= g.lo[q] && mx < g.hi[q]) c = q;
    return c;
}

// The blocks of low rows: the rows [0, R1) whose columns all lie in one
// candidate, with one set of limits and |phi| band <= kBlkPhiL, cut at |phi|
// band = kBlkPhiLow and into parts of kGaussMaxN rows.  Along t in [-1, 1] over
// N rows upsilon1 (so the weight and phi) is exp-like with D = N ds / 2.  phi is
// upsilon1 times the bracket of Eq. phi, and the bracket may vanish towards the block's
// last row (the (+,-) quadrant of a CUT near the zero-dispersion wavelength, where rows
// shrink to f1 = -f2): neither |phi| there nor the largest one bounds the swing then.
// q_last, the block's largest bracket at the last row's upsilon1, does: |phi| band of
// row r is below q_last e^{-(R1 - 1 - r) ds} and swings by at most q_last D.  (Rows of
// the CUT's own cell at 1310 nm, 96 GBaud, G 256, 20 spans: with |phi| of the last row
// 1.9e-5 of Sigma, with the largest 6.7e-7, with q_last 2.6e-8, 739 / 759 / 766 nodes.)
// Whole warp; writes ns.blk.
struct PieceBlocks {
    int units;                  // rows of the rules, all blocks
    int R1, nblk, cand;         // rows covered, blocks, their F_c candidate
};

template <int Cap>
__device__ __forceinline__ PieceBlocks row_blocks(WarpNodes<Cap> &ns, const float2 *gauss, int G)
{
    PieceBlocks pb = {0, 0, 0, -1};
    int &R1 = pb.R1, &nblk = pb.nblk, &cand = pb.cand, &units = pb.units;
    const PieceGeo &g = ns.geo;
    const int lane = threadIdx.x & 31;
    float q_max = 0.0f;              // largest |phi| band at the middle row's upsilon1
    const float k_mid = 0.5f * (float)G;
    // candidate and limits of row r (-1: not in one candidate), |phi| band
    const auto test = [&](int r, float &ph) {
        NodeRow o;
        const int lim = node_row(g, gauss, G, (float)(G - r) - 0.5f, 0.0f, o);
        ph = 0.0f;
        const int c = lim >= 0 ? row_whole(g, o, G, ph) : -1;
        return c >= 0 ? (c << 2 | lim) : -1;
    };
    // lanes take rows step apart; the first that fails bounds the next, finer
    // sweep.  A row between two that pass passes too: with both limits of |f2|
    // following upsilon1, or f1 and f2 of one sign, the ends of the row's u are
    // monotone in upsilon1; otherwise every row is tested.
    const int step = (G + 31) / 32;
    int key0 = -1;
#pragma unroll 1
    for (int r0 = -1; r0 < G;) {
        const bool coarse = r0 < 0;
        const int r = coarse ? lane * step : r0 + lane;
        float ph;
        const int key = test(min(r, G - 1), ph);
        if (coarse) {
            key0 = __shfl_sync(0xffffffffu, key, 0);
            if (key0 < 0 || !(__shfl_sync(0xffffffffu, ph, 0) <= kBlkPhiL)) return pb;
        }
        const bool ok = r < G && key == key0 && ph <= kBlkPhiL;
        const int bad = __ffs(~__ballot_sync(0xffffffffu, ok)) - 1;          // -1: none
        const int n = bad < 0 ? 32 : bad;
        if (coarse) {
            if ((key0 & 3) != 3 && g.s1 != g.s2) {
                r0 = 0;
                continue;
            }
            R1 = bad < 0 ? min(G, 31 * step + 1) : (bad - 1) * step + 1;
        } else {
            R1 += n;
        }
        // (between two rows tested the bracket lies between theirs)
        const float q = lane < n ? ph * ex2_approx(((float)(G - r) - 0.5f - k_mid) * g.ds2.x) : 0.0f;
        q_max = fmaxf(q_max, __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(q))));
        if (!coarse && n < 32) break;
        r0 = R1;
    }
    cand = key0 >> 2;
    const float q_last = q_max * ex2_approx((k_mid - (float)(G - R1) - 0.5f) * g.ds2.x);
    // rows from the block's top down to |phi| band = kBlkPhiLow
    const float tops = q_last > kBlkPhiLow ? ceilf(__fdividef(__logf(q_last / kBlkPhiLow), g.ds)) : 0.0f;
    const int top = (int)fminf(tops, (float)R1);
#pragma unroll 1
    for (int low = 1; low >= 0; --low) {
        const int n_rows = low ? R1 - top : top, parts = (n_rows + kGaussMaxN - 1) / kGaussMaxN;
#pragma unroll 1
        for (int s = 0; s < parts; ++s) {
            const int a = n_rows * s / parts, b = n_rows * (s + 1) / parts, N = b - a;
            const float D = 0.5f * (float)N * g.ds;
            const int need = block_need((low ? fminf(q_last, kBlkPhiLow) : q_last) * D, D, low && top > 0);
            const int n = need <= kGaussMaxNodes ? gauss_nodes(gauss_pick(need)) : N;
            if (lane == 0)
                ns.blk[nblk] = RowBlock{units, (low ? 0 : R1 - top) + a, N,
                                        n < N ? (N - 1) * kGaussPerN + gauss_offset(gauss_pick(need)) : -1};
            ++nblk;
            units += min(n, N);
        }
    }
    __syncwarp();
    return pb;
}

// Unit q of the piece: a row of a block's rule (q < nv) or a row of its own.
template <int Cap>
__device__ __forceinline__ void unit_row(const WarpNodes<Cap> &ns, const float2 *gauss, int G, int q, int nv, int R1,
                                         int nblk, NodeRow &o)
{
    float k = (float)(G - (R1 + q - nv)) - 0.5f, k_lo = 0.0f;
    float wt = 1.0f;
    if (q < nv) {
        int b = 0;
#pragma unroll 1
        while (b + 1 < nblk && ns.blk[b + 1].unit0 <= q) ++b;
        const RowBlock bl = ns.blk[b];
        if (bl.toff >= 0) {
            const float2 e = __ldg(gauss + bl.toff + (q - bl.unit0));
            const float h = -0.5f * (float)bl.N, kc = (float)(G - bl.r0) + h, kt = h * e.x;
            k = __fadd_rn(kc, kt);                            // |kt| <= kc
            k_lo = __fadd_rn(__fadd_rn(kc, -k), kt) + fmaf(h, e.x, -kt);
            wt = e.y;
        } else {
            k = (float)(G - (bl.r0 + q - bl.unit0)) - 0.5f;
        }
    }
    node_row(ns.geo, gauss, G, k, k_lo, o);
    o.w *= wt;
}

// Lists runs [first, first + kRowRuns) of unit `row` of the warp's 32 (candidates
// [ca, cb); whole >= 0: the one candidate that holds every column), their slots
// counted from 0; returns the slots, `more` whether further runs follow.
template <int Cap>
__device__ __forceinline__ int node_emit(WarpNodes<Cap> &ns, const NodeRow &o, int G, int row, int ca, int cb,
                                         int whole, int first, bool &more)
{
    int slots = 0, k = 0;
    const auto take_run = [&](int c, int j0, int N) {
        run_parts(ns.geo, o, G, j0, N, [&](int j, int Ns, int n) {
            if (k >= first && k < first + kRowRuns) {
                NodeRun r;
                r.jc = (float)j + 0.5f * (float)(Ns - G);
                r.half = 0.5f * (float)Ns;
                r.toff = n == Ns ? -1 : (Ns - 1) * kGaussPerN + gauss_offset(gauss_pick(n));
                r.id = (unsigned)slots | (unsigned)c << 16 | (unsigned)n << 24;
                ns.run[row * kRowRuns + (k - first)] = r;
                slots += n;
            }
            ++k;
        });
    };
    if (o.w != 0.0f) row_runs(ns.geo, o, G, ca, cb, whole, take_run);
    more = k > first + kRowRuns;
    return slots | min(max(k - first, 0), kRowRuns) << 16;
}

// One node: its row, candidate, f1 and f2 from the corner, phi and weight.
struct Node {
    int ci, N;                  // N: columns of a row's run at its first node, else 0
    float x, y, phi, phi_lo, wq;
};

template <int Cap>
__device__ __forceinline__ void node_get(const WarpNodes<Cap> &ns, const float2 *gauss, int c0, int q, Node &nd)
{
    const int id = ns.of[q];
    const NodeRun r = ns.run[id];
    const int k = c0 + q - (int)(r.id & 0xffffu);
    nd.ci = (int)(r.id >> 16 & 31u);
    nd.N = k == 0 && !(r.id >> 21 & 1u) ? (int)(2.0f * r.half) : 0;
    float pos, wt = 1.0f;
    if (r.toff >= 0) {
        const float2 e = __ldg(gauss + r.toff + k);
        pos = fmaf(e.x, r.half, r.jc);
        wt = e.y;
    } else {
        pos = r.jc - r.half + 0.5f + (float)k;
    }
    const PieceGeo &g = ns.geo;
    const NodeRow o = ns.row[id / kRowRuns];
    float ep, em, p1, p2;
    expm1_pair(pos * o.du2, ep, em);
    row_slopes(g, o, p1, p2);
    const float dx = g.s1 * o.xc * ep, dy = g.s2 * o.yc * em, du = dx + dy;
    nd.x = o.x0 + dx;
    nd.y = o.y0 + dy;
    const float dphi = du * fmaf(p2, du, p1);
    nd.phi = __fadd_rn(o.phi0, dphi);                 // two-sum
    const float t = __fadd_rn(nd.phi, -o.phi0);
    nd.phi_lo = __fadd_rn(__fadd_rn(o.phi0, -__fadd_rn(nd.phi, -t)), __fadd_rn(dphi, -t)) + o.phi0_lo;
    nd.wq = o.w * wt;
}

// The nodes of a piece in chunks: f(c0, number of slots) is called by the whole
// warp for each chunk, with ns filled for node_get (candidates [ca, cb)).
template <int Cap, typename F>
__device__ __forceinline__ void piece_nodes(WarpNodes<Cap> &ns, const PieceBlocks &pb, const float2 *gauss, int G,
                                            int ca, int cb, const F &f)
{
    const int lane = threadIdx.x & 31;
    const int nv = pb.units, R1 = pb.R1, nblk = pb.nblk, cand = pb.cand;
    const bool mine = cand >= ca && cand < cb;        // the blocks' candidate belongs to this sweep
    const int units = nv + (G - R1);
#pragma unroll 1
    for (int u0 = mine ? 0 : nv; u0 < units; u0 += 32) {
        const int q = u0 + lane;
        const int whole = q < nv ? cand : -1;
        NodeRow o;
        o.w = 0.0f;
        if (q < units) {
            unit_row(ns, gauss, G, q, nv, R1, nblk, o);
            ns.row[lane] = o;
        }
        bool more = false;
        int first = 0;
        do {
            const int got = node_emit(ns, o, G, lane, ca, cb, whole, first, more);
            const int slots = got & 0xffff, runs = got >> 16;
            int incl = slots;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += v;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31), base = incl - slots;
#pragma unroll 1
            for (int k = 0; k < runs; ++k) {          // slots of the warp's rows; bit 21: a block's row
                unsigned &id = ns.run[lane * kRowRuns + k].id;
                id = id + (unsigned)base + (whole >= 0 ? 1u << 21 : 0u);
            }
#pragma unroll 1
            for (int c0 = 0; c0 < total; c0 += Cap) {
                if (base < c0 + Cap && incl > c0)
#pragma unroll 1
                    for (int k = 0; k < runs; ++k) {
                        const unsigned id = ns.run[lane * kRowRuns + k].id;
                        const int s0 = (int)(id & 0xffffu) - c0, s1 = s0 + (int)(id >> 24);
#pragma unroll 1
                        for (int s = max(s0, 0); s < min(s1, Cap); ++s)
                            ns.of[s] = (unsigned char)(lane * kRowRuns + k);
                    }
                __syncwarp();
                f(c0, min(total - c0, Cap));
                __syncwarp();
            }
            first += kRowRuns;
        } while (__any_sync(0xffffffffu, more));
    }
}

}  // namespace isrs
