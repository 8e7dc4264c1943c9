// Device helpers shared by the quadrature kernels (forward and adjoint).
#pragma once
#include <cuda_runtime.h>

#include "isrs_internal.cuh"

namespace isrs {

// ---------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Fraction of a phase a b in revolutions, in [-1/2, 1/2]: the integer nearest
// to the exact product comes out of one FMA against 1.5 2^23 (|a b| < 2^22) and
// the fraction out of a second one, rounded once.  Three instructions on the FMA
// pipe; rounding the product first, with its residual as a second float, took
// five, and FRND would go to the XU pipe, which the sin, cos and ex2 of a z-step
// keep busy for 20 cycles per warp and step.
__device__ __forceinline__ float rev_fraction(float a, float b)
{
    const float k = __fadd_rn(__fmaf_rn(-a, b, 12582912.0f), -12582912.0f);
    return __fmaf_rn(a, b, k);
}

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ln(sinh(x) / x) and its derivative coth(x) - 1/x in FP64.  Up to |x| = 0.2
// (kappa B / 2 of any practical channel) the Taylor series of either, dropped
// terms below 2e-16: a few FMAs where sinh, log, tanh and two divisions were most
// of the small per-step kernels' time.
__device__ __forceinline__ double log_sinhc(double x)
{
    const double q = x * x;
    if (q > 0.04) return log(sinh(x) / x);
    double p = -691.0 / 3831077250.0;
    p = fma(p, q, 1.0 / 467775.0);
    p = fma(p, q, -1.0 / 37800.0);
    p = fma(p, q, 1.0 / 2835.0);
    p = fma(p, q, -1.0 / 180.0);
    p = fma(p, q, 1.0 / 6.0);
    return p * q;
}

__device__ __forceinline__ double dlog_sinhc(double x)
{
    const double q = x * x;
    if (q > 0.04) return 1.0 / tanh(x) - 1.0 / x;
    double p = -1382.0 / 638512875.0;
    p = fma(p, q, 2.0 / 93555.0);
    p = fma(p, q, -1.0 / 4725.0);
    p = fma(p, q, 2.0 / 945.0);
    p = fma(p, q, -1.0 / 45.0);
    p = fma(p, q, 1.0 / 3.0);
    return p * x;
}

// Block maximum (every thread gets it; scratch holds 32 values).
__device__ __forceinline__ double block_max_d(double v, double *scratch)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) scratch[wid] = v;
    __syncthreads();
    double m = -1e300;
    for (int w = 0; w < nw; ++w) m = fmax(m, scratch[w]);
    return m;
}

// Deterministic block sum of one double per thread (blockDim multiple of 32).
__device__ __forceinline__ double block_sum_d(double v, double *scratch)
{
    v = warp_sum_d(v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) scratch[wid] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0) {
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += scratch[w];
        scratch[0] = r;
    }
    __syncthreads();
    r = scratch[0];
    __syncthreads();
    return r;
}

// Grid points and z-sums of a launch (QuadParams::path_count, isrs_last_path_counts and
// isrs_last_node_counts).  A point counts by its phase, the low ones first, so that each
// counts once also where the z-grid is so coarse that low points are telescoped.
constexpr float kSmallPhiL = 6.0f;       // |phi| n_spans L of the low points

struct PathCount {                       // of one lane
    unsigned long long small = 0;
    unsigned direct = 0, tele = 0, sums_direct = 0, sums_tele = 0;
    // a z-sum that stands for n points
    __device__ __forceinline__ void points(float aphi, float phi_small, bool telescoped, int n)
    {
        const bool low = aphi <= phi_small;
        small += low ? n : 0;
        direct += low || telescoped ? 0 : n;
        tele += !low && telescoped ? n : 0;
    }
    __device__ __forceinline__ void sums(bool telescoped, int n)
    {
        if (telescoped) sums_tele += n;
        else sums_direct += n;
    }
    // whole warp
    __device__ __forceinline__ void store(unsigned long long *out) const
    {
        unsigned long long c[5] = {small, direct, tele, sums_direct, sums_tele};
#pragma unroll
        for (int k = 0; k < 5; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c[k] += __shfl_xor_sync(0xffffffffu, c[k], o);
            if ((threadIdx.x & 31) == 0) atomicAdd(out + k, c[k]);
        }
    }
};

// ---------------------------------------------------------------------------
// Piece set-up of the FP64 kernels, once per piece.
// Row r (uniform in s = ln upsilon1): upsilon1 = exp(s_r); the |f2| range
// [ymin, ymax] of that row; upsilon2 spans ln(ymax/ymin) in G columns.
// Stored relative to the row centre:
//   x_j = xc e^{d_j}, y_j = yc e^{-d_j}, d_j = (j + 1/2 - G/2) du2,
//   weight = upsilon1 ds du2 (the Jacobian of (f1, f2) -> (u1, u2) is 1).
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void piece_rows(const DevPiece &pc, int G, double eps, T *rows)
{
    const double u1hi = pc.xhi * pc.yhi;
    const double u1lo = fmax(pc.xlo * pc.ylo, eps * u1hi);
    const double llo = log(u1lo);
    const double ds = (log(u1hi) - llo) / G;
    for (int r = threadIdx.x; r < G; r += blockDim.x) {
        const double u1 = exp(llo + (r + 0.5) * ds);
        const double ymin = fmax(pc.ylo, u1 / pc.xhi);
        const double ymax = pc.xlo > 0.0 ? fmin(pc.yhi, u1 / pc.xlo) : pc.yhi;
        T rw;
        if (ymax > ymin) {
            const double du2 = log1p((ymax - ymin) / ymin) / G;
            const double yc = sqrt(ymin * ymax);
            rw.xc = u1 / yc;
            rw.yc = yc;
            rw.du2 = du2;
            rw.w = u1 * ds * du2;
        } else {
            rw.xc = 0; rw.yc = 0; rw.du2 = 0; rw.w = 0;
        }
        rows[r] = rw;
    }
}

struct RowD { double xc, yc, du2, w; };

// Per-piece constants: CUT offset, signs, the PSD factors of F_a and F_b, the
// attenuation part of ln p and the candidate channels of F_c (edges relative
// to the CUT so that F_c - f_i = f1 + f2 is compared without cancellation).
template <typename T>
struct PieceConst {
    T fi, s1, s2, wab, at_ab, mult;
    int nc;
    T lo[kMaxCand], hi[kMaxCand], pd[kMaxCand], hat[kMaxCand];
};

template <typename T>
__device__ __forceinline__ void piece_consts(const QuadParams &qp, const DevPiece &pc, int prof, T at_scale,
                             const T *pdv, PieceConst<T> &k)
{
    if (threadIdx.x == 0) {
        const int coff = qp.plan_ch_off[pc.plan];
        const int poff = qp.prof_ch_off[prof];
        const double fi = qp.ch_frel[coff + pc.cut];
        k.fi = (T)fi;
        k.s1 = (pc.flags & 1) ? T(-1) : T(1);
        k.s2 = (pc.flags & 2) ? T(-1) : T(1);
        k.wab = pdv[poff + pc.a] * pdv[poff + pc.b];
        k.at_ab = (T)(0.5 * (qp.ch_alpha[coff + pc.a] + qp.ch_alpha[coff + pc.b] -
                             qp.ch_alpha[coff + pc.cut])) * at_scale;
        k.mult = (T)pc.mult;
        int nc = 0;
        for (int c = pc.c_lo; c <= pc.c_hi && nc < kMaxCand; ++c, ++nc) {
            const double fc = qp.ch_frel[coff + c], hb = 0.5 * qp.ch_B[coff + c];
            k.lo[nc] = (T)((fc - hb) - fi);
            k.hi[nc] = (T)((fc + hb) - fi);
            k.pd[nc] = pdv[poff + c];
            k.hat[nc] = (T)(0.5 * qp.ch_alpha[coff + c]) * at_scale;
        }
        k.nc = nc;
    }
}

// Beyond 2^21 revolutions (the MCI cells) the constant 1.5 2^23 is too small: past 2^22
// the sum with it leaves the binade whose spacing is 1, and "the nearest integer" becomes a
// half-integer.  With 1.5 2^31 it is a multiple of 256 (up to 2^30 revolutions), and a
// second rounding takes the rest.
constexpr float kTurnMagic = 12582912.0f, kTurnMagicWide = 3221225472.0f;
constexpr float kTurnsWide = 2097152.0f;
__device__ __forceinline__ float turn_magic(float revs)
{
    return fabsf(revs) > kTurnsWide ? kTurnMagicWide : kTurnMagic;
}

// e^{j phi z}: the phase (phi + phi_lo)(hi + lo) in revolutions, |.| < 2^22 (Wide: 2^30)
template <bool Wide = false>
__device__ __forceinline__ void phasor_rev_ff(float phi, float hi, float lo, float &sn, float &cs,
                                              float phi_lo = 0.0f)
{
    float fr;
    if constexpr (Wide) {
        const float mg = turn_magic(phi * hi);
        fr = fmaf(phi, lo, __fmaf_rn(phi, hi, __fadd_rn(__fmaf_rn(-phi, hi, mg), -mg)));
        fr = rev_fraction(fr, 1.0f);
    } else {
        fr = fmaf(phi_lo, hi, fmaf(phi, lo, rev_fraction(phi, hi)));
    }
    __sincosf(fr * 6.283185307179586f, &sn, &cs);
}

// e^x by its Taylor series: to x^7 for |x| <= 1/64 (remainder 9e-20; in pairs, five
// FMAs deep, for the ODE steps are one chain of them), to x^11 for |x| <= 1/8
// (3e-20), else the library's
__device__ __forceinline__ double exp_small(double x)
{
    if (fabs(x) <= 0.015625) {
        const double x2 = x * x;
        const double a = fma(x, 1.0 / 5040.0, 1.0 / 720.0), b = fma(x, 1.0 / 120.0, 1.0 / 24.0);
        const double c = fma(x, 1.0 / 6.0, 0.5);
        return fma(x2, fma(x2, fma(x2, a, b), c), 1.0 + x);
    }
    if (fabs(x) > 0.125) return exp(x);
    double p = 1.0 / 39916800.0;
    p = fma(p, x, 1.0 / 3628800.0);
    p = fma(p, x, 1.0 / 362880.0);
    p = fma(p, x, 1.0 / 40320.0);
    p = fma(p, x, 1.0 / 5040.0);
    p = fma(p, x, 1.0 / 720.0);
    p = fma(p, x, 1.0 / 120.0);
    p = fma(p, x, 1.0 / 24.0);
    p = fma(p, x, 1.0 / 6.0);
    p = fma(p, x, 0.5);
    p = fma(p, x, 1.0);
    return fma(p, x, 1.0);
}

// |S|^2 of Eq. slow_vary in FP64, p(m) the power of step m, sz[m] = {z_m, dz_m}.
// dz sinc(phi dz/2) e^{j phi z_m} = (E_{m+1} - E_m) / (j phi) exactly, so above
// |phi| dz_max = 0.1 a step takes one phasor (the smallest step still turns by
// 0.1 dz_min / dz_max, so the difference keeps 13 digits); below, sinc by its
// Taylor series to x^8 (|x| <= 0.05: remainder 3e-21).  The FP64 pipe runs at
// 1/64 of the FP32 rate here: sincos, sin, a division and a full exp per step
// took ~130 instructions, this form ~50.
constexpr double kF64Direct = 0.1;

template <typename F>
__device__ __forceinline__ double zsum_f64(double phi, double phi_direct, const double2 *sz, int M, const F &p)
{
    double Sr = 0.0, Si = 0.0;
    const double ph = phi * 0.31830988618379067154;      // phases in half-turns
    if (fabs(phi) > phi_direct) {
        double Er = 1.0, Ei = 0.0;
        for (int m = 0; m < M; ++m) {
            const double2 z = sz[m];
            double sn, cs;
            sincospi(ph * fma(0.5, z.y, z.x), &sn, &cs);
            const double w = p(m);
            Sr = fma(w, cs - Er, Sr);
            Si = fma(w, sn - Ei, Si);
            Er = cs;
            Ei = sn;
        }
        return (Sr * Sr + Si * Si) / (phi * phi);
    }
    for (int m = 0; m < M; ++m) {
        const double2 z = sz[m];
        const double x = 0.5 * phi * z.y, x2 = x * x;
        double sc = fma(x2, 1.0 / 362880.0, -1.0 / 5040.0);
        sc = fma(x2, sc, 1.0 / 120.0);
        sc = fma(x2, sc, -1.0 / 6.0);
        sc = fma(x2, sc, 1.0);
        double sn, cs;
        sincospi(ph * z.x, &sn, &cs);
        const double w = p(m) * z.y * sc;
        Sr = fma(w, cs, Sr);
        Si = fma(w, sn, Si);
    }
    return Sr * Sr + Si * Si;
}

// Phased-array factor of n identical spans (Eq. new_gn_model with
// L-tilde_k = (k-1) L): |sum_{k<n} e^{j k phi L}|^2, by rotation from the
// float-float phase phi L / 2pi (Wide: as phasor_rev_ff).
template <bool Wide = false>
__device__ __forceinline__ float array_factor_f(float phi, const QuadParams &qp, float phi_lo = 0.0f)
{
    if (qp.n_spans <= 1) return 1.0f;
    float sn, cs;
    phasor_rev_ff<Wide>(phi, qp.Lrev_hi, qp.Lrev_lo, sn, cs, phi_lo);
    float sr = 0.0f, si = 0.0f, zr = 1.0f, zi = 0.0f;
    for (int k = 0; k < qp.n_spans; ++k) {
        sr += zr;
        si += zi;
        const float t = fmaf(zr, cs, -zi * sn);
        zi = fmaf(zr, sn, zi * cs);
        zr = t;
    }
    return fmaf(sr, sr, si * si);
}

__device__ __forceinline__ double array_factor_d(double phi, const QuadParams &qp)
{
    if (qp.n_spans <= 1) return 1.0;
    double sn, cs;
    sincos(phi * qp.Ld, &sn, &cs);
    double sr = 0.0, si = 0.0, zr = 1.0, zi = 0.0;
    for (int k = 0; k < qp.n_spans; ++k) {
        sr += zr;
        si += zi;
        const double t = zr * cs - zi * sn;
        zi = zr * sn + zi * cs;
        zr = t;
    }
    return sr * sr + si * si;
}

}  // namespace isrs
