// FP32 z-sums of the closed-form profile, shared by the quadrature kernels.
#pragma once
#include <cuda_runtime.h>

#include "quad_common.cuh"

namespace isrs {

// ---------------------------------------------------------------------------
// FP32 z-sums.  Per-step tables staged in shared memory:
//   sT[m] = {A2_m + log2 dz_m, K2_m, z_m, c_m = z_m^2 + dz_m^2/12}
//   sR[m] = {A2_m + log2 dz_m, K2_m, z_m, dz_m}
//   sE[m] = {z_{m+1}/2pi hi, lo (float-float), A2_m, K2_m}
// with log2 p_m = A2_m + K2_m Fc - at z_m (Eq. pk for the closed-form
// profile).  The phase is carried in revolutions (z / 2pi).
//
// Exact-to-FP32 evaluations of S = sum_m p_m dz_m sinc(phi dz_m/2)
// e^{j phi z_m} (Eq. slow_vary), chosen per grid point by |phi|:
//  * contracted small phase (|phi| L <= 6, when the piece's Chebyshev
//    contraction applies): the centred series about the span centre with
//    6, 11 or 19 moments by phase (quad_common.cuh), no per-step work;
//  * small (|phi| L <= 0.02, otherwise): second-order expansion in phi,
//      |S|^2 = M0^2 - phi^2 (M0 M2 - M1^2) + O((phi L)^4),
//    M0 = sum p dz, M1 = sum p dz z, M2 = sum p dz (z^2 + dz^2/12); the
//    truncation is below 1e-9 relative (one exp per step, no phasor).
//  * direct (|phi| dz_max <= pi): the formula as written, sinc by its even
//    Taylor polynomial in x = phi dz/2 (|x| <= pi/2, truncation < 4e-8),
//    phase phi z/2pi < L/(2 dz_max) revolutions formed in FP32.
//  * telescoped (otherwise): dz sinc(phi dz/2) e^{j phi z_m} equals
//    (E_{m+1} - E_m)/(j phi) with E_e = e^{j phi z_e}, so one complex
//    exponential per edge suffices; the phase phi z_e / 2pi (up to ~1e5
//    revolutions) is an error-free float-float product reduced to [-1/2, 1/2].
// The final division by phi^2 takes the MUFU reciprocal (2 ulp; phi^2 lies
// far inside the range where it is accurate): an IEEE division there costs
// a branch to its slow path at every point.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float zsum_small_f(float phi, float Fc, float at, const float4 *sT, int M)
{
    float M0 = 0.0f, M1 = 0.0f, M2 = 0.0f;
#pragma unroll 4
    for (int m = 0; m < M; ++m) {
        const float4 a = sT[m];
        float lp = fmaf(a.y, Fc, a.x);
        lp = fmaf(-at, a.z, lp);
        const float w = ex2_approx(lp);          // p_m dz_m
        M0 += w;
        M1 = fmaf(w, a.z, M1);
        M2 = fmaf(w, a.w, M2);
    }
    return fmaf(-phi * phi, fmaf(M0, M2, -M1 * M1), M0 * M0);
}

__device__ __forceinline__ float zsum_direct_f(float phi, float Fc, float at, const float4 *sR, int M)
{
    // sR[m] = {A2_m + log2 dz_m, K2_m, z_m, dz_m}; phase in revolutions phi/2pi * z_m
    float Sr = 0.0f, Si = 0.0f;
    const float hphi = 0.5f * phi;
    const float phir = phi * 0.15915494309189535f;
#pragma unroll 4
    for (int m = 0; m < M; ++m) {
        const float4 a = sR[m];
        float sn, cs;
        sincos_rev(phir, a.z, sn, cs);
        const float x = hphi * a.w;
        const float x2 = x * x;
        float sc = fmaf(x2, -2.5052108e-8f, 2.7557319e-6f);   // -1/11!, 1/9!
        sc = fmaf(x2, sc, -1.9841270e-4f);                     // -1/7!
        sc = fmaf(x2, sc, 8.3333333e-3f);                      // 1/5!
        sc = fmaf(x2, sc, -1.6666667e-1f);                     // -1/3!
        sc = fmaf(x2, sc, 1.0f);
        float lp = fmaf(a.y, Fc, a.x);
        lp = fmaf(-at, a.z, lp);
        const float amp = ex2_approx(lp) * sc;   // p_m dz_m sinc
        Sr = fmaf(amp, cs, Sr);
        Si = fmaf(amp, sn, Si);
    }
    return Sr * Sr + Si * Si;
}

__device__ __forceinline__ float zsum_tele_f(float phi, float Fc, float at, const float4 *sT,
                                             const float4 *sE, int M)
{
    float Er = 1.0f, Ei = 0.0f, Sr = 0.0f, Si = 0.0f;
#pragma unroll 4
    for (int m = 0; m < M; ++m) {
        const float4 e = sE[m];
        const float zm = sT[m].z;
        float sn, cs;
        phasor_rev_ff(phi, e.x, e.y, sn, cs);
        float lp = fmaf(e.w, Fc, e.z);
        lp = fmaf(-at, zm, lp);
        const float p = ex2_approx(lp);
        Sr = fmaf(p, cs - Er, Sr);
        Si = fmaf(p, sn - Ei, Si);
        Er = cs;
        Ei = sn;
    }
    return __fdividef(Sr * Sr + Si * Si, phi * phi);
}

// The same two forms for a node of the row sums: zt[m] = {z_{m+1}/2pi hi, lo,
// z_m, dz_m} and, for the node's F_c candidate, ek[m] = {log2 p_m at the
// channel's centre, K2_m}, so log2 p_m = ek.x + K2_m dF with dF = F_c - f_c; phi
// is a float-float value (the direct form's phases need only its head).
__device__ __forceinline__ float zsum_direct_n(float phi, float dF, const float4 *zt, const float2 *ek, int M)
{
    float Sr = 0.0f, Si = 0.0f;
    const float hphi = 0.5f * phi;
    const float phir = phi * 0.15915494309189535f;
#pragma unroll 4
    for (int m = 0; m < M; ++m) {
        const float4 a = zt[m];
        const float2 e = ek[m];
        float sn, cs;
        sincos_rev(phir, a.z, sn, cs);
        const float x = hphi * a.w;
        const float x2 = x * x;
        float sc = fmaf(x2, -2.5052108e-8f, 2.7557319e-6f);   // -1/11!, 1/9!
        sc = fmaf(x2, sc, -1.9841270e-4f);                     // -1/7!
        sc = fmaf(x2, sc, 8.3333333e-3f);                      // 1/5!
        sc = fmaf(x2, sc, -1.6666667e-1f);                     // -1/3!
        sc = fmaf(x2, sc, 1.0f);
        const float amp = ex2_approx(fmaf(e.y, dF, e.x)) * (sc * a.w);
        Sr = fmaf(amp, cs, Sr);
        Si = fmaf(amp, sn, Si);
    }
    return Sr * Sr + Si * Si;
}

__device__ __forceinline__ float zsum_tele_n(float phi, float phi_lo, float dF, const float4 *zt, const float2 *ek,
                                             int M)
{
    float Er = 1.0f, Ei = 0.0f, Sr = 0.0f, Si = 0.0f;
#pragma unroll 4
    for (int m = 0; m < M; ++m) {
        const float4 a = zt[m];
        const float2 e = ek[m];
        float sn, cs;
        phasor_rev_ff(phi, a.x, a.y, sn, cs, phi_lo);
        const float p = ex2_approx(fmaf(e.y, dF, e.x));
        Sr = fmaf(p, cs - Er, Sr);
        Si = fmaf(p, sn - Ei, Si);
        Er = cs;
        Ei = sn;
    }
    return __fdividef(Sr * Sr + Si * Si, phi * phi);
}

// ... with the tabulated profile: q[m] = {log2 p_m, slope along the node's
// longer axis, along the shorter}, dl and dd the offsets of F_a, F_b inside
// their channels (in that order of axes).
__device__ __forceinline__ float zsum_direct_nt(float phi, float dl, float dd, const float4 *zt, const float4 *q,
                                                int M)
{
    float Sr = 0.0f, Si = 0.0f;
    const float hphi = 0.5f * phi;
    const float phir = phi * 0.15915494309189535f;
#pragma unroll 4
    for (int m = 0; m < M; ++m) {
        const float4 a = zt[m];
        const float4 e = q[m];
        float sn, cs;
        sincos_rev(phir, a.z, sn, cs);
        const float x = hphi * a.w;
        const float x2 = x * x;
        float sc = fmaf(x2, -2.5052108e-8f, 2.7557319e-6f);   // -1/11!, 1/9!
        sc = fmaf(x2, sc, -1.9841270e-4f);                     // -1/7!
        sc = fmaf(x2, sc, 8.3333333e-3f);                      // 1/5!
        sc = fmaf(x2, sc, -1.6666667e-1f);                     // -1/3!
        sc = fmaf(x2, sc, 1.0f);
        const float amp = ex2_approx(fmaf(e.z, dd, fmaf(e.y, dl, e.x))) * (sc * a.w);
        Sr = fmaf(amp, cs, Sr);
        Si = fmaf(amp, sn, Si);
    }
    return Sr * Sr + Si * Si;
}

__device__ __forceinline__ float zsum_tele_nt(float phi, float phi_lo, float dl, float dd, const float4 *zt,
                                              const float4 *q, int M)
{
    float Er = 1.0f, Ei = 0.0f, Sr = 0.0f, Si = 0.0f;
#pragma unroll 4
    for (int m = 0; m < M; ++m) {
        const float4 a = zt[m];
        const float4 e = q[m];
        float sn, cs;
        phasor_rev_ff(phi, a.x, a.y, sn, cs, phi_lo);
        const float p = ex2_approx(fmaf(e.z, dd, fmaf(e.y, dl, e.x)));
        Sr = fmaf(p, cs - Er, Sr);
        Si = fmaf(p, sn - Ei, Si);
        Er = cs;
        Ei = sn;
    }
    return __fdividef(Sr * Sr + Si * Si, phi * phi);
}

// As phasor_rev_ff, for phases far beyond 2^22 revolutions (the MCI cells, up
// to 2^29): there the first rounding is to a multiple of 2 or more and leaves a
// few revolutions; a second rounding removes them.
__device__ __forceinline__ void phasor_rev_ff_wide(float phi, float hi, float lo, float &sn, float &cs)
{
    float fr = fmaf(phi, lo, rev_fraction(phi, hi));
    fr = __fadd_rn(fr, -__fadd_rn(__fadd_rn(fr, 12582912.0f), -12582912.0f));
    __sincosf(fr * 6.283185307179586f, &sn, &cs);
}

__device__ __forceinline__ float zsum_tele_wide_f(float phi, float Fc, float at, const float4 *sT,
                                                  const float4 *sE, int M)
{
    float Er = 1.0f, Ei = 0.0f, Sr = 0.0f, Si = 0.0f;
#pragma unroll 4
    for (int m = 0; m < M; ++m) {
        const float4 e = sE[m];
        const float zm = sT[m].z;
        float sn, cs;
        phasor_rev_ff_wide(phi, e.x, e.y, sn, cs);
        float lp = fmaf(e.w, Fc, e.z);
        lp = fmaf(-at, zm, lp);
        const float p = ex2_approx(lp);
        Sr = fmaf(p, cs - Er, Sr);
        Si = fmaf(p, sn - Ei, Si);
        Er = cs;
        Ei = sn;
    }
    return __fdividef(Sr * Sr + Si * Si, phi * phi);
}

}  // namespace isrs
