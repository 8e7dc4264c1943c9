// FP32 z-sums of the closed-form profile, shared by the quadrature kernels.
#pragma once
#include <cuda_runtime.h>

#include "f32x2.cuh"
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

// The same two forms for a node of the row sums, two steps at a time (f32x2.cuh):
// pair k of eB = {z_{m+1}/2pi hi, hi', lo, lo'}, of zD = {z_m, z', dz_m, dz'},
// and lp(k) gives log2 p of the pair at the node; an odd last step stands beside one
// of weight 2^-1000 with the same edge.  phi is float-float (the direct form's
// phases need only its head).  Packed, a step takes ~13 instructions where the
// scalar form took ~19; bound by the XU pipe (20 cycles per warp and step).
// The _part forms give Re S and Im S (times phi for the telescoped one) of the
// pairs [k0, k1), so that a few lanes can share a node.
template <typename LP>
__device__ __forceinline__ float2 zsum_direct_part(float phi, const LP &lp, const float4 *zD, int k0, int k1)
{
    const f32x2 hph = dup2(0.5f * phi), phr = dup2(phi * 0.15915494309189535f),
                nphr = dup2(-phi * 0.15915494309189535f);
    const f32x2 mg = dup2(12582912.0f), nm = dup2(-12582912.0f);
    f32x2 Sr = dup2(0.0f), Si = dup2(0.0f);
#pragma unroll 2
    for (int k = k0; k < k1; ++k) {
        const float4 z = zD[k];
        const f32x2 zz = pack2(z.x, z.y), dz = pack2(z.z, z.w);
        float s0, c0, s1, c1, l0, l1;
        sincos_turn2(fma2(phr, zz, add2(fma2(nphr, zz, mg), nm)), s0, c0, s1, c1);
        const f32x2 x = mul2(hph, dz), x2 = mul2(x, x);       // sinc to x^10, |x| <= pi/2
        f32x2 sc = fma2(x2, dup2(-2.5052108e-8f), dup2(2.7557319e-6f));
        sc = fma2(x2, sc, dup2(-1.9841270e-4f));
        sc = fma2(x2, sc, dup2(8.3333333e-3f));
        sc = fma2(x2, sc, dup2(-1.6666667e-1f));
        sc = fma2(x2, sc, dup2(1.0f));
        unpack2(lp(k), l0, l1);
        const f32x2 amp = mul2(pack2(ex2_approx(l0), ex2_approx(l1)), mul2(sc, dz));
        Sr = fma2(amp, pack2(c0, c1), Sr);
        Si = fma2(amp, pack2(s0, s1), Si);
    }
    float r0, r1, i0, i1;
    unpack2(Sr, r0, r1);
    unpack2(Si, i0, i1);
    return make_float2(r0 + r1, i0 + i1);
}

template <typename LP>
__device__ __forceinline__ float zsum_direct_n(float phi, const LP &lp, const float4 *zD, int M2)
{
    const float2 s = zsum_direct_part(phi, lp, zD, 0, M2);
    return s.x * s.x + s.y * s.y;
}

// The telescoped sum by parts, sum p_m (E_{m+1} - E_m) = p_last E_last - p_0 E_0 -
// sum (p_m - p_{m-1}) E_m: two differences per pair of steps instead of four.
template <int Form, typename LP>
__device__ __forceinline__ float2 zsum_tele_part(float phi, float phi_lo, const LP &lp, const float4 *eB, int k0,
                                                 int k1)
{
    const f32x2 ph = dup2(phi), nph = dup2(-phi), pl = dup2(phi_lo);
    float Er = 1.0f, Ei = 0.0f, pp = 0.0f;
    if (k0 > 0) {                        // phasor at the edge before
        const float4 e = eB[k0 - 1];
        float s0, c0;
        sincos_turn2(rev_fraction2<Form>(ph, nph, pl, pack2(e.x, e.y), pack2(e.z, e.w)), s0, c0, Ei, Er);
    }
    f32x2 Sr = dup2(0.0f), Si = dup2(0.0f);
#pragma unroll 4
    for (int k = k0; k < k1; ++k) {
        const float4 e = eB[k];
        float s0, c0, s1, c1, l0, l1;
        sincos_turn2(rev_fraction2<Form>(ph, nph, pl, pack2(e.x, e.y), pack2(e.z, e.w)), s0, c0, s1, c1);
        unpack2(lp(k), l0, l1);
        const float p0 = ex2_approx(l0), p1 = ex2_approx(l1);
        const f32x2 d = pack2(pp - p0, p0 - p1);
        Sr = fma2(d, pack2(Er, c0), Sr);
        Si = fma2(d, pack2(Ei, s0), Si);
        Er = c1;
        Ei = s1;
        pp = p1;
    }
    float r0, r1, i0, i1;
    unpack2(Sr, r0, r1);
    unpack2(Si, i0, i1);
    return make_float2(fmaf(pp, Er, r0 + r1), fmaf(pp, Ei, i0 + i1));
}

template <int Form, typename LP>
__device__ __forceinline__ float zsum_tele_n(float phi, float phi_lo, const LP &lp, const float4 *eB, int M2)
{
    const float2 s = zsum_tele_part<Form>(phi, phi_lo, lp, eB, 0, M2);
    return __fdividef(s.x * s.x + s.y * s.y, phi * phi);
}

// Steps in pairs: pair k holds steps 2k, 2k + 1.
__host__ __device__ constexpr int step_pairs(int n_steps) { return (n_steps + 1) / 2; }

// eB and zD of every pair, filled by the whole block
__device__ __forceinline__ void pair_tables(const QuadParams &qp, float4 *eB, float4 *zD)
{
    const int M = qp.n_steps;
    for (int k = threadIdx.x; k < step_pairs(M); k += blockDim.x) {
        const int m0 = 2 * k, m1 = min(2 * k + 1, M - 1);
        const float4 b0 = qp.zs_b[m0], b1 = qp.zs_b[m1], a0 = qp.zs_a[m0], a1 = qp.zs_a[m1];
        eB[k] = make_float4(b0.x, b1.x, b0.y, b1.y);
        zD[k] = make_float4(a0.x, a1.x, a0.w, a1.w);
    }
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
