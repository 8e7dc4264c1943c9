// FP32 z-sums, shared by the forward quadrature kernels.
#pragma once
#include <cuda_runtime.h>

#include "f32x2.cuh"
#include "quad_common.cuh"

namespace isrs {

// FP32 evaluations of S = sum_m p_m dz_m sinc(phi dz_m/2) e^{j phi z_m} (Eq.
// slow_vary), chosen per node or point by |phi|:
//  * direct (|phi| dz_max <= pi): the formula as written, sinc by its even
//    Taylor polynomial in x = phi dz/2 (|x| <= pi/2, truncation < 4e-8), phase
//    phi z/2pi < L/(2 dz_max) revolutions formed in FP32;
//  * telescoped (otherwise): dz sinc(phi dz/2) e^{j phi z_m} equals
//    (E_{m+1} - E_m)/(j phi) with E_e = e^{j phi z_e}, so one complex
//    exponential per edge suffices; the phase phi z_e / 2pi (up to ~1e5
//    revolutions) is an error-free float-float product reduced to [-1/2, 1/2].
// Both take two steps at a time (f32x2.cuh): pair k of eB = {z_{m+1}/2pi hi, hi',
// lo, lo'}, of zD = {z_m, z', dz_m, dz'}, and lp(k) gives log2 p of the pair; an odd
// last step stands beside one of weight 2^-1000 with the same edge.  phi is
// float-float (the direct form's phases need only its head).  Packed, a step takes
// ~13 instructions where the scalar form took ~19; bound by the XU pipe (20 cycles
// per warp and step).  The final division by phi^2 takes the MUFU reciprocal (2
// ulp): an IEEE division costs a branch to its slow path.
// The _part forms give Re S and Im S (times phi for the telescoped one) of the
// pairs [k0, k1), so that a few lanes can share a node.
// The special-function unit truncates: its ex2 is 5.1e-8 low on average and the phasor
// of its sin and cos 7.3e-8 short (mean over a turn), so |S|^2 comes out 2.5e-7 low in
// the direct form and 1.0e-7 to 1.2e-7 in the telescoped one, whose first edge is exact.  Every
// node's value is raised by that, which costs one multiplication a node: the eta of 5
// channels at G 64 was 2.2e-7 off FP64, of 65 channels over three spans 3.1e-7 (and the
// moments that summed small phases before, 1.4e-7 and 1.7e-7).
constexpr float kUlp1 = 1.1920929e-7f;                  // 2^-23
__device__ __forceinline__ float zsum_gain(bool telescoped) { return telescoped ? 1.0f + kUlp1 : 1.0f + 2.0f * kUlp1; }

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
    return (s.x * s.x + s.y * s.y) * zsum_gain(false);
}

// The telescoped sum by parts, sum p_m (E_{m+1} - E_m) = p_last E_last - p_0 E_0 -
// sum (p_m - p_{m-1}) E_m: two differences per pair of steps instead of four.
template <int Form, typename LP>
__device__ __forceinline__ float2 zsum_tele_part(float phi, float phi_lo, const LP &lp, const float4 *eB, int k0,
                                                 int k1, float magic = kTurnMagic)
{
    const f32x2 ph = dup2(phi), nph = dup2(-phi), pl = dup2(phi_lo);
    float Er = 1.0f, Ei = 0.0f, pp = 0.0f;
    if (k0 > 0) {                        // phasor at the edge before
        const float4 e = eB[k0 - 1];
        float s0, c0;
        sincos_turn2(rev_fraction2<Form>(ph, nph, pl, pack2(e.x, e.y), pack2(e.z, e.w), magic), s0, c0, Ei, Er);
    }
    f32x2 Sr = dup2(0.0f), Si = dup2(0.0f);
#pragma unroll 4
    for (int k = k0; k < k1; ++k) {
        const float4 e = eB[k];
        float s0, c0, s1, c1, l0, l1;
        sincos_turn2(rev_fraction2<Form>(ph, nph, pl, pack2(e.x, e.y), pack2(e.z, e.w), magic), s0, c0, s1, c1);
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
    return __fdividef(s.x * s.x + s.y * s.y, phi * phi) * zsum_gain(true);
}

// Steps in pairs: pair k holds steps 2k, 2k + 1.
__host__ __device__ constexpr int step_pairs(int n_steps) { return (n_steps + 1) / 2; }

// eB and zD of every pair, filled by the whole block
__device__ __forceinline__ void pair_tables(const QuadParams &qp, float4 *eB, float4 *zD)
{
    const int M = qp.n_steps;
    for (int k = threadIdx.x; k < step_pairs(M); k += blockDim.x) {
        const int m0 = 2 * k, m1 = min(2 * k + 1, M - 1);
        const float2 b0 = qp.zs_b[m0], b1 = qp.zs_b[m1], a0 = qp.zs_a[m0], a1 = qp.zs_a[m1];
        eB[k] = make_float4(b0.x, b1.x, b0.y, b1.y);
        zD[k] = make_float4(a0.x, a1.x, a0.y, a1.y);
    }
}

}  // namespace isrs
