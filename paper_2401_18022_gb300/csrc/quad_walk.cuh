// Half-warp walks of the FP32 adjoint kernels: the z-sum of one grid point or
// node (App. A, Eq. slow_vary) spread over the 16 lanes of a half-warp, each lane
// owning 2 K2 consecutive steps in K2 pairs (f32x2.cuh), with the terms kept in
// registers for the bucket terms d|S|^2/d ln p_m = 2 Re(conj(S) t_m).
//
// Steps in pairs: the multiply-adds of two steps share an issue slot, and what
// bounds the walk is the XU pipe (20 cycles per warp and step: sin and cos 8 each,
// ex2 4) instead of issue.  The span's M steps fill 16 x 2 K2 places (112 steps:
// 14 lanes of 16); the places past M carry log2 weight -1000 and repeat the last
// edge.
#pragma once
#include <cuda_runtime.h>

#include "f32x2.cuh"
#include "quad_common.cuh"
#include "quad_zsum.cuh"

namespace isrs {

constexpr unsigned kWarpAll = 0xffffffffu;
constexpr float kPadLog2 = -1000.0f;   // log2 weight of the padding steps (ex2 -> 0)

// step of place o of pair k of lane l
template <int K2>
__device__ __forceinline__ int walk_step(int k, int l, int o)
{
    return l * 2 * K2 + 2 * k + o;
}

// ze[k][16] = {edge/2pi hi, hi', lo, lo'}, zd[k][16] = {z, z', dz, dz'} of the
// pairs of all 16 lanes, filled by the whole block.
template <int K2>
__device__ __forceinline__ void walk_tables(const QuadParams &qp, float4 *ze, float4 *zd)
{
    for (int t = threadIdx.x; t < K2 * 16; t += blockDim.x) {
        const int m0 = min(walk_step<K2>(t >> 4, t & 15, 0), qp.n_steps - 1);
        const int m1 = min(walk_step<K2>(t >> 4, t & 15, 1), qp.n_steps - 1);
        const float2 b0 = qp.zs_b[m0], b1 = qp.zs_b[m1], a0 = qp.zs_a[m0], a1 = qp.zs_a[m1];
        ze[t] = make_float4(b0.x, b1.x, b0.y, b1.y);
        zd[t] = make_float4(a0.x, a1.x, a0.y, a1.y);
    }
}

// sum over the 16 lanes of each half-warp (both halves in step)
__device__ __forceinline__ float half_sum(float v)
{
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(kWarpAll, v, o, 16);
    return v;
}

template <int K2>
__device__ __forceinline__ void walk_sum(const f32x2 (&tr)[K2], const f32x2 (&ti)[K2], float &sr, float &si)
{
    f32x2 a = tr[0], b = ti[0];
#pragma unroll
    for (int k = 1; k < K2; ++k) {
        a = add2(a, tr[k]);
        b = add2(b, ti[k]);
    }
    float x, y;
    unpack2(a, x, y);
    sr = half_sum(x + y);
    unpack2(b, x, y);
    si = half_sum(x + y);
}

__device__ __forceinline__ f32x2 ex2_pair(f32x2 x)
{
    float a, b;
    unpack2(x, a, b);
    return pack2(ex2_approx(a), ex2_approx(b));
}

// Terms t_m = p_m dz_m sinc(phi dz_m/2) e^{j phi z_m} and their sum; lp(k) gives
// log2 p of pair k (zd offset by the lane).
template <int K2, typename LP>
__device__ __forceinline__ void walk_direct(const float4 *zd, float ph, const LP &lp, f32x2 (&tr)[K2], f32x2 (&ti)[K2],
                                            float &sr, float &si)
{
    const f32x2 hph = dup2(0.5f * ph), phr = dup2(ph * 0.15915494309189535f), nphr = dup2(-ph * 0.15915494309189535f);
    const f32x2 mg = dup2(12582912.0f), nm = dup2(-12582912.0f);
#pragma unroll
    for (int k = 0; k < K2; ++k) {
        const float4 z = zd[k * 16];
        const f32x2 zz = pack2(z.x, z.y), dz = pack2(z.z, z.w);
        float s0, c0, s1, c1;
        sincos_turn2(fma2(phr, zz, add2(fma2(nphr, zz, mg), nm)), s0, c0, s1, c1);
        const f32x2 x = mul2(hph, dz), x2 = mul2(x, x);       // sinc to x^10, |x| <= pi/2
        f32x2 sc = fma2(x2, dup2(-2.5052108e-8f), dup2(2.7557319e-6f));
        sc = fma2(x2, sc, dup2(-1.9841270e-4f));
        sc = fma2(x2, sc, dup2(8.3333333e-3f));
        sc = fma2(x2, sc, dup2(-1.6666667e-1f));
        sc = fma2(x2, sc, dup2(1.0f));
        const f32x2 amp = mul2(ex2_pair(lp(k)), mul2(sc, dz));
        tr[k] = mul2(amp, pack2(c0, c1));
        ti[k] = mul2(amp, pack2(s0, s1));
    }
    walk_sum<K2>(tr, ti, sr, si);
}

// Telescoped: terms p_m (E_{m+1} - E_m), E_e = e^{j phi z_e}, and their sum U,
// |S|^2 = |U|^2 / phi^2 (ze offset by the lane; phi float-float, or Wide: up to
// 2^30 revolutions, magic by turn_magic).
template <int K2, bool Wide, typename LP>
__device__ __forceinline__ void walk_tele(const float4 *ze, int l16, float ph, float ph_lo, const LP &lp,
                                          f32x2 (&tr)[K2], f32x2 (&ti)[K2], float &ur, float &ui,
                                          float magic = kTurnMagic)
{
    const f32x2 p2 = dup2(ph), np2 = dup2(-ph), pl2 = dup2(ph_lo);
    float Er = 0.0f, Ei = 0.0f, f0r = 0.0f, f0i = 0.0f, f1r = 0.0f, f1i = 0.0f;
    f32x2 p0 = p2;
#pragma unroll
    for (int k = 0; k < K2; ++k) {
        const float4 e = ze[k * 16];
        float s0, c0, s1, c1;
        sincos_turn2(rev_fraction2<Wide>(p2, np2, pl2, pack2(e.x, e.y), pack2(e.z, e.w), magic), s0, c0, s1, c1);
        const f32x2 p = ex2_pair(lp(k));
        if (k == 0) {
            p0 = p;
            f0r = c0;
            f0i = s0;
            f1r = c1 - c0;
            f1i = s1 - s0;
        } else {
            tr[k] = mul2(p, pack2(c0 - Er, c1 - c0));
            ti[k] = mul2(p, pack2(s0 - Ei, s1 - s0));
        }
        Er = c1;
        Ei = s1;
    }
    // the lower edge of this lane's first step is the previous lane's last edge
    float elr = __shfl_up_sync(kWarpAll, Er, 1, 16);
    float eli = __shfl_up_sync(kWarpAll, Ei, 1, 16);
    elr = l16 == 0 ? 1.0f : elr;
    eli = l16 == 0 ? 0.0f : eli;
    tr[0] = mul2(p0, pack2(f0r - elr, f1r));
    ti[0] = mul2(p0, pack2(f0i - eli, f1i));
    walk_sum<K2>(tr, ti, ur, ui);
}

// 2 Re(conj(S) t) / 2 of pair k
template <int K2>
__device__ __forceinline__ f32x2 walk_term(const f32x2 (&tr)[K2], const f32x2 (&ti)[K2], int k, f32x2 sr, f32x2 si)
{
    return fma2(sr, tr[k], mul2(si, ti[k]));
}

}  // namespace isrs
