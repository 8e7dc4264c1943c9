// Packed FP32 pairs (sm_100 and later): one instruction for two independent
// operations with the rounding of the scalar ones.  A z-sum takes two steps at a
// time, so its multiply-adds cost half the issue slots; what then bounds it is
// the XU pipe (sin and cos at 16 lanes a clock, ex2 at 32).
#pragma once
#include <cuda_runtime.h>

namespace isrs {

struct f32x2 {
    unsigned long long v;
};

__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ f32x2 dup2(float a) { return pack2(a, a); }

__device__ __forceinline__ void unpack2(f32x2 x, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// sin and cos of 2 pi x for both halves
__device__ __forceinline__ void sincos_turn2(f32x2 x, float &s0, float &c0, float &s1, float &c1)
{
    float a, b;
    unpack2(mul2(x, dup2(6.283185307179586f)), a, b);
    __sincosf(a, &s0, &c0);
    __sincosf(b, &s1, &c1);
}

// As rev_fraction and phasor_rev_ff (quad_common.cuh): the fraction of (phi +
// phi_lo)(hi + lo) in revolutions; nphi =
// -phi.  Form 0: as written.  1: phi_lo = 0 and phases up to 2^30 revolutions, rounded
// twice, first to what `magic` (turn_magic) leaves.  2: phi_lo = 0, up to 2^20 revolutions.
template <int Form>
__device__ __forceinline__ f32x2 rev_fraction2(f32x2 phi, f32x2 nphi, f32x2 phi_lo, f32x2 hi, f32x2 lo,
                                               float magic = 12582912.0f)
{
    const f32x2 mg = dup2(12582912.0f), nm = dup2(-12582912.0f);
    f32x2 fr = Form == 1 ? fma2(phi, hi, add2(fma2(nphi, hi, dup2(magic)), dup2(-magic)))
                         : fma2(phi, hi, add2(fma2(nphi, hi, mg), nm));
    fr = fma2(phi, lo, fr);
    if constexpr (Form == 1) fr = add2(fr, add2(fma2(fr, dup2(-1.0f), mg), nm));
    if constexpr (Form == 0) fr = fma2(phi_lo, hi, fr);
    return fr;
}

}  // namespace isrs
