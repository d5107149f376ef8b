// rick_screen.cuh -- the w-term phase screen of a pixel (Eq. 1) in float-pair
// arithmetic, shared by the kernels that apply it (rick_stack.cu,
// rick_strip.cu).
#pragma once

#include "rick_internal.cuh"

namespace rick {

struct FF {
    float hi, lo;
};

// a * b for float pairs, lo terms to first order.
__device__ __forceinline__ FF ff_mul(FF a, FF b)
{
    const float p = a.hi * b.hi;
    const float e = __fmaf_rn(a.hi, b.hi, -p);
    return FF{p, e + __fmaf_rn(a.hi, b.lo, a.lo * b.hi)};
}

// exp(2 pi i (hi + lo)) with the integer part of hi removed exactly.
__device__ __forceinline__ float2 turns_to_phasor(float hi, float lo)
{
    const float f = (hi - rintf(hi)) + lo;
    float s, c;
    sincospif(2.0f * f, &s, &c);
    return make_float2(c, s);
}

// Phase in turns of plane k: A + k B, A = wb (n-1), B = dw (n-1).
__device__ __forceinline__ float2 screen(FF A, FF B, int k)
{
    const float kf = (float)k;
    const float kb = kf * B.hi;
    const float kbe = __fmaf_rn(kf, B.hi, -kb);
    const float s = A.hi + kb;                 // two-sum of A.hi + kb
    const float bb = s - A.hi;
    const float err = (A.hi - (s - bb)) + (kb - bb);
    return turns_to_phasor(s, err + kbe + A.lo + kf * B.lo);
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

struct PixelScreen {
    FF A, B;
    float nm1;
    bool sky;
};

__device__ __forceinline__ PixelScreen pixel_screen(const StackArgs& a, int x, int y)
{
    PixelScreen ps;
    const int ix = x - a.n / 2, iy = y - a.n / 2;
    const int q = ix * ix + iy * iy;                        // exact integer
    const float qh = (float)q;
    const float ql = (float)(q - (int)qh);
    const FF r2 = ff_mul(FF{qh, ql}, FF{a.dl2_hi, a.dl2_lo});  // l^2 + m^2
    ps.sky = r2.hi < 1.0f;
    // n - 1 = -r2 / (2 + (n - 1)); eps is a binary32 first guess of n - 1
    const float eps = ps.sky ? -r2.hi / (1.0f + sqrtf(1.0f - r2.hi)) : 0.0f;
    const float he = 0.5f * eps;
    FF nm1;
    nm1.hi = -0.5f * r2.hi;
    nm1.lo = -0.5f * r2.lo + (0.5f * r2.hi) * (he / (1.0f + he));
    ps.nm1 = nm1.hi + nm1.lo;
    ps.A = ff_mul(FF{a.wb_hi, a.wb_lo}, nm1);
    ps.B = ff_mul(FF{a.dw_hi, a.dw_lo}, nm1);
    return ps;
}

}  // namespace rick
