// rick_dft.cuh -- short DFTs in registers (2, 4, 8 and 16 points, natural
// order in and out, either exponent sign) of values as cpx, one 64-bit register
// pair whose additions are packed binary32 instructions: half the issue slots
// of the scalar form at the same arithmetic rate (measured on
// a GB300: 120 scalar or 2 x 64 packed multiply-adds per clock and SM).
#pragma once

#include <cuda_runtime.h>

namespace rick {

// ------------------------------------------------------------- one value

__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 c_mul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// ------------------------------------------------ one value in a register pair

// a pair of binary32 values in one 64-bit register pair
struct f2 {
    unsigned long long v;
};

__device__ __forceinline__ f2 f2_make(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 f2_get(f2 a)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
    return r;
}
__device__ __forceinline__ f2 f2_dup(float a) { return f2_make(a, a); }
__device__ __forceinline__ f2 f2_add(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// a - b: the product with -1 is exact, so this rounds once like a subtraction
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) { return f2_fma(b, f2_dup(-1.0f), a); }

// a complex value in one register pair: additions are packed (one instruction
// each), products and rotations work on its halves
struct cpx {
    f2 v;
};

__device__ __forceinline__ cpx cpx_make(float re, float im) { return cpx{f2_make(re, im)}; }
__device__ __forceinline__ float2 cpx_get(cpx a) { return f2_get(a.v); }
__device__ __forceinline__ cpx c_add(cpx a, cpx b) { return cpx{f2_add(a.v, b.v)}; }
__device__ __forceinline__ cpx c_sub(cpx a, cpx b) { return cpx{f2_sub(a.v, b.v)}; }
__device__ __forceinline__ cpx c_mul(cpx a, float2 w)
{
    const float2 x = cpx_get(a);
    return cpx_make(x.x * w.x - x.y * w.y, x.x * w.y + x.y * w.x);
}

// ---------------------------------------------------- additions with (s i)

// x + s i y and x - s i y
template <int SIGN>
__device__ __forceinline__ void c_rot_pair(cpx x, cpx y, cpx& p, cpx& m)
{
    const float2 u = cpx_get(x), w = cpx_get(y);
    const cpx a = cpx_make(u.x - w.y, u.y + w.x), b = cpx_make(u.x + w.y, u.y - w.x);
    p = SIGN > 0 ? a : b;
    m = SIGN > 0 ? b : a;
}

// ------------------------------------------------------------------- DFTs

template <int SIGN, typename C>
__device__ __forceinline__ void dft2(C& a, C& b)
{
    const C t = a;
    a = c_add(t, b);
    b = c_sub(t, b);
}

template <int SIGN, typename C>
__device__ __forceinline__ void dft4(C& x0, C& x1, C& x2, C& x3)
{
    const C a0 = c_add(x0, x2), a2 = c_sub(x0, x2);
    const C a1 = c_add(x1, x3), a3 = c_sub(x1, x3);
    x0 = c_add(a0, a1);
    x2 = c_sub(a0, a1);
    c_rot_pair<SIGN>(a2, a3, x1, x3);
}

// w_8^k, k = 1, 3 (w_8^2 = s i)
constexpr float kR2 = 0.70710678118654752f;

template <int SIGN, typename C>
__device__ __forceinline__ void dft8(C (&v)[8])
{
    // two 4-point transforms over the even and odd samples and one radix-2 pass
    C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<SIGN>(e0, e1, e2, e3);
    dft4<SIGN>(o0, o1, o2, o3);
    // twiddles w_8^k on the odd transform
    const float s = (float)SIGN;
    o1 = c_mul(o1, make_float2(kR2, s * kR2));
    o3 = c_mul(o3, make_float2(-kR2, s * kR2));
    v[0] = c_add(e0, o0);
    v[4] = c_sub(e0, o0);
    v[1] = c_add(e1, o1);
    v[5] = c_sub(e1, o1);
    c_rot_pair<SIGN>(e2, o2, v[2], v[6]);
    v[3] = c_add(e3, o3);
    v[7] = c_sub(e3, o3);
}

// cos and sin of 2 pi k / 16, k = 0 .. 9
__device__ __forceinline__ float2 w16(int k, int sign)
{
    const float c[10] = {1.0f, 0.92387953251128676f, 0.70710678118654752f, 0.38268343236508977f, 0.0f,
                         -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128676f, -1.0f,
                         -0.92387953251128676f};
    const float s[10] = {0.0f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128676f, 1.0f,
                         0.92387953251128676f, 0.70710678118654752f, 0.38268343236508977f, 0.0f,
                         -0.38268343236508977f};
    return make_float2(c[k], sign * s[k]);
}

template <int SIGN, typename C>
__device__ __forceinline__ void dft16(C (&v)[16])
{
    // 16 = 4 x 4, in place: sample 4 c1 + c2; first 4-point DFTs over c1 (for
    // each c2), times w_16^(c2 j1), then over c2 (for each j1): output j1 + 4 j2
#pragma unroll
    for (int c2 = 0; c2 < 4; ++c2) {
        dft4<SIGN>(v[c2], v[4 + c2], v[8 + c2], v[12 + c2]);
#pragma unroll
        for (int j1 = 1; j1 < 4; ++j1)
            if (c2 > 0 && c2 * j1 != 4) v[4 * j1 + c2] = c_mul(v[4 * j1 + c2], w16(c2 * j1, SIGN));
    }
    // v[4 j1 + c2]; the factor w_16^4 = s i of (c2, j1) = (2, 2) is left to its additions
    C o[16];
#pragma unroll
    for (int j1 = 0; j1 < 4; ++j1) {
        C x0 = v[4 * j1], x1 = v[4 * j1 + 1], x2 = v[4 * j1 + 2], x3 = v[4 * j1 + 3];
        if (j1 == 2) {
            C a0, a2;
            c_rot_pair<SIGN>(x0, x2, a0, a2);
            const C a1 = c_add(x1, x3), a3 = c_sub(x1, x3);
            o[j1] = c_add(a0, a1);
            o[j1 + 8] = c_sub(a0, a1);
            c_rot_pair<SIGN>(a2, a3, o[j1 + 4], o[j1 + 12]);
            continue;
        }
        dft4<SIGN>(x0, x1, x2, x3);
        o[j1] = x0;
        o[j1 + 4] = x1;
        o[j1 + 8] = x2;
        o[j1 + 12] = x3;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = o[k];
}

template <int R, int SIGN, typename C>
__device__ __forceinline__ void dft_small(C (&v)[R])
{
    if constexpr (R == 2) {
        dft2<SIGN>(v[0], v[1]);
    } else if constexpr (R == 4) {
        dft4<SIGN>(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 8) {
        dft8<SIGN>(v);
    } else if constexpr (R == 16) {
        dft16<SIGN>(v);
    }
}

}  // namespace rick
