// gc_f32x2.cuh -- packed FP32 arithmetic (sm_100+) and the sine and cosine built on it.
#pragma once

#include <cuda_runtime.h>

namespace gcp {

// Two FP32 values in one 64-bit register and the packed f32x2 arithmetic of sm_100+ (two
// independent IEEE operations per instruction, the same results as two scalar ones).
__device__ __forceinline__ unsigned long long p2_sub(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ unsigned long long p2_fma(unsigned long long a, unsigned long long b,
                                                     unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ unsigned long long p2_bcast(float x)
{
    unsigned long long d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
    return d;
}

__device__ __forceinline__ unsigned long long p2_pack(float lo, float hi)
{
    unsigned long long d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}

__device__ __forceinline__ unsigned long long p2_mul(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ void p2_split(unsigned long long v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// Sine and cosine of two values at once, for |z| <= kSincosMax: Cody and Waite's reduction
// r = z - q pi/2 (q = z 2/pi rounded to an integer by adding 1.5 2^23, pi/2 in three parts)
// and minimal-error polynomials on |r| <= pi/4 (fitted by sincos_coeffs.py). At most 1.55 ulp
// from the exact values, 16 % of them not the correctly rounded ones (the library's bound is
// 2 ulp). 18 instructions a value, half of the library's, without its branch for large
// arguments: the caller sends those elsewhere.
constexpr float kSincosMax = 30000.0f;

__device__ __forceinline__ void sincos2(unsigned long long z, float (&sn)[2], float (&cs)[2])
{
    const unsigned long long t = p2_fma(z, p2_bcast(6.366197467e-01f), p2_bcast(12582912.0f));
    const unsigned long long q = p2_sub(t, p2_bcast(12582912.0f));
    unsigned long long r = p2_fma(q, p2_bcast(-1.570796371e+00f), z);
    r = p2_fma(q, p2_bcast(4.371138829e-08f), r);
    r = p2_fma(q, p2_bcast(1.715099417e-15f), r);
    const unsigned long long r2 = p2_mul(r, r);
    unsigned long long s = p2_fma(p2_bcast(-1.949563593e-04f), r2, p2_bcast(8.331978694e-03f));
    s = p2_fma(s, r2, p2_bcast(-1.666665077e-01f));
    s = p2_fma(p2_mul(r, r2), s, r);
    unsigned long long c = p2_fma(p2_bcast(2.443845005e-05f), r2, p2_bcast(-1.388736768e-03f));
    c = p2_fma(c, r2, p2_bcast(4.166664556e-02f));
    c = p2_fma(c, r2, p2_bcast(-0.5f));
    c = p2_fma(c, r2, p2_bcast(1.0f));
    float tk[2], s2[2], c2[2];
    p2_split(t, tk[0], tk[1]);
    p2_split(s, s2[0], s2[1]);
    p2_split(c, c2[0], c2[1]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const unsigned k = __float_as_uint(tk[i]); // low bits: q modulo 4
        const float a = (k & 1u) ? c2[i] : s2[i], b = (k & 1u) ? s2[i] : c2[i];
        sn[i] = __uint_as_float(__float_as_uint(a) ^ ((k << 30) & 0x80000000u));
        cs[i] = __uint_as_float(__float_as_uint(b) ^ (((k + 1u) << 30) & 0x80000000u));
    }
}

} // namespace gcp
