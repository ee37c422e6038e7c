// What the kernels share that form scores with mma.sync on fp16 operands: a row or centroid scaled by a power of two of its own, its
// measured rounding error, fp32 arithmetic in pairs, keys and candidate masks.
#pragma once

#include "cat_tc.cuh"

namespace cat {
namespace {

__device__ __forceinline__ void mma_16816(float (&c)[4], const uint4 a, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// Pairs of fp32 values in one 64-bit register: one instruction does both.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// exponent shift that brings m > 0 to [2^13, 2^14), clamped to +-100; 0 for zero or non-finite m
__device__ __forceinline__ int half_shift(float m)
{
    if (!(m > 0.f) || !(m < CUDART_INF_F)) return 0;
    int s = 13 - ((int)(__float_as_uint(m) >> 23) - 127);
    s = s > 100 ? 100 : s;
    return s < -100 ? -100 : s;
}
__device__ __forceinline__ float pow2i(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }
// two columns' fp16 roundings and what they leave, squared
__device__ __forceinline__ uint32_t round_pair(float a, float b, float &left2)
{
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    const float da = a - f.x, db = b - f.y;
    left2 = fmaf(da, da, fmaf(db, db, left2));
    return *reinterpret_cast<const uint32_t *>(&h);
}
__device__ __forceinline__ float sqrt_approx(float x)   // (2^-23 relative; callers have slack for more)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float max4(float4 a, float m)
{
    return fmaxf(fmaxf(m, fmaxf(fabsf(a.x), fabsf(a.y))), fmaxf(fabsf(a.z), fabsf(a.w)));
}

// Keys: scores with the centroid's index in the low seven bits; b1 and b2 are the smallest two.  (Those of an infinite or NaN score
// may get lost, but a row that has one also has a bound that decides nothing.)
__device__ __forceinline__ void take_key(float s, int k, float &b1, float &b2)
{
    const float key = __uint_as_float((__float_as_uint(s) & 0xFFFFFF80u) | (uint32_t)k);
    b2 = fminf(b2, fmaxf(b1, key));
    b1 = fminf(b1, key);
}
// ... of this lane and of the one `o` lanes off
__device__ __forceinline__ void merge_keys(int o, float &b1, float &b2)
{
    const float q1 = __shfl_xor_sync(0xffffffffu, b1, o), q2 = __shfl_xor_sync(0xffffffffu, b2, o);
    b2 = fminf(fminf(b2, q2), fmaxf(b1, q1));
    b1 = fminf(b1, q1);
}

// index of the lowest set bit, which it clears; -1 if none
template <int W>
__device__ __forceinline__ int pop_bit(uint32_t (&m)[W])
{
#pragma unroll
    for (int i = 0; i < W; ++i)
        if (m[i]) {
            const int k = 32 * i + __ffs(m[i]) - 1;
            m[i] &= m[i] - 1;
            return k;
        }
    return -1;
}

}  // namespace
}  // namespace cat
