// f32x2.cuh -- Blackwell's packed single-precision operations: two numbers an
// instruction, each rounded as the scalar operation rounds it; and sums of such
// pairs that are exact but for the last places of a double.
//
// The host build (for the host-side checks) takes the scalar operations.
#pragma once

#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#include <cmath>
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace rms {

// Two single-precision numbers at a time (Blackwell's packed operations).
struct F2 {
    uint64_t v;
};
__host__ __device__ __forceinline__ int32_t float_word(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_int(x);
#else
    int32_t u;
    std::memcpy(&u, &x, 4);
    return u;
#endif
}
__host__ __device__ __forceinline__ float word_float(uint32_t u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float x;
    std::memcpy(&x, &u, 4);
    return x;
#endif
}
__host__ __device__ __forceinline__ F2 pair_of(float x, float y)
{
    F2 r;
#ifdef __CUDA_ARCH__
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
#else
    r.v = (uint64_t)(uint32_t)float_word(y) << 32 | (uint32_t)float_word(x);
#endif
    return r;
}
__host__ __device__ __forceinline__ float first(F2 a) { return word_float((uint32_t)a.v); }
__host__ __device__ __forceinline__ float second(F2 a) { return word_float((uint32_t)(a.v >> 32)); }
__host__ __device__ __forceinline__ F2 operator+(F2 a, F2 b)
{
#ifdef __CUDA_ARCH__
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
#else
    return pair_of(first(a) + first(b), second(a) + second(b));
#endif
}
__host__ __device__ __forceinline__ F2 operator-(F2 a, F2 b)
{
#ifdef __CUDA_ARCH__
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
#else
    return pair_of(first(a) - first(b), second(a) - second(b));
#endif
}
__host__ __device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
#ifdef __CUDA_ARCH__
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
#else
    return pair_of(fmaf(first(a), first(b), first(c)), fmaf(second(a), second(b), second(c)));
#endif
}

// Sums of at most 64 pairs of numbers of at most 1: each is split at 2^-16 and
// 2^-33 by adding it to a number of fixed exponent, whose last place that is, so
// that all sums but the last level's (below 2^-28) are exact.  Seven packed
// additions, in place of two on the FP64 pipe.
struct SplitSum {
    static constexpr float kTop = 192.0f, kMid = 0x1.8p-10f;
    F2 a = pair_of(kTop, kTop), b = pair_of(kMid, kMid), c = pair_of(0.0f, 0.0f);
    __host__ __device__ __forceinline__ void add(F2 x)
    {
        const F2 ta = a + x;
        x = x - (ta - a);
        a = ta;
        const F2 tb = b + x;
        c = c + (x - (tb - b));
        b = tb;
    }
    // one sum with 48 fraction bits
    static __host__ __device__ __forceinline__ int64_t fixed(float a, float b, float c)
    {
#ifdef __CUDA_ARCH__
        const int32_t last = __float2int_rn(c * 0x1p48f);
#else
        const int32_t last = (int32_t)std::lrint(c * 0x1p48f);
#endif
        return ((int64_t)(float_word(a) - float_word(kTop)) << 32) +
               ((int64_t)(float_word(b) - float_word(kMid)) << 15) + last;
    }
};

}  // namespace rms
