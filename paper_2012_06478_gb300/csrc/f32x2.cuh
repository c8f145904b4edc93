// f32x2.cuh -- Blackwell's packed single-precision operations: two numbers an
// instruction, each rounded as the scalar operation rounds it.
#pragma once

#include <cstdint>

namespace rms {

// Two single-precision numbers at a time (Blackwell's packed operations).
struct F2 {
    uint64_t v;
};
__device__ __forceinline__ F2 pair_of(float x, float y)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float first(F2 a) { return __uint_as_float((uint32_t)a.v); }
__device__ __forceinline__ float second(F2 a) { return __uint_as_float((uint32_t)(a.v >> 32)); }
__device__ __forceinline__ F2 operator+(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b)
{
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

}  // namespace rms
