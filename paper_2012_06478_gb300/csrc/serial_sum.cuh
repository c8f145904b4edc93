// serial_sum.cuh -- a chain of FP64 additions, each rounded, taken 32 at a time.
//
// t_i = t_{i-1} + x_i, rounded to nearest even at every step, is one FP64
// latency after another (about 110 clocks a step on GB300).  But while t stays
// inside one binade, its doubles are the multiples of one unit u, so t_i =
// t_{i-1} + (x_i rounded to a multiple of u), and the rounded x_i are integers
// whose prefix sums a warp forms in five exchanges.  That gives the chain's own
// values wherever no x_i lies half way between two multiples (whose rounding
// depends on t) and no t_i leaves the binade; the first step where that fails
// is added as it is, and the rest tried again from there.
//
// Host and device share the arithmetic, so that it is checked on the CPU.
#pragma once

#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace rms {
namespace chain {

__host__ __device__ __forceinline__ uint64_t bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    std::memcpy(&u, &x, 8);
    return u;
#endif
}
__host__ __device__ __forceinline__ double number(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    std::memcpy(&x, &u, 8);
    return x;
#endif
}

constexpr int64_t kLow = 1ll << 52;  // significands of normal doubles: [kLow, 2 kLow)

// x in units of t's last place, rounded to nearest.
struct Units {
    int64_t n;
    bool ok;     // not half way, t and x in range
    bool exact;  // nothing was rounded
};
__host__ __device__ __forceinline__ Units units_of(double t, double x)
{
    const uint64_t ub = bits(x) & 0x7FFFFFFFFFFFFFFFULL;
    const int e = (int)((bits(t) >> 52) & 0x7FFu), ex = (int)(ub >> 52);
    if (ub == 0) return Units{0, true, true};
    const int down = e - ex;
    if (e == 0 || e == 0x7FF || ex == 0 || ex == 0x7FF || down < 0) return Units{0, false, false};
    const int64_t m = (int64_t)(ub & 0x000FFFFFFFFFFFFFULL) | kLow;
    Units r{m, true, true};
    if (down > 0) {
        const int sh = down < 60 ? down : 60;  // below a quarter of the unit from 55 on
        const int64_t rest = m & ((1ll << sh) - 1), half = 1ll << (sh - 1);
        r.n = (m >> sh) + (rest > half ? 1 : 0);
        r.ok = rest != half;
        r.exact = rest == 0;
    }
    if (bits(x) >> 63) r.n = -r.n;
    return r;
}

// t's significand with its sign.
__host__ __device__ __forceinline__ int64_t significand(double t)
{
    const int64_t m = (int64_t)(bits(t) & 0x000FFFFFFFFFFFFFULL) | kLow;
    return (bits(t) >> 63) ? -m : m;
}

// Whether t plus n units in all, the last addend u among them, is the chain's
// value, given that the one before is: inside t's binade (at its lower end only
// if nothing was rounded: below it the units are finer).  t = 0 stays for x = 0.
__host__ __device__ __forceinline__ bool in_binade(double t, int64_t n, const Units &u)
{
    if (!u.ok) return false;
    if ((bits(t) << 1) == 0) return true;  // units_of took no x but 0
    const int64_t s = significand(t) + n, m = s < 0 ? -s : s;
    return ((s < 0) == (bool)(bits(t) >> 63)) && m < 2 * kLow && (m > kLow || (m == kLow && u.exact));
}
__host__ __device__ __forceinline__ double advanced(double t, int64_t n)
{
    if ((bits(t) << 1) == 0) return t;
    const int64_t s = significand(t) + n;
    const uint64_t m = (uint64_t)(s < 0 ? -s : s);
    return number((bits(t) & 0xFFF0000000000000ULL) | (m & 0x000FFFFFFFFFFFFFULL));
}

#ifdef __CUDACC__
// A warp's 32 steps: lane i < n gets t_i for its x_i; returns t after step n - 1.
__device__ __forceinline__ double serial_sums(double t, double x, int n, double &mine)
{
    const int lane = threadIdx.x & 31;
    int done = 0;
    for (int tries = 0; done < n; ++tries) {
        if (tries < 4) {
            const bool todo = lane >= done && lane < n;
            const Units u = todo ? units_of(t, x) : Units{0, true, true};
            int64_t s = u.n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t y = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += y;
            }
            const unsigned bad = __ballot_sync(0xffffffffu, todo && !in_binade(t, s, u));
            const int stop = bad ? __ffs((int)bad) - 1 : n;
            if (todo && lane < stop) mine = advanced(t, s);
            if (stop > done) t = __shfl_sync(0xffffffffu, mine, stop - 1);
            done = stop;
            if (done >= n) break;
        }
        t = t + __shfl_sync(0xffffffffu, x, done);
        if (lane == done) mine = t;
        ++done;
    }
    return t;
}
#endif

}  // namespace chain
}  // namespace rms
