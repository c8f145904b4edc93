// rms_readout.cuh -- the FP64 read-out's arithmetic in integers (Eq. 7).
//
// A term alpha e^{-i q g.Phi} costs sincos and two multiply-adds: some 45
// operations on GB300's FP64 pipe, which issues two a clock and SM.  Here the
// phase is a fraction of a turn in 64-bit fixed point, its sine and cosine
// come from a table of 4096 angles and a second-order step to the angle, and
// the sums are 64-bit integers (exact): 20 products of 32-bit words in place
// of the FP64 operations.
//
// Precision, against sincos and FP64 sums: the phase is within 2^-57 of the
// largest |phase| P of 64 walkers (a double's last place is 2^-53 of it), the
// term's parts within 2^-51.8 + 2^-55 P of their largest alpha (2^-55 in the mean
// square at |phase| < 1), its rounding is not biased and the sum over 64 walkers is
// exact, so a signal is nearer to its exact value than FP64 sums over 4096
// walkers bring it.  Phases too small (below 2^-6
// rad), too large (above 2^20 rad) or not finite, and alphas that are not
// finite or all zero, take sincos in FP64 (rms_readout.cu).
//
// Host and device share the code, so that the arithmetic is checked on the CPU.
#pragma once

#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace rms {
namespace fix {

constexpr int kAngles = 4096;  // table angles a turn, at (k + 1/2) / 4096

struct Words {  // a signed 64-bit number hi 2^32 + lo with a signed low word
    int32_t hi, lo;
};
__host__ __device__ __forceinline__ Words words(int64_t x)
{
    const int32_t lo = (int32_t)(uint32_t)(uint64_t)x;
    return Words{(int32_t)((x - lo) >> 32), lo};
}
struct alignas(16) Angle {  // cosine and sine, 62 fraction bits
    Words c, s;
};

__host__ __device__ __forceinline__ int64_t mul_ss(int32_t a, int32_t b) { return (int64_t)a * b; }
__host__ __device__ __forceinline__ int64_t mul_uu(uint32_t a, uint32_t b) { return (int64_t)((uint64_t)a * b); }
__host__ __device__ __forceinline__ int32_t hi32(int64_t x) { return (int32_t)(x >> 32); }
__host__ __device__ __forceinline__ uint32_t lo32(int64_t x) { return (uint32_t)(uint64_t)x; }
__host__ __device__ __forceinline__ uint64_t mulhi_u64(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
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
__host__ __device__ __forceinline__ uint64_t double_word(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    std::memcpy(&u, &x, 8);
    return u;
#endif
}
__host__ __device__ __forceinline__ float fma_f(float a, float b, float c)
{
#ifdef __CUDA_ARCH__
    return fmaf(a, b, c);
#else
    return __builtin_fmaf(a, b, c);
#endif
}

// The significand of a finite |x| shifted so that a number of biased exponent
// `em`, at least x's own, has `top` bits (top >= 53).
__host__ __device__ __forceinline__ int64_t scaled(double x, int em, int top)
{
    const uint64_t u = double_word(x);
    const int e = (int)((u >> 52) & 0x7FFu);
    const uint64_t m = (u & 0x000FFFFFFFFFFFFFULL) | (e ? 0x0010000000000000ULL : 0ULL);
    const int sh = e - em + (top - 53);
    const int64_t r = sh >= 0 ? (int64_t)(m << sh) : (sh > -64 ? (int64_t)(m >> -sh) : 0);
    return (u >> 63) ? -r : r;
}

// q / 2 pi of a normal q > 0 of biased exponent eq: Q 2^(eq - 1087).
__host__ __device__ __forceinline__ int64_t turns_of(double q)
{
    const uint64_t m = (double_word(q) & 0x000FFFFFFFFFFFFFULL) | 0x0010000000000000ULL;
    return (int64_t)(mulhi_u64(m << 11, 0xA2F9836E4E441529ULL) >> 1);  // 2 / pi in 64 bits
}

// Whether a combination of amplitude q may take phases q x, |x| of biased
// exponent em at most, as turns; then with X = scaled(x, em, 62) and Q (its
// first words) the turns' fraction in 64 bits is the high word of X Q << shift.
struct Scale {
    int32_t Qh, Ql, shift;
    bool ok;
};
__host__ __device__ __forceinline__ Scale scale_of(double q, int64_t Q, int em)
{
    const int eq = (int)(double_word(q) >> 52);  // a negative q or a NaN falls out of the range
    const int e2 = em + eq - 2046;               // 2^e2 <= q |x|max < 2^(e2 + 2)
    Scale r;
    r.ok = em > 0 && em < 0x7FF && eq > 0 && eq < 0x7FF && e2 >= -6 && e2 <= 20;
    const int sh = e2 + 3;
    const Words w = words(sh < 0 ? Q >> (r.ok ? -sh : 0) : Q);
    r.Qh = w.hi;
    r.Ql = w.lo;
    r.shift = r.ok && sh > 0 ? sh : 0;
    return r;
}

// Adds alpha cos(phi) and alpha sin(phi), phi = 2 pi turns of X Q, to the sums
// (56 fraction bits); alpha in 58 bits.  The turns are rounded, and the low words'
// product that is left out averages to zero, as both have signs: rounded down, the
// phases of all walkers were 2^-57 to 2^-58 too small together, which an imaginary
// part near zero of 3e6 walkers showed (3.9e-15 of it off, 2.5e-15 with sincos; now
// 4e-16).
__host__ __device__ __forceinline__ void add_term(Words X, const Scale &q, Words al, const Angle *table, int64_t &re,
                                                  int64_t &im)
{
    const int64_t mid = mul_ss(X.hi, q.Ql) + mul_ss(X.lo, q.Qh) + 0x80000000LL;
    const uint64_t T = (uint64_t)(mul_ss(X.hi, q.Qh) + hi32(mid)) << q.shift;  // turns, 64 fraction bits
    const Angle a = table[T >> 52];
    // the angle from the table's: F 2^-64 of 2 pi / 4096, R = r 2^72 radians, |r| < 2^-10.3
    const int64_t F = (int64_t)((T << 12) ^ 0x8000000000000000ULL);
    constexpr uint32_t kKh = 0x6487ED51u;  // pi / 8 in 64 bits
    constexpr int32_t kKl = 0x10B4611A;
    const int64_t midR = mul_ss(hi32(F), kKl) + mul_uu(lo32(F), kKh);
    const int64_t R = mul_ss(hi32(F), (int32_t)kKh) + hi32(midR);
    // cos r - 1 = -(r^2/2 - r^4/24) with 52 fraction bits; sin r = r - r^3/6 + r^5/120
    // with 72: the terms beyond the first in single precision, rounded to integers by
    // adding 1.5 2^23
    const int32_t Rh = hi32(R);
    const int64_t r2 = mul_ss(Rh, Rh) + 4 * (int64_t)hi32(mul_ss(Rh, (int32_t)(lo32(R) >> 1)));
    const float rf = (float)Rh;
    const float a2 = (rf * rf) * 0x1p-64f;  // r^2 2^16
    const int32_t r4 = float_word(fma_f(a2 * a2, 0x1p31f / 24.0f, 12582912.0f)) - 0x4B400000;
    const int32_t m = -(int32_t)((r2 + mul_ss(r4, -(1 << 18)) + (1 << 28)) >> 29);
    const int32_t r3 = float_word(fma_f(rf * a2, fma_f(a2, -0x1p-17f / 120.0f, 1.0f / 12.0f), 12582912.0f)) -
                       (0x4B400000 + (1 << 14));
    const int64_t s = R + mul_ss(r3, -(1 << 17));  // sin r + 2^31, so that the low word is signed
    const int32_t sh = hi32(s), sl = (int32_t)(lo32(s) ^ 0x80000000u);
    // cos(a + r) = C + (C (cos r - 1) - S sin r), sin(a + r) = S + (S (cos r - 1) + C sin r)
    const int64_t zc = mul_ss(a.c.hi, m) + (-(mul_ss(a.s.hi, sl) + mul_ss(a.s.lo, sh)) >> 20);
    const int64_t zs = mul_ss(a.s.hi, m) + ((mul_ss(a.c.hi, sl) + mul_ss(a.c.lo, sh)) >> 20);
    const int64_t yc = (zc >> 12) - mul_ss(a.s.hi, sh);
    const int64_t ys = mul_ss(a.c.hi, sh) + (zs >> 12);
    const int64_t cs = (yc >> 8) + a.c.lo + (int64_t)((uint64_t)(uint32_t)a.c.hi << 32);
    const int64_t sn = (ys >> 8) + a.s.lo + (int64_t)((uint64_t)(uint32_t)a.s.hi << 32);
    const int64_t mc = mul_ss(al.lo, hi32(cs)) + mul_uu((uint32_t)al.hi, lo32(cs)) + 0x80000000LL;
    const int64_t ms = mul_ss(al.lo, hi32(sn)) + mul_uu((uint32_t)al.hi, lo32(sn)) + 0x80000000LL;
    re += mul_ss(al.hi, hi32(cs)) + hi32(mc);
    im += mul_ss(al.hi, hi32(sn)) + hi32(ms);
}

__host__ __device__ __forceinline__ void add_term(int64_t X, const Scale &q, Words al, const Angle *table, int64_t &re,
                                                  int64_t &im)
{
    add_term(words(X), q, al, table, re, im);
}

// Cosines and sines of the first octant's table angles, (2j + 1) pi / 4096 for
// j < 512, by their Taylor series in 63-bit fixed point.
struct Octant {
    int64_t c[kAngles / 8], s[kAngles / 8];
};
constexpr uint64_t mulhi_const(uint64_t a, uint64_t b)
{
    const uint64_t al = a & 0xFFFFFFFFu, ah = a >> 32, bl = b & 0xFFFFFFFFu, bh = b >> 32;
    const uint64_t m1 = ah * bl + ((al * bl) >> 32), m2 = al * bh + (m1 & 0xFFFFFFFFu);
    return ah * bh + (m1 >> 32) + (m2 >> 32);
}
constexpr Octant octant_table()
{
    Octant t{};
    constexpr uint64_t kOne = 1ull << 63;
    for (int j = 0; j < kAngles / 8; ++j) {
        const uint64_t n = (uint64_t)(2 * j + 1), pi62 = 0xC90FDAA22168C235ull;
        const uint64_t x = (mulhi_const(pi62, n) << 53) | ((pi62 * n) >> 11);  // the angle, 63 fraction bits
        const uint64_t x2 = mulhi_const(x, x);                                  // 62
        uint64_t c = kOne, s = kOne;
        for (uint64_t k = 10; k >= 1; --k) {  // 1 - x^2 / ((2k - 1) 2k) (...), and likewise for sin x / x
            c = kOne - 4 * (mulhi_const(x2, c) / ((2 * k - 1) * (2 * k)));
            s = kOne - 4 * (mulhi_const(x2, s) / ((2 * k) * (2 * k + 1)));
        }
        t.c[j] = (int64_t)((c + 1) >> 1);
        t.s[j] = (int64_t)(mulhi_const(x, s));  // 63 + 63 - 64
    }
    return t;
}

// Table angle k from the first octant's.
__host__ __device__ __forceinline__ Angle angle_of(const Octant &t, int k)
{
    const int quadrant = k >> 10, i = k & 1023;
    const bool swap = i >= 512;
    const int j = swap ? 1023 - i : i;
    const int64_t x = swap ? t.s[j] : t.c[j], y = swap ? t.c[j] : t.s[j];  // cos, sin in the first quadrant
    int64_t c = (quadrant & 1) ? -y : x, s = (quadrant & 1) ? x : y;
    if (quadrant >= 2) {
        c = -c;
        s = -s;
    }
    return Angle{words(c), words(s)};
}

}  // namespace fix
}  // namespace rms
