// soft_fp64.cuh -- correctly rounded FP64 division, square root and
// multiplication built on the integer ALU, bit-identical to IEEE 754
// round-to-nearest-even.
//
// Why: GB300's FP64 pipe issues about two operations per clock per SM, a
// sixty-fourth of its FP32 rate, and an FP64 division or square root is a
// sequence of several of them.  The plain FP64 form of the walker step keeps
// that pipe busy; computing its quotients and its square root with 64-bit
// integer arithmetic (multiplies on the integer pipe, a single-precision
// seed) gives the same bits at a fraction of the pipe time.
//
// Method: a reciprocal (or square root and its reciprocal) seed from single
// precision, one Newton-Raphson step in fixed point (for the reciprocal x' = x +
// x(1 - b x); for the square root q' = q + (X - q^2)/(2q) with 1/(2q) from the
// seed), then exact integer remainders that bring the result to its last unit
// and decide the rounding -- the classical scheme of, e.g.,
// Muller et al., Handbook of Floating-Point Arithmetic (2nd ed., 2018),
// ch. 4 (Newton-Raphson based division and square root) with the final
// correction by the remainder.  Division and square root have no exact
// half-way cases, but the rounding rule is written out in full anyway.
//
// Each function handles the operands the walker step produces -- finite,
// normal, with a normal result -- and returns false for anything else, so
// the caller falls back to the hardware operation for zeros, subnormals,
// infinities, NaNs and out-of-range results.  Host and device share the
// code: the host build (for the host-side checks) replaces the single-precision
// seeds, the funnel shift and the carry chain by their exact definitions.
#pragma once

#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace rms {
namespace sfp {

constexpr uint64_t kMant = 0x000FFFFFFFFFFFFFULL;  // the 52 stored mantissa bits
constexpr uint64_t kHidden = 0x0010000000000000ULL;  // 2^52

__host__ __device__ __forceinline__ uint64_t bits_of(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    std::memcpy(&u, &x, 8);
    return u;
#endif
}

__host__ __device__ __forceinline__ double double_of(uint64_t u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    std::memcpy(&x, &u, 8);
    return x;
#endif
}

__host__ __device__ __forceinline__ uint32_t float_bits(float x)
{
#ifdef __CUDA_ARCH__
    return (uint32_t)__float_as_uint(x);
#else
    uint32_t u;
    std::memcpy(&u, &x, 4);
    return u;
#endif
}

// single-precision reciprocal and square root, correctly rounded on both sides
__host__ __device__ __forceinline__ float rcp_rn(float x)
{
#ifdef __CUDA_ARCH__
    return __frcp_rn(x);
#else
    return 1.0f / x;
#endif
}
__host__ __device__ __forceinline__ float sqrt_rn(float x)
{
#ifdef __CUDA_ARCH__
    return __fsqrt_rn(x);
#else
    return __builtin_sqrtf(x);
#endif
}

// a / b for a and b known to be normal and positive, with a quotient known to be
// normal (the caller's ranges guarantee it).
__host__ __device__ __forceinline__ double div_normal(double a, double b)
{
    const uint64_t ua = bits_of(a), ub = bits_of(b);
    const int32_t ea = (int32_t)(ua >> 52), eb = (int32_t)(ub >> 52);
    const uint64_t A = (ua & kMant) | kHidden, B = (ub & kMant) | kHidden;  // [2^52, 2^53)
    const bool ge = A >= B;
    const int32_t e = ea - eb + 1022 + (ge ? 1 : 0);  // biased exponent of the quotient
    // X0 ~ 2^76 / B in 24 bits, from the single-precision reciprocal of B's top 24
    // (relative error below 2^-22)
    const float fr = rcp_rn((float)(uint32_t)(B >> 29));  // in (2^-24, 2^-23]
    const uint32_t fb = float_bits(fr);
    const uint32_t X0 = ((fb & 0x7FFFFFu) | 0x800000u) << ((fb >> 23) - 103u);  // fr 2^47
    // one Newton step: X1 ~ 2^108 / B in (2^55, 2^56], relative error below 2^-44, with
    // e = 2^55 - B X0 / 2^21, |e| < 2^33
    const uint32_t Bh = (uint32_t)(B >> 21), Bl = (uint32_t)B & 0x1FFFFFu;
    const int64_t e0 = (int64_t)(0x0080000000000000ULL - ((uint64_t)Bh * X0 + (((uint64_t)Bl * X0) >> 21)));
    const uint64_t X1 = ((uint64_t)X0 << 32) + (uint64_t)(((int64_t)(int32_t)X0 * (int32_t)(e0 >> 3)) >> 20);
    // Q = floor(A 2^s / B), s = 52 (A >= B) or 53: A X1 / 2^(108 - s) is within 2^9 of
    // it; its exact remainder (below 2^62) over B brings it within one unit, and
    // the remainder of that fixes it.  Products of 32-bit words throughout: a second
    // Newton step in 64-bit ones takes twice as many
    const int s = ge ? 52 : 53;
    const uint64_t As = A << s;  // mod 2^64
    const uint32_t Ah = (uint32_t)(A >> 21), Al = (uint32_t)A << 11;  // A 2^11
    const uint32_t Xh = (uint32_t)(X1 >> 25), Xl = (uint32_t)X1 << 7;  // X1 2^7
    // (A 2^11) (X1 2^7) / 2^64, without the low words' product
    const uint64_t P = (uint64_t)Ah * Xh + (((uint64_t)Ah * Xl) >> 32) + (((uint64_t)Al * Xh) >> 32);
    uint64_t Q = P >> (ge ? 10 : 9);
    int64_t R = (int64_t)(As - Q * B);
    const int32_t dq = (int32_t)(((int64_t)(int32_t)(R >> 32) * (int32_t)(X1 >> 26)) >> 50);  // R X1 / 2^108
    Q += (uint64_t)(int64_t)dq;
    R -= (int64_t)dq * (int64_t)B;
    if (R < 0) {
        --Q;
        R += (int64_t)B;
    } else if (R >= (int64_t)B) {
        ++Q;
        R -= (int64_t)B;
    }
    // round to nearest, ties to even (no ties occur for a quotient): up iff
    // 2R > B, or 2R == B and Q odd
    const uint64_t up = ((uint64_t)R << 1) + (Q & 1ULL) > B ? 1ULL : 0ULL;
    return double_of((((uint64_t)(e - 1)) << 52) + Q + up);  // Q carries the hidden bit; a carry moves into the exponent
}

// a / b for a >= +0 and b > +0 (sign bits clear).  Returns false when a or b
// is subnormal, infinite or NaN, or the quotient leaves the normal range
// (except an overflow to infinity by rounding, which is the IEEE result).
__host__ __device__ __forceinline__ bool div_pos(double a, double b, double &q)
{
    const uint64_t ua = bits_of(a), ub = bits_of(b);
    if (ua == 0) {  // 0 / b = +0
        q = 0.0;
        return true;
    }
    const int32_t ea = (int32_t)(ua >> 52), eb = (int32_t)(ub >> 52);
    if ((uint32_t)(ea - 1) >= 0x7FEu || (uint32_t)(eb - 1) >= 0x7FEu) return false;
    const int32_t e = ea - eb + 1022 + ((ua & kMant) >= (ub & kMant) ? 1 : 0);
    if ((uint32_t)(e - 1) >= 0x7FEu) return false;
    q = div_normal(a, b);
    return true;
}

// A B of two 53-bit significands in two words: their high words have 21 bits, so
// the middle products add up without a carry -- four products of 32-bit words
// with their additions, where separate low and high products take seven and the
// carries.
__host__ __device__ __forceinline__ void mul_significands(uint64_t A, uint64_t B, uint64_t &lo, uint64_t &hi)
{
    const uint32_t a0 = (uint32_t)A, a1 = (uint32_t)(A >> 32), b0 = (uint32_t)B, b1 = (uint32_t)(B >> 32);
    const uint64_t p = (uint64_t)a0 * b0;
    const uint64_t m = (uint64_t)a0 * b1 + ((uint64_t)a1 * b0 + (p >> 32));
    hi = (uint64_t)a1 * b1 + (m >> 32);
    lo = (m << 32) | (uint32_t)p;
}

// The upper word of (hi 2^32 + lo) 2^s, s < 32.
__host__ __device__ __forceinline__ uint32_t funnel_left(uint32_t lo, uint32_t hi, uint32_t s)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_l(lo, hi, s);
#else
    return (uint32_t)(((((uint64_t)hi << 32) | lo) << s) >> 32);
#endif
}

// m1 2^32 + m0 + head 2^32, plus the carry of (r1 2^32 + r0) + (x1 2^32 + x0).
__host__ __device__ __forceinline__ double add_carry_of(uint32_t r0, uint32_t r1, uint32_t x0, uint32_t x1, uint32_t m0,
                                                        uint32_t m1, uint32_t head)
{
#ifdef __CUDA_ARCH__
    uint32_t p0, p1;
    asm("{\n\t.reg .u32 t;\n\t"
        "add.cc.u32 t, %2, %3;\n\t"
        "addc.cc.u32 t, %4, %5;\n\t"
        "addc.cc.u32 %0, %6, 0;\n\t"
        "addc.u32 %1, %7, %8;\n\t}"
        : "=r"(p0), "=r"(p1)
        : "r"(r0), "r"(x0), "r"(r1), "r"(x1), "r"(m0), "r"(m1), "r"(head));
    return __hiloint2double((int)p1, (int)p0);
#else
    const uint64_t c0 = ((uint64_t)r0 + x0) >> 32, c1 = ((uint64_t)r1 + x1 + c0) >> 32;
    const uint64_t p0 = (uint64_t)m0 + c1;
    const uint32_t p1 = m1 + head + (uint32_t)(p0 >> 32);
    return double_of(((uint64_t)p1 << 32) | (uint32_t)p0);
#endif
}

// The product of the significands of a and b rounded to 53 bits, given the
// biased exponent e of the result: the 106-bit product is exact in two words,
// `top` says that it is at least 2^105; rounding is to nearest with ties to even
// (products do have ties).  The kept bits and, left-aligned, the ones below them
// come from funnel shifts; the carry of the latter plus one half -- less one unit
// where the kept part is even -- is the rounding (10 operations of the ALU in
// place of 17 for a comparison).
__host__ __device__ __forceinline__ double mul_core(uint64_t ua, uint64_t ub, uint64_t lo, uint64_t hi, bool top,
                                                    int32_t e)
{
    const uint32_t s = top ? 11u : 12u;
    const uint32_t l0 = (uint32_t)lo, l1 = (uint32_t)(lo >> 32), h0 = (uint32_t)hi, h1 = (uint32_t)(hi >> 32);
    const uint32_t m0 = funnel_left(l1, h0, s), m1 = funnel_left(h0, h1, s);
    const uint32_t r0 = l0 << s, r1 = funnel_left(l0, l1, s), odd = m0 & 1u;
    const uint32_t head = ((uint32_t)((ua ^ ub) >> 32) & 0x80000000u) | ((uint32_t)(e - 1) << 20);
    return add_carry_of(r0, r1, odd - 1u, odd + 0x7FFFFFFFu, m0, m1, head);
}

// a * b, both finite, normal and of any sign, with a normal product
// (including an overflow to infinity by rounding).  Returns false for a zero,
// subnormal, infinite or NaN operand, or a product out of the normal range.
__host__ __device__ __forceinline__ bool mul_rn(double a, double b, double &p)
{
    const uint64_t ua = bits_of(a), ub = bits_of(b);
    const int32_t ea = (int32_t)((ua >> 52) & 0x7FFu), eb = (int32_t)((ub >> 52) & 0x7FFu);
    if ((uint32_t)(ea - 1) >= 0x7FEu || (uint32_t)(eb - 1) >= 0x7FEu) return false;
    const uint64_t A = (ua & kMant) | kHidden, B = (ub & kMant) | kHidden;
    uint64_t lo, hi;  // A B in [2^104, 2^106)
    mul_significands(A, B, lo, hi);
    const bool top = (hi >> 41) != 0ULL;          // A B >= 2^105
    const int32_t e = ea + eb - 1023 + (top ? 1 : 0);
    if ((uint32_t)(e - 1) >= 0x7FEu) return false;
    p = mul_core(ua, ub, lo, hi, top, e);
    return true;
}

// a * b for operands that are known to be normal, with a product known to be
// normal (the caller's ranges guarantee it): mul_rn without its checks.
__host__ __device__ __forceinline__ double mul_normal(double a, double b)
{
    const uint64_t ua = bits_of(a), ub = bits_of(b);
    const int32_t ea = (int32_t)((ua >> 52) & 0x7FFu), eb = (int32_t)((ub >> 52) & 0x7FFu);
    const uint64_t A = (ua & kMant) | kHidden, B = (ub & kMant) | kHidden;
    uint64_t lo, hi;
    mul_significands(A, B, lo, hi);
    const bool top = (hi >> 41) != 0ULL;
    return mul_core(ua, ub, lo, hi, top, ea + eb - 1023 + (top ? 1 : 0));
}

// sqrt(x) for an x known to be normal and positive (no checks).
__host__ __device__ __forceinline__ double sqrt_normal(double x)
{
    const uint64_t ux = bits_of(x);
    const int32_t ex = (int32_t)(ux >> 52);
    const uint64_t M = (ux & kMant) | kHidden;
    const int32_t E = ex - 1023;                        // x = M 2^(E - 52)
    const bool odd = (E & 1) != 0;
    // X = M 2^52 (E even) or M 2^53 (E odd): sqrt(x) = sqrt(X) 2^((E - odd)/2 - 52),
    // sqrt(X) in [2^52, 2^53)
    const int sh = odd ? 53 : 52;
    const uint64_t Xlo = M << sh;  // mod 2^64
    // single precision's root of X 2^-80 = M 2^(sh - 80) in [2^24, 2^26) and its
    // reciprocal: sqrt(X) ~ S 2^29 (relative error below 2^-23), 1 / 2 sqrt(X) ~ r 2^-77
    const float sf = sqrt_rn((float)(uint32_t)(M >> (80 - sh)));  // in [2^12, 2^13)
    const uint32_t sb = float_bits(sf);
    const uint32_t S = ((sb & 0x7FFFFFu) | 0x800000u) << ((sb >> 23) - 139u);  // sf 2^11
    const uint32_t rb = float_bits(rcp_rn(sf));                                // in (2^-13, 2^-12]
    const int32_t r = (int32_t)(((rb & 0x7FFFFFu) | 0x800000u) << ((rb >> 23) - 114u));  // rf 2^36
    // q1 = S 2^29 + (X - S^2 2^58) / 2 sqrt(X), the difference exact in units of 2^52 (below
    // 2^32 of them): within 2^8 of sqrt(X)
    const int64_t D0 = (int64_t)((M << (sh - 52)) - (((uint64_t)S * S) << 6));
    uint64_t q = ((uint64_t)S << 29) + (uint64_t)(((int64_t)(int32_t)(D0 >> 2) * r) >> 23);
    // its exact remainder (below 2^62) over 2 sqrt(X) brings it to floor(sqrt(X)) or a
    // unit beside it, and the remainder of that, in [0, 2q] for the floor, fixes it
    int64_t R = (int64_t)(Xlo - q * q);
    const int32_t dq = (int32_t)(((int64_t)(int32_t)(R >> 32) * r) >> 45);
    R -= (int64_t)dq * (int64_t)(2 * q + (uint64_t)(int64_t)dq);
    q += (uint64_t)(int64_t)dq;
    if (R < 0) {
        R += (int64_t)(2 * q - 1);
        --q;
    } else if (R > (int64_t)(2 * q)) {
        R -= (int64_t)(2 * q + 1);
        ++q;
    }
    // round to nearest: sqrt(X) >= q + 1/2 iff X - q^2 > q (no ties)
    const uint64_t up = (uint64_t)R > q ? 1ULL : 0ULL;
    const int32_t er = ((E - (odd ? 1 : 0)) >> 1) + 1023;
    return double_of((((uint64_t)(er - 1)) << 52) + q + up);
}

// sqrt(x) for a normal x > 0.  Returns false otherwise (zero, subnormal,
// negative, infinite or NaN x).
__host__ __device__ __forceinline__ bool sqrt_pos(double x, double &r)
{
    const int32_t ex = (int32_t)(bits_of(x) >> 52);
    if ((uint32_t)(ex - 1) >= 0x7FEu) return false;
    r = sqrt_normal(x);
    return true;
}

}  // namespace sfp
}  // namespace rms
