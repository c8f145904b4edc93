// walk_kernel.cuh -- the random-walker time step (Sec. 2.2 items 2-5 of
// Lee, Fieremans & Novikov, arXiv 2012.06478), templated on the arithmetic
// type.  Included by walk_fp64.cu (built without FMA contraction: the plain
// form reproduces the CPU FP64 reference bit for bit) and walk_fp32.cu (the
// precision form: voxel index + FP32 offset, FP32 Kahan-compensated phase),
// and by walk_reject_fp{64,32}.cu and walk_mt_fp{64,32}.cu for the other
// particle-membrane interactions and for absorbing membranes.
//
// One thread owns one walker for a slice of steps; its state stays in registers
// (the plain form's phases and start offsets in shared memory) for the slice and
// goes back to global memory (structure of arrays, coalesced) at the end.  Per
// step and walker the only memory traffic is one byte for each voxel entered --
// its face bits, which say whether each of the voxel's faces leads into the same
// label (Sec. 2.1.1: the volume is the lookup table) -- at a membrane the label
// across it and the threshold of the label pair (and its saturation threshold,
// with absorbing membranes), and warp-uniform broadcasts of the waveform.
//
// What bounds it: the FP32 step issues (332 warp-instructions per warp-step on
// 200x200x400 axons, issue slots 77 % used, ALU pipe 64 %).  Deciding the
// events from face bits instead of a label gather with wrapped coordinates,
// with selects in place of branches, the step's weight asked for before the
// walk and nothing done for relaxation when no label relaxes took 1e6 walkers x
// 2000 steps from 27.4 ms (428 warp-instructions) to 21.8 ms; packed phase sums
// and octants without selects took the call of 10 000 steps from 112.6 ms to
// 108.4; the same bits.  The plain form's step uses the ALU, the integer
// products' and the FP64 pipe alike (72, 72 and 68 %, issue 77 %): 170 ms for
// the same launch, 269 before the loops over axes, unchecked arithmetic and
// shorter products, quotients and roots.
#pragma once

#include <cstdint>
#include <type_traits>

#include "f32x2.cuh"
#include "rms_device.cuh"
#include "soft_fp64.cuh"

namespace rms {

constexpr int kWalkBlock = 128;
constexpr int kWalkWarps = kWalkBlock / 32;

template <typename Real>
__device__ __forceinline__ Real clamp01(Real x)
{
    if (x < Real(0)) return Real(0);
    if (x > Real(1)) return Real(1);
    return x;
}
// FP32: the same clamp as __saturatef, which the compiler folds into the
// preceding multiply-add as its saturating form (identical results for the
// non-NaN positions; measured 7 % faster on the FP32 step).
template <>
__device__ __forceinline__ float clamp01<float>(float x)
{
    return __saturatef(x);
}

// FP64 comparisons on the integer ALU.  GB300's FP64 pipe is the scarce
// resource of the plain form, and every comparison or clamp of a double
// would occupy it.  The signed 64-bit pattern of a double orders exactly like
// its value among the non-negative doubles, and its sign bit tells x > 0 and
// x < 0 apart from +-0; the walk's positions, times and step vectors are
// never NaN, so these give the same booleans as the IEEE comparisons.
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ bool dgt0(double x) { return dbits(x) > 0; }  // x > 0
__device__ __forceinline__ bool dlt0(double x)                           // x < 0
{
    const long long b = dbits(x);
    return b < 0 && b != (long long)0x8000000000000000ULL;
}
// a < b for a, b >= +0 (no -0 and no NaN among the arguments)
__device__ __forceinline__ bool dlt_nn(double a, double b) { return dbits(a) < dbits(b); }
// if (x < 0) 0; else if (x > 1) 1; else x -- as clamp01, for any non-NaN x
__device__ __forceinline__ double dclamp01(double x)
{
    const long long b = dbits(x);
    if (b < 0) return b == (long long)0x8000000000000000ULL ? x : 0.0;
    return b > 0x3FF0000000000000LL ? 1.0 : x;
}

// -x by its sign bit, in assembly: the compiler negates a double with an
// addition, a slot of the FP64 pipe (a dozen of a step's 44).
__device__ __forceinline__ double dneg(double x)
{
    int hi = __double2hiint(x);
    asm("xor.b32 %0, %0, 0x80000000;" : "+r"(hi));
    return __hiloint2double(hi, __double2loint(x));
}
__device__ __forceinline__ double negated(double x) { return dneg(x); }
__device__ __forceinline__ float negated(float x) { return -x; }
// x != 0, NaNs among them
__device__ __forceinline__ bool nonzero(double x) { return (dbits(x) << 1) != 0; }
__device__ __forceinline__ bool nonzero(float x) { return x != 0.0f; }

// Sec. 2.2 item 2, the direction.  z = 1 - 2u is uniform on [-1, 1] for a
// uniform point of the sphere (Archimedes); the azimuth is
// phi = 2 pi (x1 + 1/2) 2^-32.  Its sine and cosine come from Taylor
// polynomials after an octant reduction in integers -- in the FP64 form a
// table of 1024 angles of [0, pi/4] (filled by poly_sincos), a 5th-order
// polynomial for the offset from the nearest table angle and the
// angle-addition formula -- so the FP64 form uses only +, * and sqrt (the
// same bits as any IEEE machine given the same operation order), and no
// warp ever loops on a rejection.
__device__ __forceinline__ void octant_map(uint32_t oct, double cs, double sn, double &cx, double &sy)
{
    const bool swap = ((oct + 1u) >> 1) & 1u;                      // octants 1, 2, 5, 6
    const int negx = (int)(((oct + 2u) << 29) & 0x80000000u);      // octants 2..5
    const int negy = (int)((oct << 29) & 0x80000000u);             // octants 4..7
    const double a = swap ? sn : cs, b = swap ? cs : sn;
    cx = __hiloint2double(__double2hiint(a) ^ negx, __double2loint(a));
    sy = __hiloint2double(__double2hiint(b) ^ negy, __double2loint(b));
}

// The hardware FP64 operations, for the operands the integer-ALU versions
// hand back (zeros, subnormals, out-of-range results).  Out of line, so that
// the compiler cannot evaluate them speculatively beside the integer path:
// inlined, a predicated copy would run on the FP64 pipe at every call.
static __device__ __noinline__ double hw_mul(double a, double b) { return a * b; }
static __device__ __noinline__ double hw_div(double a, double b) { return a / b; }

// FP64 products and quotients of non-negative operands on the integer ALU
// (sfp::mul_rn, div_pos: the IEEE results bit for bit).
__device__ __forceinline__ double dmul(double a, double b)
{
    double p;
    if (!sfp::mul_rn(a, b, p)) p = hw_mul(a, b);
    return p;
}
__device__ __forceinline__ double ddiv_nn(double a, double b)
{
    double q;
    if (!sfp::div_pos(a, b, q)) q = hw_div(a, b);
    return q;
}

// SANE: the run's numbers are within ranges (sane_ranges, rms_api.cu) where every
// operand and result of the step is zero or far inside the normal numbers: no
// range checks, no branches to the hardware operations (3.3e5 walkers x 300 steps on
// 200x200x400 axons: 2469 warp-instructions a warp-step against 2752, 8.43 ms against
// 9.54).  Otherwise the checked versions.  The same bits.
//
// Why the ranges hold: steps are 2^-200 to 1 voxels and directions' components at
// least 2^-60; offsets are 0 or, but for a chance of 2^-300, above 2^-300; so face
// times, their differences and all products stay above 2^-900, and quotients
// below 2^300.
__device__ __forceinline__ bool is_zero(double x)  // of a zero or normal number
{
    return (__double2hiint(x) & 0x7FF00000) == 0;
}
// the product where neither operand is zero (SANE)
template <bool SANE>
__device__ __forceinline__ double times_nz(double a, double b)
{
    if constexpr (SANE)
        return sfp::mul_normal(a, b);
    else
        return dmul(a, b);
}
// where a may be
template <bool SANE>
__device__ __forceinline__ double times(double a, double b)
{
    if constexpr (SANE) {
        const double p = sfp::mul_normal(a, b);
        return is_zero(a) ? __hiloint2double((__double2hiint(a) ^ __double2hiint(b)) & (int)0x80000000, 0) : p;
    } else {
        return dmul(a, b);
    }
}
// where both may be
template <bool SANE>
__device__ __forceinline__ double times_any(double a, double b)
{
    if constexpr (SANE) {
        const double p = sfp::mul_normal(a, b);
        return is_zero(a) || is_zero(b)
                   ? __hiloint2double((__double2hiint(a) ^ __double2hiint(b)) & (int)0x80000000, 0)
                   : p;
    } else {
        return dmul(a, b);
    }
}
// a / b for a >= +0, b > 0
template <bool SANE>
__device__ __forceinline__ double over(double a, double b)
{
    if constexpr (SANE) {
        const double q = sfp::div_normal(a, b);
        return is_zero(a) ? 0.0 : q;
    } else {
        return ddiv_nn(a, b);
    }
}

// Exact doubles built from their bits on the integer ALU, so that values
// which need no rounding do not occupy GB300's narrow FP64 pipe.
// k * 2^e2 for an odd |k| < 2^32: no rounding, the same bits as converting k
// and multiplying by the power of two.
__device__ __forceinline__ double odd_scaled(uint32_t mag, bool neg, int e2)
{
    const int p = 31 - __clz((int)mag);  // position of the leading one
    const unsigned long long mant = ((unsigned long long)mag << (52 - p)) & 0x000FFFFFFFFFFFFFULL;
    const unsigned long long bits = (neg ? 0x8000000000000000ULL : 0ULL) |
                                    ((unsigned long long)(p + e2 + 1023) << 52) | mant;
    return __longlong_as_double((long long)bits);
}
// N 2^-64 rounded to the nearest double, ties to even (0 < N < 2^64): the
// IEEE result of a product of doubles whose exact value is N 2^-64.
__device__ __forceinline__ double u64_scaled_rn(unsigned long long N)
{
    // the leading one to bit 63: 53 bits kept, 11 below them
    const int z = __clzll((long long)N);
    const unsigned long long t = (unsigned long long)N << z, m = t >> 11;
    const unsigned long long up = ((uint32_t)t & 0x7FFu) + ((uint32_t)m & 1u) > 0x400u ? 1ULL : 0ULL;
    return __longlong_as_double((long long)(((unsigned long long)(1021 - z) << 52) + m + up));
}

// UNROLL: all products side by side (the four-lane kernel, bound by their latency).
template <bool UNROLL = false>
__device__ __forceinline__ void direction_from(uint32_t x0, uint32_t x1, const double *__restrict__ trig,
                                               double n[3])
{
    // z = 1 - 2 u(x0) = k 2^-32 with the odd integer k = 2^32 - 1 - 2 x0, and
    // (1 - z)(1 + z) = (2^64 - k^2) 2^-64 rounded once: both from integers,
    // the same bits as the CPU FP64 reference's step-by-step evaluation.
    const bool zneg = x0 >= 0x80000000u;
    const uint32_t kmag = zneg ? 2u * x0 + 1u : 0xFFFFFFFFu - 2u * x0;  // |k|
    const double z = odd_scaled(kmag, zneg, -32);
    // Every value below is normal and nonzero for every pair of words, so the
    // integer-ALU products and square root need neither range checks nor a
    // hardware fallback: the argument of the root is at least (2^33 - 1) 2^-64;
    // |e| lies in [2^-30, 2^-11] pi/4, t = e^2 in [2^-61, 2^-22], the table's
    // cosines and sines in [3.8e-4, 1], cs and sn in [7e-10, 1] (the angle is at
    // least 2^-30 pi/4), r in [2^-16, 1]; every product stays far inside the
    // normal range.
    const double r = sfp::sqrt_normal(u64_scaled_rn(0ULL - (unsigned long long)kmag * kmag));
    const uint32_t oct = x1 >> 29;
    uint32_t m = x1 & 0x1FFFFFFFu;
    if (oct & 1u) m = 0x1FFFFFFFu - m;
    // angle (m + 1/2) 2^-29 pi/4 = theta_j + e, theta_j = (2j + 1) 2^-11 pi/4 the
    // centre of part j = top 10 bits of m, |e| <= 2^-11 pi/4
    const uint32_t j = m >> 19;
    const int32_t lo = (int32_t)(m & 0x7FFFFu);
    const int32_t e_int = 2 * lo + 1 - (1 << 19);  // odd
    using sfp::mul_normal;
    const double e = mul_normal(odd_scaled((uint32_t)(e_int < 0 ? -e_int : e_int), e_int < 0, -30), 0.78539816339744830962);
    const double t = mul_normal(e, e);
    const double se = e + mul_normal(mul_normal(e, t), -1.0 / 6.0 + mul_normal(t, 1.0 / 120.0));
    const double ce = 1.0 + mul_normal(t, -1.0 / 2.0 + mul_normal(t, 1.0 / 24.0));
    const double cj = __ldg(trig + 2 * j), sj = __ldg(trig + 2 * j + 1);
    // cs = cj ce - sj se, then sn = sj ce - (-cj) se
    double cs = 0.0, sn = 0.0;
    {
        double p = cj, q = sj;
#pragma unroll UNROLL ? 2 : 1
        for (int i = 0; i < 2; ++i) {
            cs = sn;
            sn = mul_normal(p, ce) - mul_normal(q, se);
            const double m = dneg(p);
            p = q;
            q = m;
        }
    }
    double cx, sy;
    octant_map(oct, cs, sn, cx, sy);
#pragma unroll UNROLL ? 2 : 1
    for (int i = 0; i < 2; ++i) {
        const double x = mul_normal(r, cx);
        cx = sy;
        sy = x;
    }
    n[0] = cx;
    n[1] = sy;
    n[2] = z;
}

// a times the approximate reciprocal of b >= 0 (within 1 ulp; a subnormal b counts
// as 0, whose reciprocal is infinite), and the approximate reciprocal square root:
// one instruction each.  The divisors |d| of the FP32 step are 0 or normal: a
// direction's components are 0 or above 2^-42, and a label's step length is 0 or at
// least kMinStepF voxels.
__device__ __forceinline__ float mul_rcp(float a, float b)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
    return a * r;
}
__device__ __forceinline__ float rsqrt_normal(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// FP32 form of the same sampler: shorter polynomials (truncation below
// 4e-7 on [0, pi/4]) and r from the hardware reciprocal square root (about
// 2 ulp) -- errors of the order of the FP32 form's own rounding, for 2 % of its
// step time.  For 129 of the 2^32 words z rounds to +-1, where r = 0 inf is not a
// number: such a step (3e-8 of them) leaves x and y without a face event and its
// clamp puts their offsets to 0.
__device__ __forceinline__ void direction_from(uint32_t x0, uint32_t x1, const double *, float n[3])
{
    const float z = -((float)(int32_t)(x0 ^ 0x80000000u) + 0.5f) * 0x1p-31f;
    const float rr = (1.0f - z) * (1.0f + z);
    const float r = rr * rsqrt_normal(rr);
    // the octant's fold, swap and signs from the word's own bits
    const uint32_t m = (x1 ^ (uint32_t)((int32_t)(x1 << 2) >> 31)) & 0x1FFFFFFFu;  // odd octants from their end
    const float th = ((float)m + 0.5f) * (0x1p-29f * 0.785398163f);
    const float t = th * th;
    const float sn = th + (th * t) * (-1.0f / 6.0f + t * (1.0f / 120.0f + t * (-1.0f / 5040.0f)));
    const float cs = 1.0f + t * (-0.5f + t * (1.0f / 24.0f + t * (-1.0f / 720.0f + t * (1.0f / 40320.0f))));
    const bool swap = ((x1 + 0x20000000u) & 0x40000000u) != 0u;  // octants 1, 2, 5, 6
    const float a = swap ? sn : cs, b = swap ? cs : sn;
    n[0] = r * __uint_as_float(__float_as_uint(a) ^ ((x1 + 0x40000000u) & 0x80000000u));  // octants 2..5
    n[1] = r * __uint_as_float(__float_as_uint(b) ^ (x1 & 0x80000000u));                  // octants 4..7
    n[2] = z;
}

// The plain form's loops over axes are not unrolled: its integer-ALU products
// and quotients are 30 to 150 instructions each, and with three copies of each
// the step's code was larger than the instruction caches (instruction fetch the
// first of the stalls): 3.3e5 walkers x 3000 steps 139 ms unrolled, 120 with the
// loops, 112.5 with the phases and start offsets in shared memory too, the
// offsets of an event's other two axes moved in one loop and 6 blocks an SM.
// Axis r is in slot 0 in the loop's turn r; after three turns every axis is back
// in its own.
template <typename T>
__device__ __forceinline__ void rotate(T x[3])
{
    const T t = x[0];
    x[0] = x[1];
    x[1] = x[2];
    x[2] = t;
}

// Saturation (Sec. 2.1.3): A = +inf (FP64 form) or kSaturatedF (FP32 form).
__device__ __forceinline__ bool saturated(double A) { return dbits(A) == 0x7FF0000000000000LL; }
__device__ __forceinline__ bool saturated(float A) { return A >= kSaturatedF; }
__device__ __forceinline__ void saturate(double &A, double &) { A = __longlong_as_double(0x7FF0000000000000LL); }
__device__ __forceinline__ void saturate(float &A, float &Ac)
{
    A = kSaturatedF;
    Ac = 0.0f;
}

// Word 0 of a step's PERM call: the Bernoulli word of a third membrane event
// in one step.  Rare, so kept out of line: inlined, the ten Philox rounds
// would sit in every pass of the face-event loop (measured: 4 % of the FP32
// step on the axon workload).
static __device__ __noinline__ uint32_t perm_word(uint64_t seed, uint64_t w, uint32_t k, uint32_t call)
{
    return draw(seed, w, k, kTagPerm, call).x;
}

// Coordinate q modulo N, in [0, N).
__device__ __forceinline__ int32_t wrapped(int32_t q, int32_t N)
{
    q %= N;
    return q < 0 ? q + N : q;
}

// A face event of an edge voxel v: the voxel across -- nv, or the one on the
// periodic other side -- or -1 for the impermeable outer wall.  The
// coordinates come from the flat index by multiplication (no division).  Out
// of line, on values: a few events in a thousand on volumes of a hundred
// voxels an edge.
static __device__ __noinline__ int32_t edge_voxel(int32_t v, int32_t nv, int best, bool up, int32_t nx, int32_t ny,
                                                  int32_t nz, FastDiv div_x, FastDiv div_xy, int32_t periodic)
{
    const int32_t row = (int32_t)div_x.quotient((uint32_t)v);    // v / nx
    const int32_t z = (int32_t)div_xy.quotient((uint32_t)v);     // v / (nx ny)
    const int32_t coord = best == 2 ? z : (best == 1 ? row - z * ny : v - row * nx);
    const int32_t N = best == 2 ? nz : (best == 1 ? ny : nx);
    if (coord != (up ? N - 1 : 0)) return nv;
    if (!((periodic >> best) & 1)) return -1;
    const int32_t sb = best == 2 ? nx * ny : (best == 1 ? nx : 1);
    return up ? v - (N - 1) * sb : v + (N - 1) * sb;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <typename Real>
__device__ __forceinline__ void kahan_add(Real &sum, Real &comp, Real x)
{
    const Real y = x - comp;
    const Real t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

// The phases of NS shapes by axis, component k = 3 shape + axis.  Plain form: in
// shared memory, with the start offsets, so that loops over axes and shapes need
// not be unrolled and the registers hold more warps.
template <typename Real, int NS>
struct Phases {
    double *p, *start;  // [component or axis][thread]
    // shared memory of a block
    static size_t bytes(int n) { return sizeof(double) * (3 * n + 3) * kWalkBlock; }
    __device__ __forceinline__ void load(const WalkerState<Real> &st, int n, int64_t W, int64_t li)
    {
        extern __shared__ double s_axes[];
        start = s_axes + threadIdx.x;
        p = start + 3 * kWalkBlock;
        for (int k = 0; k < 3 * n; ++k) p[k * kWalkBlock] = st.phase[k * W + li];
#pragma unroll
        for (int a = 0; a < 3; ++a) start[a * kWalkBlock] = st.o0[a][li];
    }
    __device__ __forceinline__ void store(const WalkerState<Real> &st, int n, int64_t W, int64_t li) const
    {
        for (int k = 0; k < 3 * n; ++k) st.phase[k * W + li] = p[k * kWalkBlock];
    }
    // component `axis` of every shape's phase += w dx
    template <bool SANE, typename Weight>
    __device__ __forceinline__ void add(int n, int axis, double dx, Weight weight)
    {
        if constexpr (NS == 1) {
            p[axis * kWalkBlock] = p[axis * kWalkBlock] + times_any<SANE>(weight(0), dx);
        } else {
#pragma unroll 1
            for (int s = 0; s < n; ++s) {
                double &x = p[(3 * s + axis) * kWalkBlock];
                x = x + times_any<SANE>(weight(s), dx);
            }
        }
    }
};
// FP32: two components an instruction (x and y of a shape, or the six of two
// shapes), the additions that bound a step of several shapes.  The
// compensation is kept negated, so that y = w dx - c is one multiply-add.
template <int NS>
struct Phases<float, NS> {
    static constexpr int kPairs = 3 * NS / 2;  // and, of an odd number of shapes, the last z
    F2 p[kPairs], nc[kPairs];
    float pz, ncz;
    static size_t bytes(int) { return 0; }
    __device__ __forceinline__ void load(const WalkerState<float> &st, int n, int64_t W, int64_t li)
    {
        const auto of = [&](const float *from, int k) { return k < 3 * n ? from[k * W + li] : 0.0f; };
#pragma unroll
        for (int k = 0; k < kPairs; ++k) {
            p[k] = pair_of(of(st.phase, 2 * k), of(st.phase, 2 * k + 1));
            nc[k] = pair_of(-of(st.phase_c, 2 * k), -of(st.phase_c, 2 * k + 1));
        }
        pz = ncz = 0.0f;
        if (NS & 1) {
            pz = of(st.phase, 3 * NS - 1);
            ncz = -of(st.phase_c, 3 * NS - 1);
        }
    }
    __device__ __forceinline__ void store(const WalkerState<float> &st, int n, int64_t W, int64_t li) const
    {
        const auto put = [&](int k, float x, float c) {
            if (k < 3 * n) {
                st.phase[k * W + li] = x;
                st.phase_c[k * W + li] = -c;
            }
        };
#pragma unroll
        for (int k = 0; k < kPairs; ++k) {
            put(2 * k, first(p[k]), first(nc[k]));
            put(2 * k + 1, second(p[k]), second(nc[k]));
        }
        if (NS & 1) put(3 * NS - 1, pz, ncz);
    }
    template <int K>
    __device__ __forceinline__ void add_pair(F2 w, F2 dx)
    {
        static_assert(K < kPairs, "a pair of this many shapes");
        const F2 y = fma2(w, dx, nc[K]), t = p[K] + y;
        nc[K] = y - (t - p[K]);
        p[K] = t;
    }
    // shapes s and s + 1; the last of an odd number alone
    template <int S, typename Weight>
    __device__ __forceinline__ void add_from(int n, F2 xy, F2 zx, F2 yz, float z, Weight weight)
    {
        if constexpr (S < NS) {
            if (S >= n) return;
            const float w0 = weight(S);
            add_pair<3 * S / 2>(pair_of(w0, w0), xy);
            if constexpr (S + 1 < NS) {
                // a shape beyond the last adds w = 0 to phases that nobody reads
                const float w1 = S + 1 < n ? weight(S + 1) : 0.0f;
                add_pair<3 * S / 2 + 1>(pair_of(w0, w1), zx);
                add_pair<3 * S / 2 + 2>(pair_of(w1, w1), yz);
                add_from<S + 2>(n, xy, zx, yz, z, weight);
            } else {
                const float y = fmaf(w0, z, ncz), t = pz + y;
                ncz = y - (t - pz);
                pz = t;
            }
        }
    }
    template <typename Weight>
    __device__ __forceinline__ void add(int n, const float dx[3], Weight weight)
    {
        add_from<0>(n, pair_of(dx[0], dx[1]), pair_of(dx[2], dx[0]), pair_of(dx[1], dx[2]), dx[2], weight);
    }
};

// The 22 moment terms at a recording step (Sec. 2.3, narrow-pulse D and K):
// alpha, alpha dx_i dx_j (i <= j), alpha dx_i dx_j dx_k dx_l (i<=j<=k<=l),
// each reduced over the warp as soon as it is formed (few live registers);
// lane 0 of each warp leaves the warp's 22 sums in red[22].
__device__ __forceinline__ void warp_moments(double al, const double dx[3], double *red)
{
    const int lane = threadIdx.x & 31;
    int p = 0;
    double r = warp_sum(al);
    if (lane == 0) red[p] = r;
    ++p;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = a; b < 3; ++b) {
            r = warp_sum(al * dx[a] * dx[b]);
            if (lane == 0) red[p] = r;
            ++p;
        }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = a; b < 3; ++b)
#pragma unroll
            for (int c = b; c < 3; ++c)
#pragma unroll
                for (int d = c; d < 3; ++d) {
                    r = warp_sum(al * dx[a] * dx[b] * dx[c] * dx[d]);
                    if (lane == 0) red[p] = r;
                    ++p;
                }
}

// Steps (k_begin, k_end] for the kWalkBlock walkers of block `block` of a
// run (walkers block*kWalkBlock ...), one walker per thread.  IM is the
// particle-membrane interaction: elastic collision (Sec. 2.1.2-2.1.3, the
// paper's method), or one of the alternatives of App. A and B, in which a
// refused face cancels the step -- rejection sampling keeps the walker where
// it was for the step, ERL draws a new direction (DIR and PERM call = the
// draw's index) until a step is admitted, at most kMaxLeaps draws.  MT adds
// absorbing membranes (Sec. 2.1.3, magnetization transfer; t.Tmt non-null).
// RELAX: 1 some label has a finite T1 or T2, 0 none has (every rate is 0, the
// exponent keeps its start value and Eq. 5 drops out), 2 decided at run time.
// RK: hold the round keys of ctl.rk (computed once on the host) for the slice;
// otherwise read them at every draw (the batched kernel, whose request
// descriptors sit in shared memory).  `rec` is the first recording step's
// index beyond k_begin.
template <typename Real, int NS, bool HASH, int IM, bool MT, int RELAX, bool RK = false, bool SANE = false>
__device__ __forceinline__ void walk_block(const Geometry &g, const Tables<Real> &t, const WalkerState<Real> &st,
                                           const RunCtl &ctl, int64_t block, int64_t k_begin, int64_t k_end,
                                           int32_t rec)
{
    constexpr bool kF64 = std::is_same<Real, double>::value;
    __shared__ int32_t s_cancel;
    __shared__ double s_red[kWalkWarps][kMoments];
    if (threadIdx.x == 0) s_cancel = ctl.cancel ? *ctl.cancel : 0;
    __syncthreads();
    if (s_cancel) return;

    // the round keys, loop-invariant and warp-uniform: read once here (read
    // from the launch parameters inside the step loop they took 16 constant
    // loads per warp-step; hoisted, the step is 1.3 % faster)
    [[maybe_unused]] uint32_t rk[kRoundKeys];
    if constexpr (RK) {
#pragma unroll
        for (int i = 0; i < kRoundKeys; ++i) rk[i] = ctl.rk[i];
    }
    // threads beyond the last walker walk a copy of it and write nothing: no
    // branch on it in the step loop, and what a copy reports (status) is what its
    // walker reports
    const bool active = block * kWalkBlock + threadIdx.x < ctl.n_walkers;
    const int64_t li = active ? block * kWalkBlock + threadIdx.x : ctl.n_walkers - 1;
    // the walker in this slot: its id picks its random streams (RMS_MORTON
    // runs keep walkers in Morton order of their voxel, not in id order)
    const uint64_t w = (uint64_t)(ctl.w_begin + (st.wid ? (int64_t)st.wid[li] : li));
    const int32_t N[3] = {g.nx, g.ny, g.nz};
    const int32_t stride[3] = {1, g.nx, g.nx * g.ny};
    const int32_t L = t.n_labels;
    const bool relax = RELAX == 2 ? t.any_relax != 0 : RELAX == 1;
    // voxel edge in the form's precision (the single-precision value comes from
    // the host: a conversion here would run on the FP64 pipe at every step)
    Real lp;
    if constexpr (kF64)
        lp = g.voxel_um;
    else
        lp = g.voxel_f;

    Real o[3];
    [[maybe_unused]] Real o0[3];  // FP32 form; the plain form's are beside its phases
    int32_t di[3];
    int32_t v = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        o[a] = st.o[a][li];
        if constexpr (!kF64) o0[a] = st.o0[a][li];
        di[a] = st.di[a][li];
        v += stride[a] * wrapped(st.i0[a][li] + di[a], N[a]);
    }
    uint32_t fm = __ldg(g.faces + v);  // face bits of voxel v (rms_device.cuh)
    int32_t c = st.c[li];
    Real sc = __ldg(t.s + c);  // step length of label c
    Real A = st.A[li], Ac = Real(0);
    if constexpr (!kF64) Ac = st.A_c[li];
    Phases<Real, NS> ph;
    ph.load(st, ctl.n_shapes, ctl.n_walkers, li);
    [[maybe_unused]] uint64_t h = 0;
    // face events, crossings into another label, reflections (verification kernel)
    [[maybe_unused]] int32_t nev = 0, ncr = 0, nrf = 0;
    if constexpr (HASH) {
        h = st.hash[li];
        if (st.counts) {
            nev = st.counts[li];
            ncr = st.counts[ctl.n_walkers + li];
            nrf = st.counts[2 * ctl.n_walkers + li];
        }
    }
    int32_t next_rec = rec < ctl.n_rec ? __ldg(t.rec_step + rec) : INT32_MAX;
    // the copies of the last walker have read its state before its own thread, in
    // another warp, writes it back at the end of the slice
    __syncthreads();

    // a 32-bit step counter (n_steps <= 2e9): uniform 32-bit arithmetic per
    // step (measured 0.8 % faster than 64-bit on the FP32 step)
    for (int32_t k = (int32_t)k_begin + 1; k <= (int32_t)k_end; ++k) {
        // the step's weight dt G_k, asked for before the walk (several shapes: a flag
        // that one of them is not zero)
        [[maybe_unused]] Real wg = Real(0);
        bool graded;
        if constexpr (NS == 1) {
            wg = __ldg(t.wG + (k - 1));
            graded = nonzero(wg);
        } else {
            graded = (__ldg(t.flags + (k - 1)) & 1u) != 0u;
        }
        int mode = 0;
        if (relax) mode = t.mode ? (int)__ldg(t.mode + (k - 1)) : 0;
        // state at the step start, restored when a membrane refuses the step
        [[maybe_unused]] Real o_s[3], A_s, Ac_s;
        [[maybe_unused]] int32_t di_s[3], v_s, c_s, nev_s, ncr_s, nrf_s;
        [[maybe_unused]] uint32_t fm_s;
        [[maybe_unused]] Real sc_s;
        if constexpr (IM != kInteractEC) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                o_s[a] = o[a];
                di_s[a] = di[a];
            }
            v_s = v;
            fm_s = fm;
            c_s = c;
            sc_s = sc;
            A_s = A;
            Ac_s = Ac;
            if constexpr (HASH) {
                nev_s = nev;
                ncr_s = ncr;
                nrf_s = nrf;
            }
        }
        uint32_t att = 0;  // draw index (ERL redraws); always 0 otherwise
        [[maybe_unused]] bool sat_any = false;  // saturated on some draw of this step (MT)
#pragma unroll 1
        for (;;) {
            // ---- direction (one DIR call: words 0, 1 -> direction; words 2, 3 ->
            //      the Bernoulli words of the step's first two membrane events)
            U4 x;
            if constexpr (RK)
                x = philox4x32_10_rk(U4{(uint32_t)w, (uint32_t)(w >> 32), (uint32_t)k, (kTagDir << 16) | att}, rk);
            else
                x = philox4x32_10_rk(U4{(uint32_t)w, (uint32_t)(w >> 32), (uint32_t)k, (kTagDir << 16) | att}, ctl.rk);
            Real n[3];
            direction_from(x.x, x.y, t.trig, n);
            // ---- face walk (Sec. 2.2 items 3-4)
            Real rate = Real(0);
            if (relax) rate = __ldg(t.dtR + mode * L + c);
            [[maybe_unused]] const Real rate0 = rate;
            Real d[3] = {};
            if constexpr (!kF64) {
#pragma unroll
                for (int a = 0; a < 3; ++a) d[a] = n[a] * sc;
            }
            [[maybe_unused]] bool refused = false;
            // A face event on axis `best` moving up/down: where the voxel's own face
            // bits say that the voxel across is inside the volume and carries the same
            // label -- nearly every event -- nothing is looked up to decide it: the
            // walker moves on, and the new voxel's bits, which the next event needs,
            // load meanwhile.  membrane() takes any other face: nv becomes the voxel
            // across; true when the walker crosses (changed: into another label).
            auto membrane = [&](int best, bool up, int ev, int32_t &nv, bool &changed) -> bool {
                if (fm & kFaceEdge)
                    nv = edge_voxel(v, nv, best, up, g.nx, g.ny, g.nz, g.div_x, g.div_xy, g.periodic);
                const int32_t c2 = nv < 0 ? -1 : (int32_t)__ldg(g.labels + nv);
                // magnetization transfer (Sec. 2.1.3): meeting an absorbing membrane
                // saturates the walker with probability P_MT -- word `ev` of the
                // step's MT call (call = the draw index)
                if constexpr (MT) {
                    if (c2 >= 0 && c2 != c) {
                        const uint32_t tm = __ldg(t.Tmt + (int64_t)c * L + c2);
                        if (tm != 0u && !saturated(A)) {
                            const U4 m = draw(ctl.seed, w, (uint32_t)k, kTagMT, att);
                            if ((ev == 0 ? m.x : (ev == 1 ? m.y : m.z)) < tm) saturate(A, Ac);
                        }
                    }
                }
                if (c2 == c) return true;
                const uint32_t T = c2 < 0 ? 0u : __ldg(t.T + (int64_t)c * L + c2);
                bool cross = false;
                if (T != 0u) {
                    // third membrane event of a step: word 0 of the step's PERM call
                    const uint32_t word =
                        ev == 0 ? x.z : (ev == 1 ? x.w : perm_word(ctl.seed, w, (uint32_t)k, att));
                    cross = word < T;
                }
                if (cross) {
                    if constexpr (HASH) ++ncr;
                    c = c2;
                    if (relax) rate = __ldg(t.dtR + mode * L + c);
                    changed = true;  // the caller switches to the new label's step length
                    return true;
                }
                if constexpr (IM != kInteractEC) {
                    refused = true;
                } else {
                    if constexpr (HASH) ++nrf;
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        if (a == best) {
                            n[a] = negated(n[a]);
                            d[a] = negated(d[a]);
                        }
                }
                return false;
            };
            // Face times from the step start: axis a meets its face at T[a] = dist/|d_a|
            // (beyond the step when >= 1); events are taken in time order (ties to the
            // lower axis), an axis meets at most one face per step (s_c < 1: the corner
            // reflector), and a crossing into a label of another step length
            // recomputes the remaining times from the current positions.
            if constexpr (kF64) {
                // Plain form: the CPU FP64 reference's operation order; comparisons on the
                // integer ALU (dgt0/dlt_nn/dclamp01 give the IEEE results).
                const double kInf = __longlong_as_double(0x7FF0000000000000LL);
                // one division per axis: (1 - o)/d moving up, o/(-d) moving down, on the
                // integer ALU (the IEEE quotient; the hardware division only for operands
                // outside its range, e.g. o = -0)
                double T[3] = {};
                const auto face_time = [](double o, double d) {
                    return over<SANE>(dgt0(d) ? 1.0 - o : o, __longlong_as_double(dbits(d) & 0x7FFFFFFFFFFFFFFFLL));
                };
#pragma unroll 1
                for (int r = 0; r < 3; ++r) {
                    d[0] = times_nz<SANE>(n[0], sc);
                    T[0] = SANE || dgt0(d[0]) || dlt0(d[0]) ? face_time(o[0], d[0]) : kInf;
                    rotate(n);
                    rotate(o);
                    rotate(d);
                    rotate(T);
                }
                double tau = 0.0;
                // not unrolled in the plain form: its event pass carries the integer-ALU
                // arithmetic (and the rare re-timing after a change of step length, with
                // three divisions); three copies of it measured 7 % slower, from
                // instruction fetch
#pragma unroll 1
                for (int ev = 0; ev < 3; ++ev) {
                    int best = 0;
                    double tmin = T[0];
                    if (dlt_nn(T[1], tmin)) {
                        best = 1;
                        tmin = T[1];
                    }
                    if (dlt_nn(T[2], tmin)) {
                        best = 2;
                        tmin = T[2];
                    }
                    if (!dlt_nn(tmin, 1.0)) break;
                    const double dts = tmin - tau;
                    if (relax) A = A + times_any<SANE>(dts, rate);
                    tau = tmin;
                    if constexpr (HASH) ++nev;
                    const bool up = dgt0(best == 2 ? d[2] : (best == 1 ? d[1] : d[0]));
                    {
                        // the two axes that meet no face move on: their offsets and steps,
                        // taken out, moved in turn, and put back beside the face
                        double oa = best == 0 ? o[1] : o[0], ob = best == 2 ? o[1] : o[2];
                        double da = best == 0 ? d[1] : d[0], db = best == 2 ? d[1] : d[2];
#pragma unroll 1
                        for (int r = 0; r < 2; ++r) {
                            const double x = dclamp01(oa + times<SANE>(dts, da)), y = da;
                            oa = ob;
                            ob = x;
                            da = db;
                            db = y;
                        }
                        const double face = up ? 0.0 : 1.0;
                        o[0] = best == 0 ? face : oa;
                        o[1] = best == 1 ? face : (best == 0 ? oa : ob);
                        o[2] = best == 2 ? face : ob;
                    }
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        if (a == best) {
                            T[a] = kInf;
                            di[a] += up ? 1 : -1;
                        }
                    const int32_t sb = best == 2 ? stride[2] : (best == 1 ? stride[1] : 1);
                    const uint32_t bit = (best == 2 ? kFaceZ : (best == 1 ? kFaceY : kFaceX)) << (up ? 3 : 0);
                    int32_t nv = up ? v + sb : v - sb;
                    if (!(fm & bit)) {
                        bool changed = false;
                        if (!membrane(best, up, ev, nv, changed)) {  // stays in its voxel, at the face
                            nv = v;
#pragma unroll
                            for (int a = 0; a < 3; ++a)
                                if (a == best) {
                                    o[a] = up ? 1.0 : 0.0;
                                    di[a] -= up ? 1 : -1;
                                }
                        }
                        if (changed) {
                            const double sn = __ldg(t.s + c);
                            if (dbits(sn) != dbits(sc)) {
                                sc = sn;
#pragma unroll 1
                                for (int r = 0; r < 3; ++r) {
                                    d[0] = times_nz<SANE>(n[0], sc);
                                    if (dbits(T[0]) != 0x7FF0000000000000LL) T[0] = tau + face_time(o[0], d[0]);
                                    rotate(n);
                                    rotate(o);
                                    rotate(d);
                                    rotate(T);
                                }
                            }
                        }
                    }
                    v = nv;
                    fm = __ldg(g.faces + v);
                    if constexpr (IM != kInteractEC) {
                        if (refused) break;
                    }
                }
                if (IM == kInteractEC || !refused) {
                    const double rem = 1.0 - tau;
#pragma unroll 1
                    for (int r = 0; r < 3; ++r) {
                        o[0] = dclamp01(o[0] + times_nz<SANE>(rem, d[0]));
                        rotate(o);
                        rotate(d);
                    }
                    if (relax) A = A + times_any<SANE>(rem, rate);
                }
            } else {
                // Precision form: the same walk in FP32.  The choices are selects and
                // predicated instructions; only the end test and the membrane branch, and a
                // membrane that is not crossed takes back the crossing assumed before it.
                constexpr Real kNever = Real(1e30);
                Real T[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const bool up = d[a] > Real(0);
                    T[a] = fminf(mul_rcp(up ? Real(1) - o[a] : o[a], fabsf(d[a])), kNever);
                }
                Real tau = Real(0);
#pragma unroll  // unrolled: each event index is a constant (measured 5 % faster, FP32)
                for (int ev = 0; ev < 3; ++ev) {
                    const bool b1 = T[1] < T[0];
                    const Real t01 = fminf(T[0], T[1]);
                    const bool b2 = T[2] < t01;
                    Real tmin = fminf(t01, T[2]);
                    if (!(tmin < Real(1))) break;
                    if (ev > 0) tmin = fmaxf(tmin, tau);
                    const Real dtt = ev > 0 ? tmin - tau : tmin;
                    if (relax) kahan_add(A, Ac, dtt * rate);
                    tau = tmin;
                    if constexpr (HASH) ++nev;
                    const int best = b2 ? 2 : (b1 ? 1 : 0);
                    const bool up = (b2 ? d[2] : (b1 ? d[1] : d[0])) > Real(0);
                    const int32_t sb = b2 ? stride[2] : (b1 ? stride[1] : 1);
                    const int32_t inc = up ? 1 : -1;
                    int32_t nv = v + inc * sb;
                    const uint32_t bit = (b2 ? kFaceZ : (b1 ? kFaceY : kFaceX)) << (up ? 3 : 0);
                    const Real at = up ? Real(0) : Real(1);
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const bool p = a == best;
                        o[a] = p ? at : clamp01(o[a] + dtt * d[a]);
                        T[a] = p ? kNever : T[a];
                        if (p) di[a] += inc;
                    }
                    if (!(fm & bit)) {
                        bool changed = false;
                        if (!membrane(best, up, ev, nv, changed)) {  // stays in its voxel, at the face
                            nv = v;
#pragma unroll
                            for (int a = 0; a < 3; ++a)
                                if (a == best) {
                                    o[a] = Real(1) - at;
                                    di[a] -= inc;
                                }
                        }
                        if (changed) {
                            const Real sn = __ldg(t.s + c);
                            if (sn != sc) {
                                sc = sn;
#pragma unroll
                                for (int a = 0; a < 3; ++a) {
                                    d[a] = n[a] * sc;
                                    if (!(T[a] < kNever)) continue;
                                    const Real dist = d[a] > Real(0) ? Real(1) - o[a] : o[a];
                                    T[a] = tau + mul_rcp(dist, fabsf(d[a]));
                                }
                            }
                        }
                    }
                    v = nv;
                    fm = __ldg(g.faces + v);
                    if constexpr (IM != kInteractEC) {
                        if (refused) break;
                    }
                }
                if (IM == kInteractEC || !refused) {
                    const Real rem = Real(1) - tau;
#pragma unroll
                    for (int a = 0; a < 3; ++a) o[a] = clamp01(o[a] + rem * d[a]);
                    if (relax) kahan_add(A, Ac, rem * rate);
                }
            }
            if constexpr (IM == kInteractEC) {
                break;
            } else {
                if (!refused) break;
                if constexpr (MT) sat_any = sat_any || saturated(A);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    o[a] = o_s[a];
                    di[a] = di_s[a];
                }
                v = v_s;
                fm = fm_s;
                c = c_s;
                sc = sc_s;
                A = A_s;
                Ac = Ac_s;
                if constexpr (HASH) {
                    nev = nev_s;
                    ncr = ncr_s;
                    nrf = nrf_s;
                }
                if constexpr (MT) {
                    if (sat_any) saturate(A, Ac);  // a saturation met on a cancelled draw stays
                }
                if (IM == kInteractRS || ++att >= kMaxLeaps) {
                    // the walker stays for the step, in its label
                    if (relax) {
                        if constexpr (kF64)
                            A = A + rate0;
                        else
                            kahan_add(A, Ac, rate0);
                    }
                    if (IM == kInteractERL) atomicOr(ctl.status, kWarnLeaps);
                    if constexpr (HASH) ++nrf;
                    break;
                }
            }
        }  // draws
        if constexpr (HASH) {  // the verification kernel: checksum and, on request, invariants
            const uint64_t x =
                (((uint64_t)k & 0xFFFFu) << 48) ^ ((uint64_t)(uint32_t)c << 32) ^ (uint64_t)(uint32_t)v;
            h = mix64(h ^ x);
            if (ctl.checked) {
                int32_t at = 0;  // the flat index of the unwrapped coordinates
#pragma unroll
                for (int a = 0; a < 3; ++a) at += stride[a] * wrapped(st.i0[a][li] + di[a], N[a]);
                bool bad = v != at;
                // indices checked first
                if (!bad) bad = (int32_t)__ldg(g.labels + v) != c || fm != __ldg(g.faces + v) || sc != __ldg(t.s + c);
#pragma unroll
                for (int a = 0; a < 3; ++a) bad = bad || !(o[a] >= Real(0) && o[a] <= Real(1));
                if (bad) atomicOr(ctl.status, kErrInvariant);
            }
        }
        // ---- phase (Eq. 7, right end point of each step)
        if (graded) {
            const auto weight = [&](int s) { return NS == 1 ? wg : __ldg(t.wG + (int64_t)s * t.n_steps + (k - 1)); };
            if constexpr (kF64) {
#pragma unroll 1
                for (int r = 0; r < 3; ++r) {
                    ph.template add<SANE>(ctl.n_shapes, r,
                                          times<SANE>((double)di[0] + (o[0] - ph.start[r * kWalkBlock]), lp), weight);
                    rotate(o);
                    rotate(di);
                }
            } else {
                Real dx[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) dx[a] = lp * ((Real)di[a] + (o[a] - o0[a]));
                ph.add(ctl.n_shapes, dx, weight);
            }
        }
        // ---- displacement moments at recording steps (block-uniform branch)
        if (k == next_rec) {
            double dx[3];
            const auto start = [&](int a) -> double {
                if constexpr (kF64)
                    return ph.start[a * kWalkBlock];
                else
                    return (double)o0[a];
            };
#pragma unroll
            for (int a = 0; a < 3; ++a)
                dx[a] = g.voxel_um * ((double)di[a] + ((double)o[a] - start(a)));
            double al = 1.0;  // alpha = exp(-A); mostly A = 0 without relaxation
            if (A != Real(0)) al = kF64 ? exp(-(double)A) : exp(-((double)A - (double)Ac));
            if (!active) al = 0.0;
            warp_moments(al, dx, s_red[threadIdx.x >> 5]);
            __syncthreads();
            if (threadIdx.x < kMoments) {
                double acc = 0.0;
#pragma unroll
                for (int ww = 0; ww < kWalkWarps; ++ww) acc += s_red[ww][threadIdx.x];
                ctl.mom_partial[((int64_t)rec * ctl.n_blocks + block) * kMoments + threadIdx.x] = acc;
            }
            __syncthreads();
            ++rec;
            next_rec = rec < ctl.n_rec ? __ldg(t.rec_step + rec) : INT32_MAX;
        }
    }

    if (active) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            st.o[a][li] = o[a];
            st.di[a][li] = di[a];
        }
        st.c[li] = c;
        st.A[li] = A;
        if (!kF64) st.A_c[li] = Ac;
        ph.store(st, ctl.n_shapes, ctl.n_walkers, li);
        if constexpr (HASH) {
            st.hash[li] = h;
            if (st.counts) {
                st.counts[li] = nev;
                st.counts[ctl.n_walkers + li] = ncr;
                st.counts[2 * ctl.n_walkers + li] = nrf;
            }
        }
    }
}

// Resident blocks per SM the register allocation must allow (0: no bound,
// the compiler's choice).  The plain form's elastic-collision kernels: 7 (72
// registers, spills of a few words), whose warps hide the latency of long
// dependent chains: 3.3e5 walkers x 3000 steps 110.4 ms against 112.5 at 6.  The
// FP32 form's: as many blocks as their phases leave registers for without spills
// -- one shape 8 (64 registers: 21.8 ms for 1e6 walkers x 2000 steps on
// 200x200x400 axons against 22.0 ms at 9 with small spills and 22.5 ms at 7;
// absorbing membranes, 3e5 walkers x 3000 steps, 14.7 ms against 16.6 at 5), six
// shapes 5 (4e6 walkers x 1000 steps 75 ms against 88 with the kernel of eight
// at 4).  RS and ERL keep a step's start beside the state and would spill at 8.
template <typename Real, int NS, bool HASH, int IM, bool MT>
constexpr int walk_min_blocks()
{
    if (std::is_same<Real, double>::value) return HASH || IM != kInteractEC || MT ? 5 : 7;
    if (HASH) return NS == 1 && IM == kInteractEC && !MT ? 7 : 0;  // the verification kernel would spill at 8
    if (IM != kInteractEC) return NS == 1 && IM == kInteractRS && !MT ? 7 : 0;
    return NS == 1 ? 8 : NS == 2 ? (MT ? 7 : 8) : NS == 3 ? 7 : NS == 4 ? 6 : NS == 6 ? 5 : 4;
}

// One run: block b of the grid advances walkers b*kWalkBlock ... of the run.
template <typename Real, int NS, bool HASH, int IM, bool MT, int RELAX, bool SANE>
__global__ void __launch_bounds__(kWalkBlock, (walk_min_blocks<Real, NS, HASH, IM, MT>()))
walk_kernel(Geometry g, Tables<Real> t, WalkerState<Real> st, RunCtl ctl, int64_t k_begin, int64_t k_end, int32_t rec)
{
    walk_block<Real, NS, HASH, IM, MT, RELAX, true, SANE>(g, t, st, ctl, blockIdx.x, k_begin, k_end, rec);
}

// Many runs in one launch (continuous batching): block i executes task i --
// a block of walkers of one request for that request's next steps.  The
// request descriptors and the task table are read once per block.
template <typename Real, int NS>
__global__ void __launch_bounds__(kWalkBlock, std::is_same<Real, double>::value ? 5 : NS > 4 ? 4 : NS > 2 ? 6 : 8)
walk_batched_kernel(const ReqDesc<Real> *reqs, const BlockTask *tasks, int32_t n_tasks)
{
    if ((int32_t)blockIdx.x >= n_tasks) return;
    __shared__ ReqDesc<Real> s_req;
    __shared__ BlockTask s_task;
    if (threadIdx.x == 0) {
        s_task = tasks[blockIdx.x];
        s_req = reqs[s_task.req];
    }
    __syncthreads();
    walk_block<Real, NS, false, kInteractEC, false, 2>(s_req.g, s_req.t, s_req.st, s_req.ctl, s_task.block,
                                                       s_task.k0, s_task.k1, s_task.rec);
}

template <typename Real>
cudaError_t launch_walk_batched(int ns_bucket, int32_t n_tasks, cudaStream_t stream, const ReqDesc<Real> *reqs,
                                const BlockTask *tasks)
{
    if (n_tasks <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)n_tasks;
#define RMS_BATCHED(NS)                                                                                             \
    walk_batched_kernel<Real, NS>                                                                                   \
        <<<grid, kWalkBlock, Phases<Real, NS>::bytes(NS), stream>>>(reqs, tasks, n_tasks)
    if (ns_bucket <= 1)
        RMS_BATCHED(1);
    else if (ns_bucket <= 2)
        RMS_BATCHED(2);
    else if (ns_bucket <= 4)
        RMS_BATCHED(4);
    else
        RMS_BATCHED(8);
#undef RMS_BATCHED
    return cudaGetLastError();
}

// Resident blocks per SM of the batched kernel (the serving scheduler's
// count of block slots).
template <typename Real>
int batched_blocks_per_sm(int ns_bucket)
{
    int n = 0;
    cudaError_t e;
    if (ns_bucket <= 1)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, walk_batched_kernel<Real, 1>, kWalkBlock,
                                                          (Phases<Real, 1>::bytes(1)));
    else if (ns_bucket <= 2)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, walk_batched_kernel<Real, 2>, kWalkBlock,
                                                          (Phases<Real, 2>::bytes(2)));
    else if (ns_bucket <= 4)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, walk_batched_kernel<Real, 4>, kWalkBlock,
                                                          (Phases<Real, 4>::bytes(4)));
    else
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, walk_batched_kernel<Real, 8>, kWalkBlock,
                                                          (Phases<Real, 8>::bytes(8)));
    return e == cudaSuccess && n > 0 ? n : 1;
}

// Host-side launcher for interaction IM and absorbing membranes MT,
// instantiated in walk_fp64.cu / walk_fp32.cu (elastic collision),
// walk_reject_fp64.cu / walk_reject_fp32.cu (rejection sampling, ERL) and
// walk_mt_fp64.cu / walk_mt_fp32.cu (the three with absorbing membranes).
template <typename Real, int IM, bool MT>
cudaError_t launch_walk(int n_shapes, bool hash, dim3 grid, cudaStream_t stream, const Geometry &g,
                        const Tables<Real> &t, const WalkerState<Real> &st, const RunCtl &ctl,
                        int64_t k_begin, int64_t k_end, int32_t rec)
{
    // the checked products and quotients: the verification kernel, the other
    // interactions and absorbing membranes, and numbers out of range
    constexpr bool kSane = std::is_same<Real, double>::value && IM == kInteractEC && !MT;
#define RMS_LAUNCH_AS(NSV, HASHV, RELAXV, SANEV)                                                                \
    walk_kernel<Real, NSV, HASHV, IM, MT, RELAXV, SANEV>                                                        \
        <<<grid, kWalkBlock, Phases<Real, NSV>::bytes(n_shapes), stream>>>(g, t, st, ctl, k_begin, k_end, rec)
#define RMS_LAUNCH(NSV, HASHV, RELAXV)                                  \
    do {                                                                \
        if (kSane && !HASHV && ctl.sane)                                \
            RMS_LAUNCH_AS(NSV, HASHV, RELAXV, (kSane && !HASHV));       \
        else                                                            \
            RMS_LAUNCH_AS(NSV, HASHV, RELAXV, false);                   \
    } while (0)
// The plain form: one shape, or any (its phases are in shared memory).  The FP32
// form's elastic collision has kernels of three and six shapes too, whose phases
// leave registers for more blocks: 1e6 walkers x 1000 steps with T2, calls of three
// shapes 17.1 ms against 18.4 in the kernel of four, of five and six 22.6 and 23.3
// against 24.3 and 25.0 in that of eight; 1e5 walkers 2.35 against 2.40, 3.53 and 3.60
// against 3.46 and 3.55.  For one, two, four and eight shapes each has its own.
#define RMS_LAUNCH_NS(HASHV, RELAXV)                                                  \
    do {                                                                              \
        constexpr bool kMore = IM == kInteractEC && !MT && !HASHV;                    \
        if (n_shapes <= 1) {                                                          \
            RMS_LAUNCH(1, HASHV, RELAXV);                                             \
        } else if constexpr (std::is_same<Real, double>::value) {                     \
            RMS_LAUNCH(8, HASHV, RELAXV);                                             \
        } else {                                                                      \
            if (n_shapes <= 2)                                                        \
                RMS_LAUNCH(2, HASHV, RELAXV);                                         \
            else if (n_shapes <= (kMore ? 3 : 0))                                     \
                RMS_LAUNCH(kMore ? 3 : 4, HASHV, RELAXV);                             \
            else if (n_shapes <= 4)                                                   \
                RMS_LAUNCH(4, HASHV, RELAXV);                                         \
            else if (n_shapes <= (kMore ? 6 : 0))                                     \
                RMS_LAUNCH(kMore ? 6 : 8, HASHV, RELAXV);                             \
            else                                                                      \
                RMS_LAUNCH(8, HASHV, RELAXV);                                         \
        }                                                                             \
    } while (0)
    if (hash)
        RMS_LAUNCH_NS(true, 2);
    else if constexpr (IM != kInteractEC)
        RMS_LAUNCH_NS(false, 2);
    else if (t.any_relax)
        RMS_LAUNCH_NS(false, 1);
    else
        RMS_LAUNCH_NS(false, 0);
#undef RMS_LAUNCH_NS
#undef RMS_LAUNCH
#undef RMS_LAUNCH_AS
    return cudaGetLastError();
}

}  // namespace rms
