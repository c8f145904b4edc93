// rms_readout.cu -- the signal read-out (Eq. 7): for every (shape,
// direction, b) combination the sums over walkers of alpha cos(phi) and
// -alpha sin(phi), phi = q (g . Phi_s), q = sqrt(b / b_s), alpha = exp(-A), in
// the plain form's 64-bit terms or the FP32 form's 32-bit ones; and the
// fixed-order sums over walker chunks.
#include <cuda_pipeline.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "f32x2.cuh"
#include "rms_internal.h"
#include "rms_readout.cuh"

namespace rms {

namespace {

__device__ const fix::Octant g_octant = fix::octant_table();

constexpr int kTile = 64;         // walkers staged at a time: their exact sums fit 64 bits
constexpr int kMaxThreads = 512;
constexpr int kFewThreads = 128;  // below kMinWalkers
constexpr int kMaxPairs = 130;    // (shape, direction) pairs of one block's combinations, at most
constexpr int64_t kMostWalkers = 16384;  // of a chunk, but for a limit on chunks
constexpr int kMinWalkers = 256;  // fewer: floating-point terms (their roundings are not averaged out)

constexpr size_t kSums = sizeof(double) * 2 * kMaxThreads;  // the last sums, where the table was

// The forms' staged numbers: the plain form's terms are integers; the FP32
// form's single precision (phi, sincosf and the product with alpha), with sums
// that are exact but for the last places of a double.
template <typename Real>
struct Form;
template <>
struct Form<double> {
    using Alpha = fix::Words;
    using Phase = fix::Words;
    static constexpr int kBlocks = 2;  // resident blocks per SM
    static constexpr size_t kTable = sizeof(fix::Angle) * fix::kAngles;  // none below kMinWalkers
};
template <>
struct Form<float> {
    using Alpha = float;
    using Phase = float;
    static constexpr int kBlocks = 3;
    static constexpr size_t kTable = kSums;
};

// alpha given in 58 bits of a power of two
__device__ __forceinline__ void put(fix::Words &to, double, int64_t bits, int) { to = fix::words(bits); }
// alpha over that power of two, below 1: x 2^(1022 - e)
__device__ __forceinline__ void put(float &to, double al, int64_t, int e)
{
    to = (float)((double)(float)al * __longlong_as_double((long long)(2045 - e) << 52));
}

// The biased double exponent of the largest |x| of a warp's pairs of numbers.
__device__ __forceinline__ int top_exponent(double a, double b)
{
    const unsigned u = (unsigned)(fix::double_word(a) >> 32) & 0x7FFFFFFFu;
    const unsigned v = (unsigned)(fix::double_word(b) >> 32) & 0x7FFFFFFFu;
    return (int)(__reduce_max_sync(0xffffffffu, max(u, v)) >> 20);
}

// g.Phi of walker j's staged phases (the FP32 form's with their compensations).
__device__ __forceinline__ double dot(const double *v, int, int j, const double *g)
{
    return fma(g[2], v[2 * kTile + j], fma(g[1], v[kTile + j], g[0] * v[j]));
}
__device__ __forceinline__ float dot(const float *v, int K, int j, const double *g)
{
    const float *c = v + K * kTile;
    return fmaf((float)g[2], v[2 * kTile + j] - c[2 * kTile + j],
                fmaf((float)g[1], v[kTile + j] - c[kTile + j], (float)g[0] * (v[j] - c[j])));
}

// A tile's sums in floating point: phases or alphas outside the integers' range.
__device__ __noinline__ double2 plain_sums(const double *v, int, const double *al, double q, const double *g, int first,
                                           int step, int n)
{
    double re = 0.0, im = 0.0;
    for (int j = first; j < n; j += step) {
        const double phi = q * (g[0] * v[j] + g[1] * v[kTile + j] + g[2] * v[2 * kTile + j]);
        double sn, cs;
        sincos(phi, &sn, &cs);
        re += al[j] * cs;
        im += -(al[j] * sn);
    }
    return make_double2(re, im);
}
__device__ __noinline__ double2 plain_sums(const float *v, int K, const double *al, double q, const double *g,
                                           int first, int step, int n)
{
    double re = 0.0, im = 0.0;
    for (int j = first; j < n; j += step) {
        const float phi = (float)q * dot(v, K, j, g);
        float sn, cs;
        sincosf(phi, &sn, &cs);
        re += (double)((float)al[j] * cs);
        im += (double)-((float)al[j] * sn);
    }
    return make_double2(re, im);
}

template <typename Real>
__host__ __device__ constexpr size_t table_bytes(int64_t W)
{
    return W >= kMinWalkers ? Form<Real>::kTable : kSums;
}

template <typename Real>
constexpr size_t smem_bytes(int64_t W, int S, int pitch)
{
    using F = Form<Real>;
    const int rows = (sizeof(Real) == 8 ? 1 : 2) * (3 * S + 1);
    return table_bytes<Real>(W) + sizeof(double) * kTile + sizeof(Real) * 2 * rows * kTile +
           sizeof(typename F::Alpha) * kTile + sizeof(typename F::Phase) * kTile * pitch + sizeof(int) * pitch;
}

// Grid: x a group of p.cpb combinations, y and z a chunk of p.per walkers (the
// groups of a chunk run together and share its walkers in the L2).  A thread has one
// combination and every p.nsub-th walker of the chunk.
//
// What bounds it: issue, and the pipe of the 32-bit products (plain form, 1e6
// walkers x 330 combinations: 59 % and 72 % used).  2.77 ms there, against 25.6
// with sincos and sums on the FP64 pipe; the FP32 form, whose sums on the FP64
// pipe took 31.9 ms for 1e7 walkers x 512 combinations, 11.7 ms.
// Tiles of 64 walkers go through shared memory twice -- the walkers' phases,
// copied asynchronously while the tile before is summed, and g.Phi of every
// pair (the plain form's in fixed point), shared by the pair's b-values; the
// table of the plain form is amortised over all of a block's walkers.
template <typename Real>
__global__ void __launch_bounds__(kMaxThreads, Form<Real>::kBlocks) readout_fixed_kernel(ReadoutPlan<Real> p)
{
    using F = Form<Real>;
    constexpr bool kF64 = sizeof(Real) == 8;
    extern __shared__ __align__(16) char smem[];
    auto *const table = (fix::Angle *)smem;  // plain form
    // staged numbers of a walker: its phases and A (FP32 form: phases, compensations, A and A's)
    const int K = 3 * p.S, KA = kF64 ? K : 2 * K, rows = kF64 ? K + 1 : 2 * K + 2;
    double *const alD = (double *)(smem + table_bytes<Real>(p.W));    // alpha of the tile
    Real *const raw = (Real *)(alD + kTile);                          // [2][rows][kTile]
    auto *const alF = (typename F::Alpha *)(raw + 2 * rows * kTile);  // over a power of two above the largest
    auto *const X = (typename F::Phase *)(alF + kTile);               // [kTile][pitch]
    int *const em = (int *)(X + kTile * p.pitch);                     // per pair: the largest |g.Phi|'s exponent
    __shared__ double s_asum;
    __shared__ int s_ea;  // exponent of the tile's largest alpha; 0: floating-point terms

    if (kF64 && p.W >= kMinWalkers)  // fewer: no term takes it
        for (int k = threadIdx.x; k < fix::kAngles; k += blockDim.x) table[k] = fix::angle_of(g_octant, k);

    const int64_t chunk = (int64_t)blockIdx.z * gridDim.y + blockIdx.y;
    if (chunk >= p.n_chunks) return;  // block-uniform
    const int64_t c0 = (int64_t)blockIdx.x * p.cpb;
    const int n_here = (int)min((int64_t)p.cpb, p.n_combo - c0);
    const int pair0 = (int)(c0 / p.n_b), n_pairs = (int)((c0 + n_here - 1) / p.n_b) - pair0 + 1;
    const int sub = threadIdx.x / p.cpb, mine = threadIdx.x - sub * p.cpb;
    const bool active = sub < p.nsub && mine < n_here;
    int s = 0, pair = 0;
    double q = 0.0;
    const double *g = p.dirs;
    if (active) {
        const int combo = (int)(c0 + mine), ib = combo % p.n_b;
        pair = combo / p.n_b;
        s = pair / p.n_dirs;
        q = p.q ? p.q[s * p.n_b + ib] : (p.b_s[s] > 0.0 ? sqrt(p.b[ib] / p.b_s[s]) : 0.0);
        g = p.dirs + 3 * (pair - s * p.n_dirs);
        pair -= pair0;
    }
    const int64_t Q = fix::turns_of(q);
    // the pairs' g.Phi: of few walkers only what b = 0 asks for, whether it is finite
    const bool pairs = __syncthreads_or(active && q == 0.0) || p.W >= kMinWalkers;

    const int64_t w0 = chunk * p.per, w1 = min(p.W, w0 + p.per);
    const auto stage = [&](int64_t base, Real *to) {  // asynchronous copy of a tile's walkers
        const int nt = (int)min((int64_t)kTile, w1 - base);
        for (int e = threadIdx.x; e < rows * (p.sw == 1 ? kTile : nt); e += blockDim.x) {
            // neighbouring threads take neighbouring numbers of memory
            const int j = p.sw == 1 ? e % kTile : e / rows, k = p.sw == 1 ? e / kTile : e % rows;
            if (j >= nt) continue;
            const Real *from;
            if (k < K)
                from = p.phase + (base + j) * p.sw + k * p.sk;
            else if (k < KA)
                from = p.phase_c + (base + j) * p.sw + (k - K) * p.sk;
            else
                from = (k == KA ? p.A : p.A_c) + base + j;
            __pipeline_memcpy_async(to + k * kTile + j, from, sizeof(Real));
        }
        __pipeline_commit();
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = (blockDim.x + 31) >> 5;
    double re = 0.0, im = 0.0, asum = 0.0;
    // FP32 form: the sums of the tiles so far that had their alphas' exponent, 48 fraction
    // bits; a tile's is at most 64, a chunk's at most 2^62 in all (launch_readout)
    [[maybe_unused]] int64_t re48 = 0, im48 = 0;
    [[maybe_unused]] int ea48 = 0;
    [[maybe_unused]] const auto flush = [&] {
        const double scale = __longlong_as_double((long long)(ea48 - 47) << 52);  // 2^(ea48 - 1022 - 48)
        re += (double)re48 * scale;
        im -= (double)im48 * scale;
        re48 = im48 = 0;
    };
    stage(w0, raw);
    int at = 0;
    for (int64_t base = w0; base < w1; base += kTile, at ^= 1) {
        const int nt = (int)min((int64_t)kTile, w1 - base);
        Real *const P = raw + at * rows * kTile;
        __pipeline_wait_prior(0);
        __syncthreads();  // the tile has come, and the sums of the one before are done
        if (base + kTile < w1) stage(base + kTile, raw + (at ^ 1) * rows * kTile);
        // a warp each: alpha, and g.Phi of one pair at a time
        for (int t = pairs ? warp : n_pairs + warp; t <= n_pairs; t += n_warps) {
            if (t == n_pairs) {
                double x[2];
                for (int h = 0; h < 2; ++h) {
                    const int j = lane + 32 * h;
                    double a = j < nt ? (double)P[KA * kTile + j] : 0.0;
                    if (!kF64 && j < nt) a = a - (double)P[(KA + 1) * kTile + j];
                    // kSaturatedF (saturated, FP32 form): exp underflows to 0
                    x[h] = j < nt ? exp(-a) : 0.0;
                }
                const int e = top_exponent(x[0], x[1]);
                // within 2^+-900: the scaled sums stay in range
                const bool fixed = e > 123 && e < 1923 && p.W >= kMinWalkers;
                double sum;
                if (fixed) {
                    uint64_t n = 0;  // 64 numbers below 2^58: exact
                    for (int h = 0; h < 2; ++h) {
                        const int64_t f = fix::scaled(x[h], e, 58);
                        put(alF[lane + 32 * h], x[h], f, e);
                        n += (uint64_t)f;
                    }
                    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
                    sum = (double)n * __longlong_as_double((long long)(e - 57) << 52);  // 2^(e - 1022 - 58)
                } else {
                    sum = x[0] + x[1];
                    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                }
                alD[lane] = x[0];
                alD[lane + 32] = x[1];
                if (lane == 0) {
                    s_asum = sum;
                    s_ea = fixed ? e : 0;
                }
            } else {
                const int ps = (pair0 + t) / p.n_dirs;
                const double *gt = p.dirs + 3 * (pair0 + t - ps * p.n_dirs);
                Real x[2];
                for (int h = 0; h < 2; ++h)
                    x[h] = lane + 32 * h < nt ? dot(P + 3 * ps * kTile, K, lane + 32 * h, gt) : Real(0);
                if constexpr (kF64) {
                    const int e = top_exponent(x[0], x[1]);
                    for (int h = 0; h < 2; ++h) X[(lane + 32 * h) * p.pitch + t] = fix::words(fix::scaled(x[h], e, 62));
                    if (lane == 0) em[t] = e;
                } else {
                    for (int h = 0; h < 2; ++h) X[(lane + 32 * h) * p.pitch + t] = x[h];
                }
            }
        }
        __syncthreads();
        const int ea = s_ea;
        if (threadIdx.x == 0) asum += s_asum;
        if (active) {
            bool alphas;  // b = 0: alpha's own sum, so that S = 1 exactly
            bool fixed = ea != 0;
            fix::Scale sc;
            if constexpr (kF64) {
                sc = fix::scale_of(q, Q, em[pair]);
                alphas = q == 0.0 && em[pair] < 0x7FF;
                fixed = fixed && sc.ok;
            } else {
                alphas = (float)q == 0.0f;
            }
            if (alphas) {
                if (sub == 0) {
                    re += s_asum;
                    if constexpr (kF64) im -= 0.0 * s_asum;
                }
            } else if (fixed) {
                if constexpr (kF64) {
                    int64_t c = 0, sn = 0;
#pragma unroll 4
                    for (int j = sub; j < nt; j += p.nsub)
                        fix::add_term(X[j * p.pitch + pair], sc, alF[j], table, c, sn);
                    const double scale = __longlong_as_double((long long)(ea - 55) << 52);  // 2^(ea - 1022 - 56)
                    re += (double)c * scale;
                    im -= (double)sn * scale;
                } else {
                    SplitSum sum;
                    const float qq = (float)q;
#pragma unroll 2
                    for (int j = sub; j < nt; j += p.nsub) {
                        float sn, cs;
                        sincosf(qq * X[j * p.pitch + pair], &sn, &cs);
                        sum.add(pair_of(alF[j] * cs, alF[j] * sn));
                    }
                    if (ea != ea48) {
                        if (ea48) flush();
                        ea48 = ea;
                    }
                    // a phase that is not finite makes the sum NaN, not an integer
                    if (isnan(first(sum.c)) || isnan(second(sum.c))) {
                        re += (double)first(sum.c);
                        im += (double)second(sum.c);
                    } else {
                        re48 += SplitSum::fixed(first(sum.a), first(sum.b), first(sum.c));
                        im48 += SplitSum::fixed(second(sum.a), second(sum.b), second(sum.c));
                    }
                }
            } else {
                const double2 r = plain_sums(P + 3 * s * kTile, K, alD, q, g, sub, p.nsub, nt);
                re += r.x;
                im += r.y;
            }
        }
    }
    if constexpr (!kF64)
        if (ea48) flush();
    // over a combination's threads, in order
    __syncthreads();
    double *const red = (double *)smem;  // [nsub][cpb][2]: at most 8 KiB, where the table was
    if (active) {
        red[2 * threadIdx.x] = re;
        red[2 * threadIdx.x + 1] = im;
    }
    __syncthreads();
    double *const out = p.part + chunk * (p.n_combo + 1) * 2;
    if (active && sub == 0) {
        for (int k = 1; k < p.nsub; ++k) {
            re += red[2 * (k * p.cpb + mine)];
            im += red[2 * (k * p.cpb + mine) + 1];
        }
        out[2 * (c0 + mine)] = re;
        out[2 * (c0 + mine) + 1] = im;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        out[2 * (int64_t)p.n_combo] = asum;
        out[2 * (int64_t)p.n_combo + 1] = 0.0;
    }
}

__device__ __forceinline__ void neumaier(double &sum, double &comp, double x)
{
    const double t = sum + x;
    if (fabs(sum) >= fabs(x))
        comp += (sum - t) + x;
    else
        comp += (x - t) + sum;
    sum = t;
}

// Sums over walker chunks in a fixed order.  A block has 32 combinations; its
// warps, eight at most, take every eighth chunk each (one thread over all chunks took
// 233 us for 2442 chunks x 513 combinations, a chain of dependent FP64
// additions; eight at once, and fewer chunks, 48 us).  NORM: the last column,
// the sum of alpha, divides the others (split real and imaginary parts,
// alpha_sum optional); otherwise all n_combo + 1 sums as they are.
constexpr int kSumWarps = 8;

template <bool NORM>
__global__ void __launch_bounds__(32 * kSumWarps)
chunk_sums_kernel(const double *part, int32_t n_chunks, int32_t n_combo, double *out_re, double *out_im, double *alpha)
{
    __shared__ double sh[kSumWarps][6][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int64_t combo = (int64_t)blockIdx.x * 32 + lane;
    const bool active = NORM ? combo < n_combo : combo <= n_combo;
    double v[6] = {};  // sum and compensation of the real and imaginary parts and of alpha
    if (active) {
        for (int64_t k = warp; k < n_chunks; k += warps) {
            const double *row = part + k * (n_combo + 1) * 2;
            neumaier(v[0], v[1], row[2 * combo]);
            neumaier(v[2], v[3], row[2 * combo + 1]);
            if (NORM) neumaier(v[4], v[5], row[2 * (int64_t)n_combo]);
        }
        for (int i = 0; i < 6; ++i) sh[warp][i][lane] = v[i];
    }
    __syncthreads();
    if (warp != 0 || !active) return;
    for (int k = 1; k < warps; ++k)
        for (int i = 0; i < (NORM ? 6 : 4); i += 2) {
            neumaier(v[i], v[i + 1], sh[k][i][lane]);
            v[i + 1] += sh[k][i + 1][lane];
        }
    if (NORM) {
        const double a = v[4] + v[5];
        out_re[combo] = (v[0] + v[1]) / a;
        out_im[combo] = (v[2] + v[3]) / a;
        if (combo == 0 && alpha) *alpha = a;
    } else {
        out_re[2 * combo] = v[0] + v[1];
        out_re[2 * combo + 1] = v[2] + v[3];
    }
}

}  // namespace

// How the read-out splits: combinations a block (one group when they fit its
// threads, at most kMaxPairs pairs), threads a combination, and walkers a
// block -- a whole wave of the blocks that are resident for few groups, four
// waves (whose last is less empty) for many, whole tiles, at most max_chunks.
// Below kMinWalkers a thread's chain of sincos takes the time: blocks of kFewThreads,
// of as few combinations as leave two blocks an SM (100 walkers x 330 combinations 32 us
// against 249 in one block of 352 threads a tile, 1 x 6 21.9 against 34.6).  The
// plain form's sums and the sum of alpha add a chunk's tiles one after another in
// FP64, which is off by n / 8 sqrt(W) for chunks of n walkers where sums over 4096
// single walkers are off by 4096 / sqrt(W): as many times the chunks, where one would
// be longer than half of 8 x 4096 (plain form, 1e6 walkers x 131 072 combinations:
// 5.6 2^-53 off in the mean square with 4 chunks, 0.88 with sums over 4096, 0.65 with
// 64; the same time).
template <typename Real>
ReadoutPlan<Real> readout_plan(int64_t W, int32_t S, int32_t n_dirs, int32_t n_b, int64_t max_chunks)
{
    ReadoutPlan<Real> p{};
    p.W = W;
    p.S = S;
    p.n_dirs = n_dirs;
    p.n_b = n_b;
    p.n_combo = S * n_dirs * n_b;
    const int64_t tiles = (W + kTile - 1) / kTile;
    const bool few = W < kMinWalkers;
    const int64_t threads = few ? kFewThreads : kMaxThreads, lanes = std::min<int64_t>(kTile, W);
    int64_t most = std::min<int64_t>(threads, (int64_t)(kMaxPairs - 2) * n_b);
    if (few) most = std::min(most, std::max(threads / lanes, p.n_combo * tiles / (2 * 152)));
    int64_t groups = (p.n_combo + most - 1) / most;
    p.cpb = (int32_t)((p.n_combo + groups - 1) / groups);
    groups = (p.n_combo + p.cpb - 1) / p.cpb;
    p.nsub = (int32_t)std::min(lanes, threads / p.cpb);
    p.threads = (p.cpb * p.nsub + 31) / 32 * 32;
    p.groups = (int32_t)groups;
    p.pitch = (int32_t)std::min<int64_t>((int64_t)S * n_dirs, (p.cpb - 1) / n_b + 2) | 1;  // odd: no bank conflicts
    constexpr int64_t kWave = Form<Real>::kBlocks * 152;
    int64_t chunks = std::max<int64_t>(1, (groups <= 8 ? kWave : 4 * kWave) / groups);
    chunks *= (W + chunks * kMostWalkers - 1) / (chunks * kMostWalkers);
    chunks = std::min(std::min(chunks, tiles), max_chunks);
    p.per = ((W + chunks - 1) / chunks + kTile - 1) / kTile * kTile;
    p.n_chunks = (int32_t)((W + p.per - 1) / p.per);
    return p;
}

template <typename Real>
cudaError_t launch_readout(const ReadoutPlan<Real> &p, cudaStream_t stream)
{
    // the FP32 form's integer sums have room for chunks of this length
    static_assert((kMostWalkers / kTile) * (64ll << 48) <= 1ll << 62, "integer sums of a chunk");
    if (sizeof(Real) == 4 && p.per > kMostWalkers) return cudaErrorInvalidValue;
    // the largest any plan needs, so that host threads do not set different limits;
    // per context, and cheap: asked for at every launch
    constexpr size_t kMost = smem_bytes<Real>(kMinWalkers, kMaxShapes, kMaxPairs | 1);
    static_assert(kMost <= 227 * 1024, "shared memory of a block");
    const cudaError_t e =
        cudaFuncSetAttribute(readout_fixed_kernel<Real>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMost);
    if (e != cudaSuccess) return e;
    const unsigned ny = (unsigned)std::min(p.n_chunks, 32768);
    const dim3 grid((unsigned)p.groups, ny, ((unsigned)p.n_chunks + ny - 1) / ny);
    readout_fixed_kernel<Real><<<grid, p.threads, smem_bytes<Real>(p.W, p.S, p.pitch), stream>>>(p);
    return cudaGetLastError();
}

template ReadoutPlan<double> readout_plan<double>(int64_t, int32_t, int32_t, int32_t, int64_t);
template ReadoutPlan<float> readout_plan<float>(int64_t, int32_t, int32_t, int32_t, int64_t);
template cudaError_t launch_readout<double>(const ReadoutPlan<double> &, cudaStream_t);
template cudaError_t launch_readout<float>(const ReadoutPlan<float> &, cudaStream_t);

cudaError_t launch_chunk_sums(const double *part, int32_t n_chunks, int32_t n_combo, double *out, cudaStream_t stream)
{
    chunk_sums_kernel<false>
        <<<(unsigned)(n_combo / 32 + 1), 32 * std::min(kSumWarps, n_chunks), 0, stream>>>(part, n_chunks, n_combo, out, nullptr, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_chunk_sums_normalised(const double *part, int32_t n_chunks, int32_t n_combo, double *S_re,
                                         double *S_im, double *alpha_sum, cudaStream_t stream)
{
    chunk_sums_kernel<true><<<(unsigned)((n_combo + 31) / 32), 32 * std::min(kSumWarps, n_chunks), 0, stream>>>(
        part, n_chunks, n_combo, S_re, S_im, alpha_sum);
    return cudaGetLastError();
}

}  // namespace rms
