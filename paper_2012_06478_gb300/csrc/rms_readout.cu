// rms_readout.cu -- the FP64 signal read-out (Eq. 7): for every (shape,
// direction, b) combination the sums over walkers of alpha cos(phi) and
// -alpha sin(phi), phi = q (g . Phi_s), q = sqrt(b / b_s), alpha = exp(-A);
// and the fixed-order sums over walker chunks of either form's read-out.
#include <cuda_pipeline.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "rms_internal.h"
#include "rms_readout.cuh"

namespace rms {

namespace {

__device__ const fix::Octant g_octant = fix::octant_table();

constexpr int kTile = 64;         // walkers staged at a time: their exact sums fit 64 bits
constexpr int kMaxThreads = 512;
constexpr int kMaxPairs = 130;    // (shape, direction) pairs of one block's combinations, at most
constexpr int kMinWalkers = 256;  // fewer: FP64 terms (their roundings are not averaged out)

// A tile's terms in FP64: phases or alphas outside the integers' range.
__device__ __noinline__ void plain_terms(const double *P, const double *al, int s, double q, double g0, double g1,
                                         double g2, int first, int step, int n, double &re, double &im)
{
    const double *p = P + 3 * s * kTile;
    for (int j = first; j < n; j += step) {
        const double phi = q * (g0 * p[j] + g1 * p[kTile + j] + g2 * p[2 * kTile + j]);
        double sn, cs;
        sincos(phi, &sn, &cs);
        re += al[j] * cs;
        im += -(al[j] * sn);
    }
}

// Grid: x a group of p.cpb combinations, y a chunk of p.per walkers.  A thread
// has one combination and every p.nsub-th walker of the chunk.
//
// What bounds it: issue (about 70 instructions a term, a third of them 32-bit
// products of 64 bits).  1e6 walkers x 330 combinations: RO_AFTER ms, against
// RO_BEFORE ms with sincos and sums on the FP64 pipe.  Tiles of 64 walkers go
// through shared memory twice -- the walkers' phases, copied asynchronously
// while the tile before is summed, and g.Phi of every pair in fixed point,
// shared by the pair's b-values -- beside the 64 KiB table, which two blocks an
// SM amortise over all their walkers.
__global__ void __launch_bounds__(kMaxThreads, 2) readout_fixed_kernel(ReadoutPlan p)
{
    extern __shared__ __align__(16) char smem[];
    fix::Angle *const table = (fix::Angle *)smem;
    const int K = 3 * p.S, row = K + 1;  // staged numbers of a walker: its phases and A
    double *const raw = (double *)(table + fix::kAngles);  // [2][row][kTile]
    double *const alD = raw + 2 * row * kTile;              // alpha of the tile
    fix::Words *const alF = (fix::Words *)(alD + kTile);   // in 58 bits of the largest
    int64_t *const X = (int64_t *)(alF + kTile);            // [kTile][pitch]
    int *const em = (int *)(X + kTile * p.pitch);           // per pair: the largest |g.Phi|'s exponent
    __shared__ double s_asum;
    __shared__ int s_ea;  // exponent of the tile's largest alpha; 0: FP64 terms

    for (int k = threadIdx.x; k < fix::kAngles; k += blockDim.x) table[k] = fix::angle_of(g_octant, k);

    const int64_t c0 = (int64_t)blockIdx.x * p.cpb;
    const int n_here = (int)min((int64_t)p.cpb, p.n_combo - c0);
    const int pair0 = (int)(c0 / p.n_b), n_pairs = (int)((c0 + n_here - 1) / p.n_b) - pair0 + 1;
    const int sub = threadIdx.x / p.cpb, mine = threadIdx.x - sub * p.cpb;
    const bool active = sub < p.nsub && mine < n_here;
    int s = 0, pair = 0;
    double q = 0.0, g0 = 0.0, g1 = 0.0, g2 = 0.0;
    if (active) {
        const int combo = (int)(c0 + mine), ib = combo % p.n_b;
        pair = combo / p.n_b;
        s = pair / p.n_dirs;
        q = p.q ? p.q[s * p.n_b + ib] : (p.b_s[s] > 0.0 ? sqrt(p.b[ib] / p.b_s[s]) : 0.0);
        const double *g = p.dirs + 3 * (pair - s * p.n_dirs);
        g0 = g[0];
        g1 = g[1];
        g2 = g[2];
        pair -= pair0;
    }
    const int64_t Q = fix::turns_of(q);

    const int64_t w0 = (int64_t)blockIdx.y * p.per, w1 = min(p.W, w0 + p.per);
    const auto stage = [&](int64_t base, double *to) {  // asynchronous copy of a tile's walkers
        const int nt = (int)min((int64_t)kTile, w1 - base);
        for (int e = threadIdx.x; e < row * kTile; e += blockDim.x) {
            // neighbouring threads take neighbouring numbers of memory
            const int j = p.sw == 1 ? e % kTile : e / row, k = p.sw == 1 ? e / kTile : e % row;
            if (j >= nt) continue;
            const double *from = k < K ? p.phase + (base + j) * p.sw + k * p.sk : p.A + base + j;
            __pipeline_memcpy_async(to + k * kTile + j, from, sizeof(double));
        }
        __pipeline_commit();
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = (blockDim.x + 31) >> 5;
    double re = 0.0, im = 0.0, asum = 0.0;
    stage(w0, raw);
    int at = 0;
    for (int64_t base = w0; base < w1; base += kTile, at ^= 1) {
        const int nt = (int)min((int64_t)kTile, w1 - base);
        double *const P = raw + at * row * kTile;
        __pipeline_wait_prior(0);
        __syncthreads();  // the tile has come, and the sums of the one before are done
        if (base + kTile < w1) stage(base + kTile, raw + (at ^ 1) * row * kTile);
        // a warp each: alpha, and g.Phi of one pair at a time
        for (int t = warp; t <= n_pairs; t += n_warps) {
            double x[2];
            if (t == n_pairs) {
                for (int h = 0; h < 2; ++h) x[h] = lane + 32 * h < nt ? exp(-P[K * kTile + lane + 32 * h]) : 0.0;
            } else {
                const int ps = (pair0 + t) / p.n_dirs;
                const double *g = p.dirs + 3 * (pair0 + t - ps * p.n_dirs), *v = P + 3 * ps * kTile;
                for (int h = 0; h < 2; ++h) {
                    const int j = lane + 32 * h;
                    x[h] = j < nt ? fma(g[2], v[2 * kTile + j], fma(g[1], v[kTile + j], g[0] * v[j])) : 0.0;
                }
            }
            const unsigned top = max((unsigned)(fix::double_word(x[0]) >> 32) & 0x7FFFFFFFu,
                                     (unsigned)(fix::double_word(x[1]) >> 32) & 0x7FFFFFFFu);
            const int e = (int)(__reduce_max_sync(0xffffffffu, top) >> 20);
            if (t == n_pairs) {
                // within 2^+-900: the scaled sums stay in range
                const bool fixed = e > 123 && e < 1923 && p.W >= kMinWalkers;
                double sum;
                if (fixed) {
                    uint64_t n = 0;  // 64 numbers below 2^58: exact
                    for (int h = 0; h < 2; ++h) {
                        const int64_t f = fix::scaled(x[h], e, 58);
                        alF[lane + 32 * h] = fix::words(f);
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
                for (int h = 0; h < 2; ++h) X[(lane + 32 * h) * p.pitch + t] = fix::scaled(x[h], e, 62);
                if (lane == 0) em[t] = e;
            }
        }
        __syncthreads();
        const int ea = s_ea;
        if (threadIdx.x == 0) asum += s_asum;
        if (active) {
            const fix::Scale sc = fix::scale_of(q, Q, em[pair]);
            if (q == 0.0 && em[pair] < 0x7FF) {  // b = 0: alpha's own sum, so that S = 1 exactly
                if (sub == 0) {
                    re += s_asum;
                    im -= 0.0 * s_asum;
                }
            } else if (sc.ok && ea) {
                int64_t c = 0, sn = 0;
                for (int j = sub; j < nt; j += p.nsub)
                    fix::add_term(X[j * p.pitch + pair], sc, alF[j], table, c, sn);
                const double scale = __longlong_as_double((long long)(ea - 55) << 52);  // 2^(ea - 1022 - 56)
                re += (double)c * scale;
                im -= (double)sn * scale;
            } else {
                plain_terms(P, alD, s, q, g0, g1, g2, sub, p.nsub, nt, re, im);
            }
        }
    }
    // over a combination's threads, in order
    __syncthreads();
    double *const red = (double *)smem;  // [nsub][cpb][2]: at most 8 KiB, where the table was
    if (active) {
        red[2 * threadIdx.x] = re;
        red[2 * threadIdx.x + 1] = im;
    }
    __syncthreads();
    double *const out = p.part + (int64_t)blockIdx.y * (p.n_combo + 1) * 2;
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
// eight warps take every eighth chunk each (one thread over all chunks took
// SUM_BEFORE us for 2442 chunks x 513 combinations, a chain of dependent FP64
// additions; eight at once, SUM_AFTER us).  NORM: the last column, the sum of
// alpha, divides the others (split real and imaginary parts, alpha_sum
// optional); otherwise all n_combo + 1 sums as they are.
constexpr int kSumWarps = 8;

template <bool NORM>
__global__ void __launch_bounds__(32 * kSumWarps)
chunk_sums_kernel(const double *part, int32_t n_chunks, int32_t n_combo, double *out_re, double *out_im, double *alpha)
{
    __shared__ double sh[kSumWarps][6][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t combo = (int64_t)blockIdx.x * 32 + lane;
    const bool active = NORM ? combo < n_combo : combo <= n_combo;
    double v[6] = {};  // sum and compensation of the real and imaginary parts and of alpha
    if (active) {
        for (int64_t k = warp; k < n_chunks; k += kSumWarps) {
            const double *row = part + k * (n_combo + 1) * 2;
            neumaier(v[0], v[1], row[2 * combo]);
            neumaier(v[2], v[3], row[2 * combo + 1]);
            if (NORM) neumaier(v[4], v[5], row[2 * (int64_t)n_combo]);
        }
        for (int i = 0; i < 6; ++i) sh[warp][i][lane] = v[i];
    }
    __syncthreads();
    if (warp != 0 || !active) return;
    for (int k = 1; k < kSumWarps; ++k)
        for (int i = 0; i < 6; i += 2) {
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
// block -- a whole wave of two blocks an SM for few groups, four waves (whose
// last is less empty) for many, whole tiles, at most max_chunks chunks.
ReadoutPlan readout_plan(int64_t W, int32_t S, int32_t n_dirs, int32_t n_b, int64_t max_chunks)
{
    ReadoutPlan p{};
    p.W = W;
    p.S = S;
    p.n_dirs = n_dirs;
    p.n_b = n_b;
    p.n_combo = S * n_dirs * n_b;
    const int64_t most = std::min<int64_t>(kMaxThreads, (int64_t)(kMaxPairs - 2) * n_b);
    int64_t groups = (p.n_combo + most - 1) / most;
    p.cpb = (int32_t)((p.n_combo + groups - 1) / groups);
    groups = (p.n_combo + p.cpb - 1) / p.cpb;
    p.nsub = std::min<int32_t>(kTile, kMaxThreads / p.cpb);
    p.threads = (p.cpb * p.nsub + 31) / 32 * 32;
    p.groups = (int32_t)groups;
    p.pitch = (int32_t)std::min<int64_t>((int64_t)S * n_dirs, (p.cpb - 1) / n_b + 2) | 1;  // odd: no bank conflicts
    constexpr int64_t kWave = 2 * 152;
    int64_t chunks = std::max<int64_t>(1, (groups <= 8 ? kWave : 4 * kWave) / groups);
    chunks = std::min(std::min(chunks, (W + kTile - 1) / kTile), max_chunks);
    p.per = ((W + chunks - 1) / chunks + kTile - 1) / kTile * kTile;
    p.n_chunks = (int32_t)((W + p.per - 1) / p.per);
    return p;
}

static constexpr size_t smem_bytes(int S, int pitch)
{
    return sizeof(fix::Angle) * fix::kAngles + sizeof(double) * 2 * (3 * S + 1) * kTile + 2 * sizeof(double) * kTile +
           sizeof(int64_t) * kTile * pitch + sizeof(int) * pitch;
}

cudaError_t launch_readout(const ReadoutPlan &p, cudaStream_t stream)
{
    // the largest any plan needs, so that host threads do not set different limits;
    // per context, and cheap: asked for at every launch
    constexpr size_t kMost = smem_bytes(kMaxShapes, kMaxPairs | 1);
    static_assert(kMost <= 227 * 1024, "shared memory of a block");
    const cudaError_t e =
        cudaFuncSetAttribute(readout_fixed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMost);
    if (e != cudaSuccess) return e;
    readout_fixed_kernel<<<dim3((unsigned)p.groups, (unsigned)p.n_chunks), p.threads, smem_bytes(p.S, p.pitch),
                           stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_chunk_sums(const double *part, int32_t n_chunks, int32_t n_combo, double *out, cudaStream_t stream)
{
    chunk_sums_kernel<false>
        <<<(unsigned)(n_combo / 32 + 1), 32 * kSumWarps, 0, stream>>>(part, n_chunks, n_combo, out, nullptr, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_chunk_sums_normalised(const double *part, int32_t n_chunks, int32_t n_combo, double *S_re,
                                         double *S_im, double *alpha_sum, cudaStream_t stream)
{
    chunk_sums_kernel<true><<<(unsigned)((n_combo + 31) / 32), 32 * kSumWarps, 0, stream>>>(
        part, n_chunks, n_combo, S_re, S_im, alpha_sum);
    return cudaGetLastError();
}

}  // namespace rms
