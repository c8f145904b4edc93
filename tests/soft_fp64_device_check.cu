// The integer-ALU FP64 products, quotients and square roots
// (paper_2012_06478_gb300/csrc/soft_fp64.cuh) as the GPU computes them, against
// the GPU's own IEEE operations: products with exact ties, with every carry of
// the rounding (all-ones kept parts, kept parts of zeros), of random and of
// extreme significands; quotients and roots a unit around a rounding midpoint; and
// the operands of soft_fp64_edges.h.  Prints the cases compared and the mismatches of each; exit status 1 on a
// mismatch.
#include <cstdio>

#include "../paper_2012_06478_gb300/csrc/soft_fp64.cuh"
#include "soft_fp64_edges.h"

using namespace rms::sfp;

__device__ uint64_t mixed(uint64_t x)  // splitmix64's output function (Steele, Lea & Flood 2014)
{
    x += 0x9E3779B97F4A7C15ULL;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
    return x ^ (x >> 31);
}
__device__ double number(uint64_t mant, int e, uint64_t sign)
{
    return double_of((sign << 63) | ((uint64_t)e << 52) | (mant & kMant));
}

struct Count {
    unsigned long long tested[3], bad[3];  // products, quotients, roots
};

__device__ void compare(Count *n, int which, double got, double want)
{
    atomicAdd(&n->tested[which], 1ULL);
    if (bits_of(got) != bits_of(want)) atomicAdd(&n->bad[which], 1ULL);
}

__global__ void check(long cases, Count *n)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < cases; i += (long)gridDim.x * blockDim.x) {
        uint64_t r[4];
        for (int k = 0; k < 4; ++k) r[k] = mixed(4 * (uint64_t)i + k);
        const uint64_t H = kHidden, ends[] = {H, H + 1, 2 * H - 1, 2 * H - 2, H | 0xFFFFFFFFULL, 2 * H - (1ULL << 32)};
        uint64_t a = r[0], b = r[1];
        switch (i % 5) {
        case 1:  // 27 and 27 bits: the part below the kept bits is often one half
            a = (a >> 37) << 25;
            b = (b >> 37) << 25;
            break;
        case 2: a = ends[r[2] % 6]; break;
        case 3:
            a = ends[r[2] % 6];
            b = ends[r[3] % 6];
            break;
        case 4: {  // a product around a kept part of ones: b ~ (2^54 - 1 or 2^53 - 1) 2^52 / a
            a = H | (a & kMant);
            const uint64_t kept = (r[2] & 1) ? 2 * H - 1 : H;
            uint64_t hi = kept >> 12, lo = kept << 52, q = 0;  // kept 2^52
            for (int bit = 0; bit < 64; ++bit) {               // long division, the quotient below 2^54
                const uint64_t top = (hi << 1) | (lo >> 63);
                lo <<= 1;
                const bool ge = top >= a;
                hi = ge ? top - a : top;
                q = (q << 1) | ge;
            }
            if (q < H) q = 2 * q + (r[3] >> 32 & 1);
            b = q + (r[3] % 3) - 1;
            break;
        }
        default: break;
        }
        const double x = number(a, 700 + (int)(r[2] >> 8 & 511), r[2] >> 63);
        const double y = number(b, 700 + (int)(r[3] >> 8 & 511), r[3] >> 63);
        const double p = __dmul_rn(x, y);
        compare(n, 0, mul_normal(x, y), p);
        double checked = 0.0;
        if (mul_rn(x, y, checked)) compare(n, 0, checked, p);
        const double ax = fabs(x), ay = fabs(y);
        compare(n, 1, div_normal(ax, ay), __ddiv_rn(ax, ay));
        // around the midpoint above a random quotient and root
        const double m = __dmul_rn(__dadd_rn(number(r[2], 1023, 0), 0x1p-53), number(b, 1023, 0));
        for (int k = -1; k <= 1; ++k) {
            const double v = double_of(bits_of(m) + (uint64_t)(int64_t)k);
            compare(n, 1, div_normal(v, number(b, 1023, 0)), __ddiv_rn(v, number(b, 1023, 0)));
            const double s = double_of(bits_of(__dmul_rn(ax, ax)) + (uint64_t)(int64_t)k);
            compare(n, 2, sqrt_normal(s), __dsqrt_rn(s));
        }
        compare(n, 2, sqrt_normal(ax), __dsqrt_rn(ax));
    }
}

__global__ void check_edges(const EdgeCase *c, long cases, Count *n)
{
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= cases) return;
    const double a = c[i].a, b = c[i].b;
    if (c[i].op == 0)
        compare(n, 0, mul_normal(a, b), __dmul_rn(a, b));
    else if (c[i].op == 1)
        compare(n, 1, div_normal(a, b), __ddiv_rn(a, b));
    else
        compare(n, 2, sqrt_normal(a), __dsqrt_rn(a));
}

int main()
{
    Count *n = nullptr, h{};
    if (cudaMalloc((void **)&n, sizeof *n) != cudaSuccess || cudaMemset(n, 0, sizeof *n) != cudaSuccess) return 2;
    check<<<608, 128>>>(2000000, n);
    const std::vector<EdgeCase> e = edges::cases(200000, 4);
    EdgeCase *d = nullptr;
    if (cudaMalloc((void **)&d, sizeof(EdgeCase) * e.size()) != cudaSuccess ||
        cudaMemcpy(d, e.data(), sizeof(EdgeCase) * e.size(), cudaMemcpyHostToDevice) != cudaSuccess)
        return 2;
    check_edges<<<(unsigned)((e.size() + 127) / 128), 128>>>(d, (long)e.size(), n);
    if (cudaGetLastError() != cudaSuccess || cudaMemcpy(&h, n, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    for (int k = 0; k < 3; ++k) std::printf("%llu %llu\n", h.tested[k], h.bad[k]);
    return h.bad[0] || h.bad[1] || h.bad[2] ? 1 : 0;
}
