// Operands at which the integer-ALU FP64 arithmetic's rare branches are taken:
//   products  whose discarded bits are a unit or two from one half, and whose kept
//             bits end in 32 ones that the rounding carries through;
//   quotients and roots a few remainders from an integer, where the estimate may be a
//             unit off to either side (5 in 1e7 of random operands).
// They are solved for, not searched.
#pragma once

#include <cstdint>
#include <cstring>
#include <random>
#include <vector>

struct EdgeCase {
    int op;  // 0 product, 1 quotient, 2 root
    double a, b;
};

namespace edges {

typedef unsigned __int128 u128;
constexpr uint64_t kBit = 1ull << 52;  // the hidden bit

inline double number(uint64_t significand, int e, uint64_t sign = 0)
{
    const uint64_t u = sign << 63 | (uint64_t)e << 52 | (significand & (kBit - 1));
    double x;
    std::memcpy(&x, &u, 8);
    return x;
}

// a^-1 modulo 2^64 of an odd a: each step doubles the bits that agree.
inline uint64_t inverse_pow2(uint64_t a)
{
    uint64_t x = a;  // three bits
    for (int k = 0; k < 5; ++k) x *= 2 - a * x;
    return x;
}

// 2^-s modulo an odd B: halved s times.
inline uint64_t inverse_of_power(int s, uint64_t B)
{
    uint64_t x = 1;
    for (int k = 0; k < s; ++k) x = x & 1 ? (x + B) >> 1 : x >> 1;
    return x;
}

// A root of x modulo 2^64, x = 1 modulo 8.
inline uint64_t root_pow2(uint64_t x)
{
    uint64_t r = 1;
    for (int k = 3; k < 64; ++k)  // r^2 = x modulo 2^k
        if ((r * r - x) >> k & 1) r += 1ull << (k - 1);
    return r;
}

inline std::vector<EdgeCase> cases(int n, uint64_t seed)
{
    std::mt19937_64 g(seed);
    std::vector<EdgeCase> out;
    const auto significand = [&] { return kBit | (g() & (kBit - 1)); };
    for (int i = 0; i < n; ++i) {
        const int ea = 900 + (int)(g() % 100), eb = 900 + (int)(g() % 100), d = (int)(g() % 5) - 2;
        const uint64_t sa = g() & 1, sb = g() & 1;
        {  // the low 53 (or 52) bits of A B are one half of a unit, and d
            const uint64_t A = significand() | 1;
            for (const int low : {53, 52}) {
                const uint64_t T = (1ull << (low - 1)) + (uint64_t)(int64_t)d;
                const uint64_t B = (T * inverse_pow2(A) & ((1ull << low) - 1)) | (low == 52 ? kBit : 0);
                // low = 52: the hidden bit changes the product by A 2^52, 0 modulo 2^52
                if (B >= kBit) out.push_back({0, number(A, ea, sa), number(B, eb, sb)});
            }
        }
        {  // A B close to a kept part that ends in 32 ones, or in ones throughout
            const uint64_t A = significand(), ones = i & 1 ? 2 * kBit - 1 : significand() | 0xFFFFFFFFull;
            const u128 P = ((u128)ones << 53) + (1ull << 52);
            for (const int s : {0, 1}) {
                const u128 B = (P >> s) / A;
                if (B >= kBit && B < 2 * kBit)
                    for (int k = 0; k < 2; ++k)
                        if (B + k < 2 * kBit) out.push_back({0, number(A, ea, sa), number((uint64_t)B + k, eb, sb)});
            }
        }
        {  // A 2^s = r modulo B for a small r of either sign
            const uint64_t B = significand() | 1, r = g() % 64;
            for (const int s : {52, 53}) {
                const uint64_t R = i & 1 ? r : B - 1 - r;
                uint64_t A = (uint64_t)((u128)(R % B) * inverse_of_power(s, B) % B);
                if (s == 52) A += B;  // A >= B
                if (A >= kBit && A < 2 * kBit) out.push_back({1, number(A, ea), number(B, eb)});
            }
        }
        for (const int sh : {52, 53}) {  // M 2^sh = q^2 + r for a small r of either sign
            const int64_t r = 8 * ((int64_t)(g() % 16) - 8) + 7;  // -r = 1 modulo 8
            const uint64_t x = root_pow2((uint64_t)-r);
            const uint64_t turn[] = {x, 0 - x, x + (1ull << (sh - 1)), (1ull << (sh - 1)) - x};
            const uint64_t low = turn[g() % 4] & ((1ull << sh) - 1), q = sh == 52 ? kBit | low : low;
            const u128 X = (u128)q * q + (u128)(__int128)r;
            const uint64_t M = (uint64_t)(X >> sh);
            if (q >= kBit && M >= kBit && M < 2 * kBit && ((uint64_t)X & ((1ull << sh) - 1)) == 0)
                out.push_back({2, number(M, sh == 52 ? 1023 + 2 * (ea % 50) : 1022 + 2 * (ea % 50)), 0.0});
        }
    }
    return out;
}

}  // namespace edges
