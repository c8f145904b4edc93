// Host check of the split sums (paper_2012_06478_gb300/csrc/f32x2.cuh): sums of up
// to 64 numbers of at most 1 against their exact values in integers.  Classes:
// random numbers, numbers at the splits' half ways, powers of two, and 64 times
// exactly 1 and -1, where the top level reaches the ends of its binade.  Prints the
// sums compared and the largest distance in units of 2^-48.
#include "../paper_2012_06478_gb300/csrc/f32x2.cuh"

#include <cstdio>
#include <random>

using namespace rms;

int main()
{
    std::mt19937_64 g(5);
    long sums = 0;
    long double worst = 0.0L;
    for (int r = 0; r < 300000; ++r) {
        const int n = r % 3 ? 64 : 1 + (int)(g() % 64);
        SplitSum sum;
        long double x0 = 0.0L, x1 = 0.0L;  // exact: 64 numbers of 24 bits above 2^-40
        for (int i = 0; i < n; ++i) {
            float v[2];
            for (float &x : v) {
                const float u = (float)((double)(g() >> 40) * 0x1p-24);  // [0, 1), a multiple of 2^-24
                switch (r % 7) {
                case 0: x = 1.0f; break;
                case 1: x = -1.0f; break;
                case 2: x = (g() & 1) ? 1.0f : -1.0f; break;
                case 3: x = 0x1p-17f * (float)(1 + (g() & 3)); break;          // half way at the first split
                case 4: x = -(0x1p-17f + 0x1p-34f * (float)(g() & 63)); break; // and at both
                case 5: x = u * word_float((uint32_t)(127 - g() % 17) << 23); break;
                default: x = 2.0f * u - 1.0f; break;
                }
            }
            x0 += v[0];
            x1 += v[1];
            sum.add(pair_of(v[0], v[1]));
        }
        const long double d0 = (long double)SplitSum::fixed(first(sum.a), first(sum.b), first(sum.c)) - x0 * 0x1p48L;
        const long double d1 = (long double)SplitSum::fixed(second(sum.a), second(sum.b), second(sum.c)) - x1 * 0x1p48L;
        worst = std::fmax(worst, std::fmax(std::fabs(d0), std::fabs(d1)));
        sums += 2;
    }
    std::printf("%ld %.3Lf\n", sums, worst);
    return 0;
}
