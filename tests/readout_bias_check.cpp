// Host check of the fixed-point read-out's phases (rms_readout.cuh): the mean over
// many terms of their phase's error -- the error of a term along e^{-i phi}'s
// derivative -- for amplitudes of several low words.  Prints, for each exponent of
// the largest phase, the largest mean and the unit of a phase before its shift, in
// radians.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "rms_readout.cuh"

using namespace rms;

static constexpr fix::Octant kOctant = fix::octant_table();

int main()
{
    std::vector<fix::Angle> table(fix::kAngles);
    for (int k = 0; k < fix::kAngles; ++k) table[k] = fix::angle_of(kOctant, k);
    std::mt19937_64 g(7);
    std::uniform_real_distribution<double> U(-1, 1);
    const fix::Words one = fix::words(1LL << 57);  // alpha: 0.5 in 58 bits
    for (int e2 = -6; e2 <= 8; ++e2) {
        double worst = 0.0;
        int shift = 0;
        for (int trial = 0; trial < 8; ++trial) {
            const double q = std::exp(3.0 * U(g)), most = std::ldexp(1.0, e2) / q;
            const int em = (int)(fix::double_word(1.999 * most) >> 52);
            const fix::Scale sc = fix::scale_of(q, fix::turns_of(q), em);
            if (!sc.ok) continue;
            shift = std::max(shift, (int)sc.shift);
            const int n = 1 << 18;
            long double sum = 0.0L;
            for (int i = 0; i < n; ++i) {
                const double x = 1.999 * most * U(g);
                int64_t re = 0, im = 0;
                fix::add_term(fix::scaled(x, em, 62), sc, one, table.data(), re, im);
                const long double phi = (long double)q * x, u = std::ldexp(1.0L, -55);
                const long double c = cosl(phi), s = sinl(phi);
                sum += (im * u - s) * c - (re * u - c) * s;
            }
            worst = std::max(worst, (double)std::fabs(sum / n));
        }
        std::printf("%d %.3e %.3e\n", e2, worst, std::ldexp(6.283185307179586, shift - 64));
    }
    return 0;
}
