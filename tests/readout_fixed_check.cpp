// Host check of the fixed-point read-out terms (rms_readout.cuh) and of the
// 32-at-a-time additions (serial_sum.cuh) against long double and plain loops.
// Prints "term <e2> <largest error> <mean error>" lines and "chain <differences>".
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "rms_readout.cuh"
#include "serial_sum.cuh"

using namespace rms;

static constexpr fix::Octant kOctant = fix::octant_table();

static void terms()
{
    std::vector<fix::Angle> table(fix::kAngles);
    for (int k = 0; k < fix::kAngles; ++k) table[k] = fix::angle_of(kOctant, k);
    std::mt19937_64 g(1);
    std::uniform_real_distribution<double> U(-1, 1);
    for (int e2 = -6; e2 <= 20; ++e2) {
        double largest = 0.0, sum = 0.0;
        int n = 0;
        for (int trial = 0; trial < 100; ++trial) {
            const double q = std::exp(3.0 * U(g)), M = std::ldexp(1.0, e2) / q;
            double x[64], al[64], xm = 0.0, am = 0.0;
            for (int i = 0; i < 64; ++i) {
                x[i] = 2.0 * M * U(g);
                al[i] = std::exp(-3.0 * std::fabs(U(g)));
                xm = std::max(xm, std::fabs(x[i]));
                am = std::max(am, al[i]);
            }
            const int em = (int)(fix::double_word(xm) >> 52), ea = (int)(fix::double_word(am) >> 52);
            const fix::Scale sc = fix::scale_of(q, fix::turns_of(q), em);
            if (!sc.ok) continue;
            for (int i = 0; i < 64; ++i) {
                int64_t re = 0, im = 0;
                fix::add_term(fix::scaled(x[i], em, 62), sc, fix::words(fix::scaled(al[i], ea, 58)), table.data(), re,
                              im);
                const long double phi = (long double)q * x[i], u = std::ldexp(1.0L, ea - 1022 - 56);
                const double er = (double)(re * u - al[i] * cosl(phi)), ei = (double)(im * u - al[i] * sinl(phi));
                largest = std::max(largest, std::max(std::fabs(er), std::fabs(ei)));
                sum += er + ei;
                n += 2;
            }
        }
        std::printf("term %d %.3e %.3e\n", e2, largest, sum / n);
    }
}

// serial_sums' steps, the lanes one after another
static double window(double t, const double *x, int n, double *mine)
{
    int done = 0;
    for (int tries = 0; done < n; ++tries) {
        if (tries < 4) {
            int64_t s = 0;
            int stop = n;
            for (int l = done; l < n; ++l) {
                const chain::Units u = chain::units_of(t, x[l]);
                s += u.n;
                if (!chain::in_binade(t, s, u)) {
                    stop = l;
                    break;
                }
                mine[l] = chain::advanced(t, s);
            }
            if (stop > done) t = mine[stop - 1];
            done = stop;
            if (done >= n) break;
        }
        t = t + x[done];
        mine[done++] = t;
    }
    return t;
}

static long differences(const std::vector<double> &x)
{
    double t = 0.0, r = 0.0, mine[32];
    long bad = 0;
    for (size_t i = 0; i < x.size(); i += 32) {
        const int n = (int)std::min<size_t>(32, x.size() - i);
        t = window(t, &x[i], n, mine);
        for (int l = 0; l < n; ++l) {
            r = r + x[i + l];
            bad += r == r ? chain::bits(r) != chain::bits(mine[l]) : mine[l] == mine[l];
        }
    }
    return bad;
}

int main()
{
    terms();
    std::mt19937_64 g(2);
    std::normal_distribution<double> N;
    long bad = 0;
    for (int trial = 0; trial < 4000; ++trial) {
        std::vector<double> x(300);
        const int kind = (int)(g() % 5);
        for (auto &v : x) {
            if (kind == 0) v = N(g);
            if (kind == 1) v = std::ldexp((double)((int)(g() % 9) - 4), (int)(g() % 60) - 30);  // many half ways
            if (kind == 2) v = N(g) * std::pow(10.0, (int)(g() % 20) - 10.0);
            if (kind == 3) v = std::ldexp(1.0, (int)(g() % 8) - 54) * (double)(g() % 3) + (g() % 50 == 0 ? 1.0 : 0.0);
            if (kind == 4) v = g() % 3 ? 0.0 : -0x1p-3 * (double)((int)(g() % 3) - 1);  // through zero and powers of two
            if (kind == 2 && g() % 300 == 0) v = g() % 3 ? 5e-324 : INFINITY;
        }
        bad += differences(x);
    }
    std::printf("chain %ld\n", bad);
    return 0;
}
