// Host check of the integer-ALU FP64 arithmetic at its rare branches
// (soft_fp64_edges.h) against the host's IEEE operations.  Prints cases and
// mismatches of each operation; exit status 1 on a mismatch.
#include "../paper_2012_06478_gb300/csrc/soft_fp64.cuh"

#include <cmath>
#include <cstdio>

#include "soft_fp64_edges.h"

using namespace rms::sfp;

int main()
{
    long tested[3] = {}, bad[3] = {};
    for (const EdgeCase &c : edges::cases(200000, 3)) {
        const double got = c.op == 0 ? mul_normal(c.a, c.b) : c.op == 1 ? div_normal(c.a, c.b) : sqrt_normal(c.a);
        const double want = c.op == 0 ? c.a * c.b : c.op == 1 ? c.a / c.b : std::sqrt(c.a);
        ++tested[c.op];
        bad[c.op] += bits_of(got) != bits_of(want);
    }
    for (int k = 0; k < 3; ++k) std::printf("%ld %ld\n", tested[k], bad[k]);
    return bad[0] || bad[1] || bad[2] ? 1 : 0;
}
