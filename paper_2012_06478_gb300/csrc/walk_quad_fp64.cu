// walk_quad_fp64.cu -- the plain form with four lanes to a walker (no FMA
// contraction, as walk_fp64.cu).
#include "rms_internal.h"
#include "walk_quad.cuh"

namespace rms {

cudaError_t launch_walk_quad(int n_shapes, cudaStream_t stream, const Geometry &g, const Tables<double> &t,
                             const WalkerState<double> &st, const RunCtl &ctl, int64_t k_begin, int64_t k_end,
                             int32_t rec)
{
    const unsigned grid = (unsigned)((ctl.n_walkers + kQuadWalkers - 1) / kQuadWalkers);
#define RMS_QUAD_AS(NS, RELAX, SANE) \
    walk_quad_kernel<NS, RELAX, SANE><<<grid, kWalkBlock, 0, stream>>>(g, t, st, ctl, k_begin, k_end, rec)
#define RMS_QUAD(NS)                       \
    do {                                   \
        if (t.any_relax && ctl.sane)       \
            RMS_QUAD_AS(NS, 1, true);      \
        else if (t.any_relax)              \
            RMS_QUAD_AS(NS, 1, false);     \
        else if (ctl.sane)                 \
            RMS_QUAD_AS(NS, 0, true);      \
        else                               \
            RMS_QUAD_AS(NS, 0, false);     \
    } while (0)
    if (n_shapes <= 1)
        RMS_QUAD(1);
    else if (n_shapes <= 2)
        RMS_QUAD(2);
    else if (n_shapes <= 4)
        RMS_QUAD(4);
    else
        RMS_QUAD(8);
#undef RMS_QUAD
#undef RMS_QUAD_AS
    return cudaGetLastError();
}

}  // namespace rms
