// rms_internal.h -- declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include "rms_device.cuh"

namespace rms {

template <typename Real, int IM, bool MT>
cudaError_t launch_walk(int n_shapes, bool hash, dim3 grid, cudaStream_t stream, const Geometry &g,
                        const Tables<Real> &t, const WalkerState<Real> &st, const RunCtl &ctl,
                        int64_t k_begin, int64_t k_end, int32_t rec);

#define RMS_EXTERN_LAUNCH_WALK(REAL, IM, MT)                                                               \
    extern template cudaError_t launch_walk<REAL, IM, MT>(int, bool, dim3, cudaStream_t, const Geometry &, \
                                                          const Tables<REAL> &, const WalkerState<REAL> &, \
                                                          const RunCtl &, int64_t, int64_t, int32_t);
RMS_EXTERN_LAUNCH_WALK(double, kInteractEC, false)
RMS_EXTERN_LAUNCH_WALK(double, kInteractRS, false)
RMS_EXTERN_LAUNCH_WALK(double, kInteractERL, false)
RMS_EXTERN_LAUNCH_WALK(float, kInteractEC, false)
RMS_EXTERN_LAUNCH_WALK(float, kInteractRS, false)
RMS_EXTERN_LAUNCH_WALK(float, kInteractERL, false)
RMS_EXTERN_LAUNCH_WALK(double, kInteractEC, true)
RMS_EXTERN_LAUNCH_WALK(double, kInteractRS, true)
RMS_EXTERN_LAUNCH_WALK(double, kInteractERL, true)
RMS_EXTERN_LAUNCH_WALK(float, kInteractEC, true)
RMS_EXTERN_LAUNCH_WALK(float, kInteractRS, true)
RMS_EXTERN_LAUNCH_WALK(float, kInteractERL, true)
#undef RMS_EXTERN_LAUNCH_WALK

// The plain form's elastic collision with four lanes to a walker (walk_quad.cuh):
// the moments' partials are per 32 walkers, four to a block of the others.
cudaError_t launch_walk_quad(int n_shapes, cudaStream_t stream, const Geometry &g, const Tables<double> &t,
                             const WalkerState<double> &st, const RunCtl &ctl, int64_t k_begin, int64_t k_end,
                             int32_t rec);

template <typename Real>
cudaError_t launch_walk_batched(int ns_bucket, int32_t n_tasks, cudaStream_t stream, const ReqDesc<Real> *reqs,
                                const BlockTask *tasks);
extern template cudaError_t launch_walk_batched<double>(int, int32_t, cudaStream_t, const ReqDesc<double> *,
                                                        const BlockTask *);
extern template cudaError_t launch_walk_batched<float>(int, int32_t, cudaStream_t, const ReqDesc<float> *,
                                                       const BlockTask *);

template <typename Real>
int batched_blocks_per_sm(int ns_bucket);
extern template int batched_blocks_per_sm<double>(int);
extern template int batched_blocks_per_sm<float>(int);

int walk_block_size();

// The read-out (rms_readout.cu): phase component k of walker w at
// phase[w sw + k sk] (one of the strides is 1); the compensations of the FP32
// form likewise; amplitudes q[shape][b], or null: from b and b_s.  part:
// [n_chunks][n_combo + 1][2] sums, the last column the sum of alpha.
template <typename Real>
struct ReadoutPlan {
    const Real *phase, *phase_c, *A, *A_c;
    const double *q, *b, *b_s, *dirs;
    int64_t sw, sk, W, per;
    double *part;
    int32_t S, n_dirs, n_b, n_combo, n_chunks, groups, cpb, nsub, threads, pitch;
};
template <typename Real>
ReadoutPlan<Real> readout_plan(int64_t W, int32_t S, int32_t n_dirs, int32_t n_b, int64_t max_chunks);
template <typename Real>
cudaError_t launch_readout(const ReadoutPlan<Real> &p, cudaStream_t stream);
cudaError_t launch_chunk_sums(const double *part, int32_t n_chunks, int32_t n_combo, double *out, cudaStream_t stream);
cudaError_t launch_chunk_sums_normalised(const double *part, int32_t n_chunks, int32_t n_combo, double *S_re,
                                         double *S_im, double *alpha_sum, cudaStream_t stream);

// Message returned by rms_last_error() on the calling thread.
void set_last_error(const char *msg);

}  // namespace rms
