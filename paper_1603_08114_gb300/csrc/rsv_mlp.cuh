// rsv_mlp.cuh -- launchers of the learned-mass kernels.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "rsv_device.cuh"

namespace rsv {

int mlp_nparam();
int mlp_sites_per_block();
int feat_grid(int64_t T);
// Gradient (and loss) of the minibatch of Adam step `step`.
cudaError_t launch_mlp_step(const float* feat, const float* target, int64_t T, float* params,
                            float* grad_out, float* partials, unsigned* counter, uint64_t seed,
                            uint64_t step, int batch, float* loss_out, const float* log_scale,
                            cudaStream_t st);
// Adam steps step0 .. step0 + n_steps - 1: one cooperative launch where the
// minibatch's blocks can all be resident and the stream is not being captured,
// else a launch per step.  counter is zero between launches, barrier any value;
// a device-side wait beyond wait_limit cycles sets ST_TIMEOUT in *status.
cudaError_t launch_mlp_train(const float* feat, const float* target, int64_t T, float* params,
                             float* adam_m, float* adam_v, float* partials, unsigned* counter,
                             unsigned* barrier, uint64_t seed, int64_t step0, int n_steps, float lr,
                             int batch, float* loss_out, const float* log_scale, bool capturing,
                             int num_sms, long long wait_limit, int* status, int64_t* launches,
                             cudaStream_t st);
// NaN while *status holds ST_TIMEOUT.
cudaError_t launch_mlp_mass(const float* feat, int64_t T, const float* params, const double* y,
                            const double* hbar, ThetaD th, const float* log_scale,
                            const int* status, float* minv, float* m_out, cudaStream_t st);
cudaError_t launch_welford(const float* x, int64_t n, int64_t T, int64_t count, double* mean,
                           double* m2, cudaStream_t st);
// partials: target_blocks() doubles (a block's sum each), counter: zero between launches.
size_t target_blocks();
cudaError_t launch_welford_target(const double* mean, const double* m2, int64_t T, int64_t count,
                                  double* hbar, float* target, float* log_scale, double* partials,
                                  unsigned* counter, cudaStream_t st);
cudaError_t launch_features(const double* y, const double* lnrv, const double* hbar, int64_t T,
                            ThetaD th, float* F, float* stats, double* partials, unsigned* counter,
                            cudaStream_t st);

}  // namespace rsv
