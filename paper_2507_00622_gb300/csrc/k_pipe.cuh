// k_pipe.cuh -- launcher of the pipelined small-ensemble kernel (k_pipe.cu).
#pragma once

#include "chs_internal.cuh"

namespace chs {

// Largest ensemble the pipeline takes (see pipe_applies).
constexpr int64_t kPipeOrbits = 14592;

// Whether an RK4 run with FP64 vectors takes the pipelined form.
bool pipe_applies(const SysPar& sp, int k, const StepArgs& a, int64_t n);
cudaError_t launch_integrate_pipe(const SysPar& sp, int k, bool ld, const StepArgs& a, const EnsPtrs& e,
                                  const OrbitList* ol, cudaStream_t st);

// The same for the Lyapunov spectrum by QR (RK4).
constexpr int64_t kLyapPipeOrbits = 14592, kLyapDenseFrom = 4864, kLyapDenseOrbits = 18432;
bool lyap_pipe_applies(const SysPar& sp, const StepArgs& a, int64_t n, const int32_t* ic_status, const int32_t* status);
cudaError_t launch_lyap_pipe(const SysPar& sp, const StepArgs& a, int64_t n, const double* ics,
                             const int32_t* ic_status, double* lambda, int32_t* status, cudaStream_t st);

}  // namespace chs
