// k_adapt_pipe.cuh -- launcher of the pipelined adaptive kernel for small
// ensembles (k_adapt_pipe.cu).
#pragma once

#include "k_dop853.cuh"

namespace chs {

// Largest ensemble the pipeline takes (see adapt_pipe_applies).
constexpr int64_t kAdaptPipeOrbits = 14592;

bool adapt_pipe_applies(const SysPar& sp, int k, bool ld, int64_t n);
cudaError_t launch_adaptive_pipe(int k, const StepArgs& a, const AdaptArgs& ad, const EnsPtrs& e, const AdaptPtrs& ap,
                                 cudaStream_t st);

}  // namespace chs
