// k_dp_pipe.cuh -- launcher of the pipelined fixed-step DOP853 kernel for small
// ensembles (k_dp_pipe.cu).
#pragma once

#include "chs_internal.cuh"

namespace chs {

// Warps of a block: the orbit's, one per vector and the LD's.
constexpr int dp_pipe_warps(int k, bool ld)
{
    return 1 + k + (ld ? 1 : 0);
}
// Blocks per SM: two where six warps leave registers for no more (168 a thread).
constexpr int dp_pipe_blocks(int k, bool ld)
{
    return (ld && k > 2) ? 2 : 3;
}
// Largest ensemble the pipeline takes: one wave on 152 SMs (see dp_pipe_applies).
constexpr int64_t dp_pipe_orbits(int k, bool ld)
{
    return 152 * 32 * dp_pipe_blocks(k, ld);
}

bool dp_pipe_applies(const SysPar& sp, int k, bool ld, const StepArgs& a, int64_t n);
cudaError_t launch_dp_pipe(const SysPar& sp, int k, bool ld, const StepArgs& a, const EnsPtrs& e, const OrbitList* ol,
                           cudaStream_t st);

}  // namespace chs
