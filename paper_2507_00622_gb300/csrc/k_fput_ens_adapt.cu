// k_fput_ens_adapt.cu -- adaptive DOP 8(5) (Sec. Functionalities) on FPUT
// ensembles with k <= 6 deviation vectors: the FPU timing workload of
// Sec. Examples (GALI_4 of 1e3 orbits per chain length) runs with it.
//
// Every orbit has its own time and step size.  A trial advances the orbit
// through the twelve stages (phase 1 of fput_stages.cuh); the error norm over
// its 2N components is an orbit-wide sum that every lane of the orbit holds
// bit for bit, so all of them take the same accept / reject decision.  The
// deviation vectors advance (phase 2, renormalised with renorm) only for accepted
// trials, and the checks of fput_ens.cuh, which holds the kernel, follow each
// accepted step.
// Controller: safety 0.9, growth at most 10 (not above 1 right after a
// rejection), shrink at least 0.2, STEP_FAIL once h < 10 ulp(t).
#include "fput_ens.cuh"
#include "k_dop853.cuh"

namespace chs {
namespace {

template <int N, bool PIPE>
__global__ void __launch_bounds__(PIPE ? 32 * (1 + fe::kVecWarps) : 32)
k_fput_ens_adapt(const StepArgs a, const AdaptArgs ad, const SysPar sp, const int K, const EnsPtrs e,
                 const AdaptPtrs ap)
{
    extern __shared__ double smem[];
    __shared__ fe::Ctl ctl;
    fe::ensemble_block<N, fs::TabDop853, true, PIPE>(a, ad, sp, K, e, ap, smem, ctl);
}

template <int N>
cudaError_t adapt_n(const SysPar& sp, int k, const StepArgs& a, const AdaptArgs& ad, const EnsPtrs& e,
                    const AdaptPtrs& ap, cudaStream_t st)
{
    using C = fe::Cfg<N, fs::TabDop853>;
    const bool pipe = C::pipelined(k, e.n);
    auto kern = pipe ? k_fput_ens_adapt<N, true> : k_fput_ens_adapt<N, false>;
    kern<<<blocks_for(e.n, C::OPW), C::threads(k, pipe), C::smem(k, pipe), st>>>(a, ad, sp, k, e, ap);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_fput_ens_adapt(const SysPar& sp, int k, const StepArgs& a, const AdaptArgs& ad,
                                  const EnsPtrs& e, const AdaptPtrs& ap, cudaStream_t st)
{
    if (e.n == 0 || a.n_steps == 0) return cudaSuccess;
    switch (sp.n_dof) {
    case 4: return adapt_n<4>(sp, k, a, ad, e, ap, st);
    case 8: return adapt_n<8>(sp, k, a, ad, e, ap, st);
    case 16: return adapt_n<16>(sp, k, a, ad, e, ap, st);
    case 32: return adapt_n<32>(sp, k, a, ad, e, ap, st);
    case 64: return adapt_n<64>(sp, k, a, ad, e, ap, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace chs
