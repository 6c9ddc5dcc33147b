// k_fput_ens_adapt.cu -- adaptive DOP 8(5) (Sec. Functionalities) on FPUT
// ensembles with k <= 6 deviation vectors: the FPU timing workload of
// Sec. Examples (GALI_4 of 1e3 orbits per chain length) runs with it.
//
// Every orbit has its own time and step size.  A trial advances the orbit
// through the twelve stages (phase 1 of fput_stages.cuh); the error norm over
// its 2N components is an orbit-wide sum that every lane of the orbit holds
// bit for bit, so all of them take the same accept / reject decision (lanes of
// fput_ens.cuh).  The
// deviation vectors advance (phase 2, renormalised with renorm) only for
// accepted trials, and the checks of fput_ens.cuh follow each accepted step.
// Controller: safety 0.9, growth at most 10 (not above 1 right after a
// rejection), shrink at least 0.2, STEP_FAIL once h < 10 ulp(t).
#include "fput_ens.cuh"
#include "k_dop853.cuh"

namespace chs {
namespace {

template <int N>
__global__ void __launch_bounds__(32)
k_fput_ens_adapt(const StepArgs a, const AdaptArgs ad, const SysPar sp, const int K, const EnsPtrs e,
                 const AdaptPtrs ap)
{
    using Tab = fs::TabDop853;
    using C = fe::Cfg<N, Tab>;
    constexpr int R = C::R;
    extern __shared__ double smem[];
    const fe::Lane<N, Tab> ln(smem);
    const int64_t o = (int64_t)blockIdx.x * C::OPW + threadIdx.x / C::L;
    const bool valid = o < e.n;
    const double inf = __longlong_as_double(0x7ff0000000000000LL);

    int32_t st = valid ? e.status[o] : CHS_ORBIT_FORBIDDEN;
    const bool runs = st == CHS_ORBIT_OK;
    double q[R], p[R], nq[R], np[R];
    ln.load(e, o, K, valid, q, p);
    const double h0 = runs ? e.h0[o] : 0.0;
    double dhm = runs ? e.dh_max[o] : 0.0;
    const int64_t exec0 = runs ? e.n_exec[o] : 0;
    double tt = runs ? ap.t[o] : 0.0, hnext = runs ? ap.h[o] : 0.0;
    double el = (runs && ap.err_last) ? ap.err_last[o] : 0.0;
    double em = (runs && ap.err_max) ? ap.err_max[o] : 0.0;
    int64_t rej = (runs && ap.n_rej) ? ap.n_rej[o] : 0;
    int64_t done = 0;
    bool rejected = false;  // the current step has had a rejected trial
    const long long t_start = clock64();

    // One iteration = one trial of every orbit that is still running.  Each
    // rejection shrinks the step by at least 0.9 until it drops below
    // 10 ulp(t), and accepted steps are capped at n_steps, so every orbit
    // leaves after finitely many iterations.
    for (;;) {
        bool active = st == CHS_ORBIT_OK && done < a.n_steps && tt < ad.t_final;
        double hh = 0.0, tn = tt;
        if (active) {
            const double min_step = 10.0 * (nextafter(tt, inf) - tt);
            if (!rejected) {
                if (ad.h_max > 0.0 && hnext > ad.h_max) hnext = ad.h_max;
                if (hnext < min_step) hnext = min_step;
            }
            if (hnext < min_step) {
                st = CHS_ORBIT_STEP_FAIL;
                active = false;
            } else {
                tn = tt + hnext;
                if (tn > ad.t_final) tn = ad.t_final;
                hh = tn - tt;
            }
        }
        if (!__any_sync(fe::kFull, active)) break;

        const dp::StepH sh = dp::step_h(hh);
        double s5, s3;
        ln.template orbit_step<true>(q, p, sh, sp, nq, np, ad.atol, ad.rtol, s5, s3);
        const double err = dp::err_of<C::D>(fe::lane_sum<C::L>(s5), fe::lane_sum<C::L>(s3));
        const double r8 = (active && err > 0.0) ? inv_root8(err) : 0.0;
        const bool accept = active && err < 1.0;
        ln.vectors_step(K, accept ? sh : dp::StepH{0.0, 0.0, 0.0}, a.renorm);
        if (active) {
            if (accept) {
                double fac = (err == 0.0) ? 10.0 : fmin(10.0, 0.9 * r8);
                if (rejected) fac = fmin(fac, 1.0);
                hnext = hh * fac;
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    q[k] = nq[k];
                    p[k] = np[k];
                }
                tt = tn;
                el = err;
                em = fmax(em, err);
                ++done;
                rejected = false;
            } else {
                double fac = 0.9 * r8;
                if (!(fac >= 0.2)) fac = 0.2;  // also for a non-finite error
                hnext = hh * fac;
                rejected = true;
                ++rej;
            }
        }
        const bool check = accept && a.sample_every > 0 && (exec0 + done) % a.sample_every == 0;
        const bool any_check = __any_sync(fe::kFull, check);
        st = ln.post_step(a, sp, K, q, p, accept, check, any_check, h0, dhm, st);
        if (any_check && a.clock_budget > 0) {  // warp-uniform: the warp's orbits stop together
            const bool over = __any_sync(fe::kFull, budget_spent(a, t_start)) != 0;
            if (over && check && st == CHS_ORBIT_OK) st = CHS_ORBIT_STEP_BUDGET;
        }
    }
    if (runs) {
        ln.store(e, o, K, q, p);
        if (ln.first) {
            e.dh_max[o] = dhm;
            e.n_exec[o] = exec0 + done;
            e.status[o] = st;
            ap.t[o] = tt;
            ap.h[o] = hnext;
            if (ap.err_last) ap.err_last[o] = el;
            if (ap.err_max) ap.err_max[o] = em;
            if (ap.n_rej) ap.n_rej[o] = rej;
        }
    }
}

template <int N>
cudaError_t adapt_n(const SysPar& sp, int k, const StepArgs& a, const AdaptArgs& ad, const EnsPtrs& e,
                    const AdaptPtrs& ap, cudaStream_t st)
{
    using C = fe::Cfg<N, fs::TabDop853>;
    k_fput_ens_adapt<N><<<blocks_for(e.n, C::OPW), 32, C::smem(k), st>>>(a, ad, sp, k, e, ap);
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
