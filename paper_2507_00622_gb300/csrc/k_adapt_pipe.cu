// k_adapt_pipe.cu -- adaptive DOP 8(5) of Henon-Heiles ensembles too small to fill
// the GPU: the trial steps of 16 orbits spread over the warps of one block.
//
// With one orbit per thread a trial of an orbit with two vectors is a stream of
// ~800 FP64 instructions on one sub-partition, while most of the GPU's 608 FP64
// units have no warp.  Here a block of 1 + k warps carries 16 orbits, two lanes
// per orbit (lane = degree of freedom i: q_i, p_i and their stage sums):
//   warp O    trial after trial of the orbits: stages, error norm, step control;
//   warp V_j  vector j through the stages of the trials that O accepted, one
//             iteration behind O.
// A trial's stage matrices (the row of -h^2 Hess V of the lane's degree of
// freedom), its step and its verdict pass through double-buffered shared memory,
// one block barrier per iteration.  An orbit at a health check pauses for one
// iteration, until its vectors have arrived.  Same method, step control and
// checks as k_integrate_adaptive (k_dop853_adapt.cu); the sums over the two
// degrees of freedom are formed in another order.
//
// SALI of a 64 x 64 grid at tolerance 1e-8 to t = 60 (GB300): 1.81 ms, 5.19 ms with
// one thread per orbit.
#include "fput_stages.cuh"
#include "k_adapt_pipe.cuh"

namespace chs {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kGroup = 16;  // orbits per block
using Tab = fs::TabDop853;

__device__ __forceinline__ double other(const double v) { return __shfl_xor_sync(kFull, v, 1); }
__device__ __forceinline__ double pair_sum(const double v) { return v + other(v); }

template <int K>
struct ApSmem {
    double diag[2][12][32], off[2][12][32];  // a trial's rows of -h^2 Hess V
    double h[2][32], rh[2][32];              // its step, 0 unless accepted
    double w[K][2][32];                      // at a health check: the vectors (u, v)
    int32_t check[2][32];
    int32_t more[2];
};

template <int K>
__global__ void __launch_bounds__(32 * (1 + K))
k_adaptive_pipe(const StepArgs a, const AdaptArgs ad, const EnsPtrs e, const AdaptPtrs ap)
{
    __shared__ ApSmem<K> sm;
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31, i = lane & 1;
    const int64_t n = e.n, o = (int64_t)blockIdx.x * kGroup + lane / 2;
    const bool mine = o < n && e.status[o] == CHS_ORBIT_OK;
    double* wg = static_cast<double*>(e.w);

    if (warp > 0) {
        // a vector: (u, v) of degree of freedom i
        const int j = warp - 1;
        double u = mine ? wg[(int64_t)(4 * j + i) * n + o] : 0.0, v = mine ? wg[(int64_t)(4 * j + 2 + i) * n + o] : 0.0;
        for (int64_t it = 0;; ++it) {
            const int b = (it & 1) ^ 1;  // the buffer of the previous iteration's trial
            const double h = it > 0 ? sm.h[b][lane] : 0.0;
            if (__any_sync(kFull, h != 0.0)) {
                const double rh = sm.rh[b][lane], hv = h * v;
                double G[12][1], sq = 0.0, sv = 0.0;
                dp::static_for<0, 12>([&](auto sc) {
                    constexpr int s = decltype(sc)::value;
                    const double us = s == 0 ? u : fs::stage_sum<s, Tab, 1>(fma(Tab::Nc<s>, hv, u), G, 0);
                    const double g = fma(sm.diag[b][s][lane], us, sm.off[b][s][lane] * other(us));
                    G[s][0] = g;
                    fs::add_stage<Tab, false, s>(g, sq, sv, nullptr);
                });
                double nu = u + (hv + sq), nv = fma(rh, sv, v), inv = 1.0;
                if (a.renorm) inv = rsqrt_ff(pair_sum(fma(nu, nu, nv * nv)));
                if (h != 0.0) {
                    u = nu * inv;
                    v = nv * inv;
                    if (sm.check[b][lane]) {
                        sm.w[j][0][lane] = u;
                        sm.w[j][1][lane] = v;
                    }
                }
            }
            __syncthreads();
            if (!sm.more[it & 1]) break;
        }
        if (mine) {
            wg[(int64_t)(4 * j + i) * n + o] = u;
            wg[(int64_t)(4 * j + 2 + i) * n + o] = v;
        }
        return;
    }

    // the orbit: (q, p) of degree of freedom i; everything else is the same in both lanes
    double q = mine ? e.x[i * n + o] : 0.0, p = mine ? e.x[(2 + i) * n + o] : 0.0;
    const double h0 = mine ? e.h0[o] : 0.0;
    double dhm = mine ? e.dh_max[o] : 0.0;
    const int64_t exec0 = mine ? e.n_exec[o] : 0;
    double tt = mine ? ap.t[o] : 0.0, hnext = mine ? ap.h[o] : 0.0;
    double el = (mine && ap.err_last) ? ap.err_last[o] : 0.0;
    double em = (mine && ap.err_max) ? ap.err_max[o] : 0.0;
    int64_t rej = (mine && ap.n_rej) ? ap.n_rej[o] : 0;
    const double inf = __longlong_as_double(0x7ff0000000000000LL);
    int32_t st = mine ? CHS_ORBIT_OK : CHS_ORBIT_FORBIDDEN;
    int64_t done = 0;
    int wait = 0;  // 2: at a health check, the vectors are under way; 1: they have arrived
    bool rejected = false;
    const long long t_start = clock64();

    // One iteration = one trial of every orbit that is running and not at a
    // health check; it ends like the loop of k_integrate_adaptive.
    for (int64_t it = 0;; ++it) {
        const int b = it & 1;
        if (wait > 0 && --wait == 0) {
            // the health check of the step accepted two iterations ago
            bool fin = isfinite(q) && isfinite(p);
#pragma unroll
            for (int j = 0; j < K; ++j) fin = fin && isfinite(sm.w[j][0][lane]) && isfinite(sm.w[j][1][lane]);
            const unsigned pair = 3u << (lane & ~1);  // the orbit's two lanes, which agree on `wait`
            const unsigned bad = __ballot_sync(pair, !fin);
            const double qo = __shfl_xor_sync(pair, q, 1), po = __shfl_xor_sync(pair, p, 1);
            const double x[4] = {i ? qo : q, i ? q : qo, i ? po : p, i ? p : po};
            if ((bad >> (lane & ~1)) & 3u) {
                st = CHS_ORBIT_NONFINITE;
            } else {
                const double dH = fabs(SysHenonHeiles::energy(x, SysPar{}) - h0);
                dhm = fmax(dhm, dH);
                bool aligned = false;
                if constexpr (K >= 2) {
                    if (a.early_exit) {
                        double y[2][4];
#pragma unroll
                        for (int j = 0; j < 2; ++j)
#pragma unroll
                            for (int c = 0; c < 4; ++c) y[j][c] = sm.w[j][c >> 1][(lane & ~1) + (c & 1)];
                        aligned = dp::sali2<4>(y[0], y[1]) < a.sali_threshold;
                    }
                }
                if (a.dh_limit > 0.0 && dH > a.dh_limit)
                    st = CHS_ORBIT_ENERGY_DRIFT;
                else if (aligned)
                    st = CHS_ORBIT_EARLY_CHAOTIC;
                else if (budget_spent(a, t_start))
                    st = CHS_ORBIT_STEP_BUDGET;
            }
            // the two lanes read different SM clock values: the orbit stops in both
            if (__shfl_xor_sync(pair, st, 1) == CHS_ORBIT_STEP_BUDGET && st == CHS_ORBIT_OK) st = CHS_ORBIT_STEP_BUDGET;
        }
        __syncwarp();
        bool active = wait == 0 && st == CHS_ORBIT_OK && done < a.n_steps && tt < ad.t_final;
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
        bool accept = false, check = false;
        if (__any_sync(kFull, active)) {
            const dp::StepH sh = dp::step_h(hh);
            const double hp = sh.h * p;
            double G[12][1], sq = 0.0, sv = 0.0, es[4] = {};
            dp::static_for<0, 12>([&](auto sc) {
                constexpr int s = decltype(sc)::value;
                const double qs = s == 0 ? q : fs::stage_sum<s, Tab, 1>(fma(Tab::Nc<s>, hp, q), G, 0);
                const double r = other(qs);  // the other degree of freedom
                // F_0 = -q - 2 q r, F_1 = -q + q^2 - r^2; Hess rows (1 + 2 y, 2 x) and (1 - 2 y, 2 x)
                const double A = fma(i ? qs : -2.0 * r, qs, i ? -(r * r) : 0.0);
                const double g = sh.nh2 * (qs - A);
                const double n2 = 2.0 * sh.nh2;
                sm.diag[b][s][lane] = fma(n2, i ? -qs : r, sh.nh2);
                sm.off[b][s][lane] = n2 * (i ? r : qs);
                G[s][0] = g;
                fs::add_stage<Tab, true, s>(g, sq, sv, es);
            });
            const double nq = q + (hp + sq), np = fma(sh.rh, sv, p);
            es[2] *= sh.rh;
            es[3] *= sh.rh;
            double s5 = 0.0, s3 = 0.0;
            fs::mass_error(q, p, nq, np, es, ad.atol, ad.rtol, s5, s3);
            const double err = dp::err_of<4>(pair_sum(s5), pair_sum(s3));
            accept = active && err < 1.0;
            bool far = false;
            if (active) {
                const double r8 = err > 0.0 ? inv_root8(err) : 0.0;
                if (accept) {
                    double fac = (err == 0.0) ? 10.0 : fmin(10.0, 0.9 * r8);
                    if (rejected) fac = fmin(fac, 1.0);
                    hnext = hh * fac;
                    q = nq;
                    p = np;
                    tt = tn;
                    el = err;
                    em = fmax(em, err);
                    ++done;
                    rejected = false;
                    far = (__double2hiint(q) & 0x7fffffff) >= a.escape_hi;
                } else {
                    double fac = 0.9 * r8;
                    if (!(fac >= 0.2)) fac = 0.2;  // also for a non-finite error
                    hnext = hh * fac;
                    rejected = true;
                    ++rej;
                }
            }
            if (__any_sync(kFull, far)) {  // sum_i q_i^2 > escape_r2, where the prefilter says it may be
                const double qo = other(q);
                const double x0 = i ? qo : q, x1 = i ? q : qo;
                if (accept && a.escape_r2 > 0.0 && fma(x1, x1, x0 * x0) > a.escape_r2) st = CHS_ORBIT_ESCAPED;
            }
            check = accept && st == CHS_ORBIT_OK && a.sample_every > 0 && (exec0 + done) % a.sample_every == 0;
            if (check) wait = 2;
            sm.rh[b][lane] = sh.rh;
        }
        sm.h[b][lane] = accept ? hh : 0.0;
        sm.check[b][lane] = check;
        const bool more = __any_sync(kFull, active || wait > 0);
        if (lane == 0) sm.more[b] = more;
        __syncthreads();
        if (!more) break;
    }
    if (!mine) return;
    e.x[i * n + o] = q;
    e.x[(2 + i) * n + o] = p;
    if (i == 0) {
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

}  // namespace

// Whether an adaptive run takes the pipelined form: Henon-Heiles without the LD,
// up to kAdaptPipeOrbits orbits.  The pipeline executes about 1.15 times the FP64
// instructions of the one-thread form, so it pays while FP64 units idle there.  ms to
// t = 30 (one thread per orbit in brackets), k = 2 and k = 4: 4864 orbits 0.90 (2.75)
// and 1.25 (3.65); 9728 1.35 (2.77) and 2.90 (3.68); 14,592 2.36 (2.74) and 3.00
// (3.66); 19,456 2.83 (2.99) and 4.33 (4.04).
bool adapt_pipe_applies(const SysPar& sp, int k, bool ld, int64_t n)
{
    return sp.model == CHS_HENON_HEILES && !ld && k >= 1 && k <= 4 && n <= kAdaptPipeOrbits;
}

cudaError_t launch_adaptive_pipe(int k, const StepArgs& a, const AdaptArgs& ad, const EnsPtrs& e, const AdaptPtrs& ap,
                                 cudaStream_t st)
{
    const unsigned g = blocks_for(e.n, kGroup);
    switch (k) {
    case 1: k_adaptive_pipe<1><<<g, 64, 0, st>>>(a, ad, e, ap); break;
    case 2: k_adaptive_pipe<2><<<g, 96, 0, st>>>(a, ad, e, ap); break;
    case 3: k_adaptive_pipe<3><<<g, 128, 0, st>>>(a, ad, e, ap); break;
    case 4: k_adaptive_pipe<4><<<g, 160, 0, st>>>(a, ad, e, ap); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace chs
