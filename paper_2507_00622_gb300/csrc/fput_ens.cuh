// fput_ens.cuh -- the FPUT ensemble kernel, shared by k_fput_ens.cu (fixed steps) and
// k_fput_ens_adapt.cu (adaptive DOP 8(5)).
//
// An ensemble orbit carries its state and k <= 6 deviation vectors.  A block
// carries the 32 / L orbits whose lanes fill a warp, L = min(N, 32) lanes each, R =
// N / L adjacent masses per lane, as a pipeline of warps:
//   warp O    step after step of the orbits (adaptive: trial after trial, the
//             error norm and the step control);
//   warps V   two vectors each through the steps that O accepted, one iteration
//             behind O, renormalised.
// Where an ensemble fills the GPU anyway (Cfg::pipelined), warp O works the vectors
// of its orbits itself, in blocks of one warp.
// Lane l of every warp works the same masses, so what O leaves for V (a step's
// stiffnesses around a lane's masses, its size and verdict) lies in the lane's
// own column of double-buffered shared memory; neighbours pass by shuffles
// inside a warp, and one block barrier per iteration joins the warps.  An orbit at
// a health check pauses for one iteration, until its vectors have arrived; a
// finished or frozen orbit takes steps of size 0, which change nothing.
//
// The FP64 pipe bounds these kernels and a warp instruction costs the same
// whatever its active lanes, so every lane carries masses in both phases (a
// thread per component of the state, half of them waiting in turn, took 1.6 times
// the FP64 instructions), and the pipeline spreads the orbits of an ensemble of a
// few hundred over two to four times as many of the GPU's 608 FP64 units as one
// warp per orbit did.  A mass computes both of its bonds: the chain has one bond
// more than masses, so one of them needs a second evaluation in any case.
// 1000 orbits of N = 32, GALI_4, adaptive to t = 50 on GB300: 22.0 ms with a thread per
// component and separate stage sums of q and p, 14.8 ms now (one warp alone).
#pragma once

#include "fput_stages.cuh"
#include "k_dop853.cuh"

namespace chs {
namespace fe {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kVecWarps = (kMaxDev + 1) / 2;  // most V warps of a block

constexpr int kFp64Units = 608;               // of the GPU: one per SM sub-partition

template <int N, class Tab>
struct Cfg {
    static constexpr int D = 2 * N;
    static constexpr int L = fs::ColShape<N>::L, R = fs::ColShape<N>::R;
    static constexpr int OPW = 32 / L;                  // orbits per block
    static constexpr int STIFF = Tab::S * (2 * R + 1);  // a lane's stage stiffnesses: R + 1 bonds, R sums
    // shared bytes and threads of a block with K vectors, pipelined or one warp alone
    static size_t smem(int K, bool pipe)
    {
        return (size_t)((pipe ? 2 : 1) * STIFF + K * 2 * R) * 32 * sizeof(double);
    }
    static int threads(int K, bool pipe) { return pipe ? 32 * (1 + (K + 1) / 2) : 32; }
    // Whether an ensemble of n orbits is pipelined.  ms pipelined (one warp alone in
    // brackets), GALI_4 adaptive to t = 15, by blocks: 100 (N = 32) 1.25 (2.71); 300 (N =
    // 16) 1.65 (3.09); 600 (N = 64) 4.78 (5.47); 1000 (N = 32) 4.60 (4.39), (N = 8) 5.48
    // (4.74); 2000 (N = 64) 14.8 (17.4), (N = 16) 8.69 (9.14).  Between one and two
    // blocks per FP64 unit the lone warps fill the units evenly and win.
    static bool pipelined(int K, int64_t n)
    {
        const int64_t blocks = (n + OPW - 1) / OPW;
        return K > 0 && (blocks <= kFp64Units || blocks > 2 * kFp64Units);
    }
};

// What passes between the warps beside the stiffnesses.
struct Ctl {
    double h[2][32], rh[2][32];           // a step's size and its reciprocal, 0 unless it is to be taken
    int32_t check[2][32];                 // it ends at a health check
    int32_t bad[kVecWarps][32];           // at a health check: a vector is not finite
    int32_t aligned[32];                  // at a health check: SALI < threshold
    int32_t more[2];                      // O has a step or a check to come
};

// Sum over the orbit's L lanes, the same value (bit for bit) in each of them:
// an xor butterfly (a + b and b + a round alike).
template <int L>
__device__ __forceinline__ double lane_sum(double v)
{
#pragma unroll
    for (int off = L / 2; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off, L);
    return v;
}

// Potential of one bond, V(r) = k/2 r^2 + alpha/3 r^3 + beta/4 r^4 (Eq. ham_FPU).
__device__ __forceinline__ double bond_v(const SysPar& sp, const double r)
{
    return r * r * (0.5 * sp.kk + r * (sp.alpha / 3.0 + 0.25 * sp.beta * r));
}

// One lane's part of its orbit: masses R r0 .. R r0 + R - 1.
template <int N, class Tab>
struct Lane {
    using C = Cfg<N, Tab>;
    static constexpr int L = C::L, R = C::R, S = Tab::S;
    int r0;  // lane of the orbit
    bool first, last;
    unsigned mates;  // the orbit's lanes

    __device__ __forceinline__ Lane()
        : r0(threadIdx.x % L), first(r0 == 0), last(r0 == L - 1),
          mates((L == 32 ? kFull : (1u << (L % 32)) - 1u) << (threadIdx.x % 32 - r0))
    {
    }
    // entry e of the lane's column of a stiffness buffer
    __device__ __forceinline__ static double& stiff(double* buf, int s, int k)
    {
        return buf[(s * (2 * R + 1) + k) * 32 + threadIdx.x % 32];
    }
    __device__ __forceinline__ static double& diag(double* buf, int s, int k)
    {
        return buf[(s * (2 * R + 1) + R + 1 + k) * 32 + threadIdx.x % 32];
    }
    // global index of component k of the lane's part (q: half 0, p: half 1)
    __device__ __forceinline__ int64_t comp(int half, int k) const { return half * N + R * r0 + k; }

    // Positions left of the lane's first mass and right of its last one (walls: 0).
    __device__ __forceinline__ void neighbours(const double* w, double& left, double& right) const
    {
        left = __shfl_up_sync(kFull, w[R - 1], 1, L);
        right = __shfl_down_sync(kFull, w[0], 1, L);
        left = first ? 0.0 : left;
        right = last ? 0.0 : right;
    }

    // (nq, np) <- the end of the step of size sh.h from (q, p), the stage
    // stiffnesses into buf; with ERR the lane's part of the error norm's sums in s5
    // and s3.
    template <bool ERR>
    __device__ __forceinline__ void orbit_step(const double* q, const double* p, const dp::StepH sh, const SysPar& sp,
                                               double* buf, double* nq, double* np, const double atol,
                                               const double rtol, double& s5, double& s3) const
    {
        const fs::Coef fc = fs::coef_of(sp, -sh.nh2);
        double G[S][R], hp[R], sq[R], sv[R], err[R][4];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            hp[k] = sh.h * p[k];
            sq[k] = sv[k] = 0.0;
            err[k][0] = err[k][1] = err[k][2] = err[k][3] = 0.0;
        }
        dp::static_for<0, S>([&](auto sc) {
            constexpr int s = decltype(sc)::value;
            double w[R + 2], c[R + 1], f[R + 1];
#pragma unroll
            for (int k = 0; k < R; ++k)
                w[k + 1] = s == 0 ? q[k] : fs::stage_sum<s, Tab, R>(fma(Tab::template Nc<s>, hp[k], q[k]), G, k);
            neighbours(w + 1, w[0], w[R + 1]);
#pragma unroll
            for (int b = 0; b <= R; ++b) {
                const double r = w[b + 1] - w[b];
                c[b] = fs::d2v(fc, r);
                f[b] = fs::dv(fc, r);
                stiff(buf, s, b) = c[b];
            }
#pragma unroll
            for (int k = 0; k < R; ++k) {
                diag(buf, s, k) = -(c[k] + c[k + 1]);
                G[s][k] = f[k + 1] - f[k];
                fs::add_stage<Tab, ERR, s>(G[s][k], sq[k], sv[k], err[k]);
            }
        });
#pragma unroll
        for (int k = 0; k < R; ++k) {
            nq[k] = q[k] + (hp[k] + sq[k]);
            np[k] = fma(sh.rh, sv[k], p[k]);
        }
        if constexpr (ERR) {
            s5 = s3 = 0.0;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                err[k][2] *= sh.rh;
                err[k][3] *= sh.rh;
                fs::mass_error(q[k], p[k], nq[k], np[k], err[k], atol, rtol, s5, s3);
            }
        }
    }

    // H of the orbit, the same in its lanes.
    __device__ __forceinline__ double energy(const SysPar& sp, const double* q, const double* p) const
    {
        double w[R + 2], term = 0.0;
#pragma unroll
        for (int k = 0; k < R; ++k) w[k + 1] = q[k];
        neighbours(w + 1, w[0], w[R + 1]);
#pragma unroll
        for (int k = 0; k < R; ++k) term += fma(0.5 * p[k], p[k], bond_v(sp, w[k + 1] - w[k]));
        if (last) term += bond_v(sp, -w[R]);  // the bond to the right wall
        return lane_sum<L>(term);
    }
};

// The deviation vectors j0 .. j0 + nv - 1 of a warp's orbits, in the lanes' columns of
// shared memory, and what a health check asks of them.
template <int N, class Tab>
struct Vectors {
    using C = Cfg<N, Tab>;
    static constexpr int L = C::L, R = C::R;
    double* sm;  // all K vectors of the block: entry e of lane l at sm[e * 32 + l]
    int j0, nv;

    __device__ __forceinline__ double& u(int j, int k) const { return sm[(j * 2 * R + k) * 32 + threadIdx.x % 32]; }
    __device__ __forceinline__ double& v(int j, int k) const
    {
        return sm[(j * 2 * R + R + k) * 32 + threadIdx.x % 32];
    }
    __device__ __forceinline__ void load(const Lane<N, Tab>& ln, const EnsPtrs& e, const int64_t o, const bool runs) const
    {
        const double* wg = static_cast<const double*>(e.w);
        for (int j = j0; j < j0 + nv; ++j)
#pragma unroll
            for (int k = 0; k < R; ++k) {
                u(j, k) = runs ? wg[(j * 2 * N + ln.comp(0, k)) * e.n + o] : 0.0;
                v(j, k) = runs ? wg[(j * 2 * N + ln.comp(1, k)) * e.n + o] : 0.0;
            }
    }
    __device__ __forceinline__ void store(const Lane<N, Tab>& ln, const EnsPtrs& e, const int64_t o) const
    {
        double* wg = static_cast<double*>(e.w);
        for (int j = j0; j < j0 + nv; ++j)
#pragma unroll
            for (int k = 0; k < R; ++k) {
                wg[(j * 2 * N + ln.comp(0, k)) * e.n + o] = u(j, k);
                wg[(j * 2 * N + ln.comp(1, k)) * e.n + o] = v(j, k);
            }
    }
    // The step of size sh.h (0: the orbit's vectors stay) with the stiffnesses in
    // buf, scaled to unit length with renorm; then, for the orbits at a health
    // check, slot `slot` of the verdicts.
    __device__ __forceinline__ void step(const Lane<N, Tab>& ln, const StepArgs& a, const dp::StepH sh, double* buf,
                                         const bool check, const int K, const int slot, Ctl& ctl) const
    {
        const int lane = threadIdx.x % 32;
#pragma unroll 1
        for (int j = j0; j < j0 + nv; ++j) {
            double x[R], y[R];
#pragma unroll
            for (int k = 0; k < R; ++k) {
                x[k] = u(j, k);
                y[k] = v(j, k);
            }
            fs::column_step<N, Tab>(x, y, sh, ln.first, ln.last,
                                    [&](int s, int k) { return Lane<N, Tab>::stiff(buf, s, k); },
                                    [&](int s, int k) { return Lane<N, Tab>::diag(buf, s, k); });
            double inv = 1.0;
            if (a.renorm) {
                double n2 = 0.0;
#pragma unroll
                for (int k = 0; k < R; ++k) n2 = fma(x[k], x[k], fma(y[k], y[k], n2));
                inv = rsqrt(lane_sum<L>(n2));
            }
            if (sh.h != 0.0) {
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    u(j, k) = x[k] * inv;
                    v(j, k) = y[k] * inv;
                }
            }
        }
        if (!__any_sync(kFull, check)) return;
        bool fin = true;
        for (int j = j0; j < j0 + nv; ++j)
#pragma unroll
            for (int k = 0; k < R; ++k) fin = fin && isfinite(u(j, k)) && isfinite(v(j, k));
        const unsigned nf = __ballot_sync(kFull, !fin);
        if (check) ctl.bad[slot][lane] = (nf & ln.mates) != 0;
        if (j0 == 0 && a.early_exit && K >= 2) {
            double na = 0.0, nb = 0.0, s2 = 0.0, d2 = 0.0;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                na = fma(u(0, k), u(0, k), fma(v(0, k), v(0, k), na));
                nb = fma(u(1, k), u(1, k), fma(v(1, k), v(1, k), nb));
            }
            na = 1.0 / sqrt(lane_sum<L>(na));
            nb = 1.0 / sqrt(lane_sum<L>(nb));
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const double u0 = u(0, k) * na, u1 = u(1, k) * nb, v0 = v(0, k) * na, v1 = v(1, k) * nb;
                s2 += (u0 + u1) * (u0 + u1) + (v0 + v1) * (v0 + v1);
                d2 += (u0 - u1) * (u0 - u1) + (v0 - v1) * (v0 - v1);
            }
            const double sali = sqrt(fmin(lane_sum<L>(s2), lane_sum<L>(d2)));
            if (check) ctl.aligned[lane] = sali < a.sali_threshold;
        }
    }
};

// A V warp of the pipeline: the vectors 2 (warp - 1) and the next one.
template <int N, class Tab>
__device__ __forceinline__ void vector_warp(const StepArgs& a, const EnsPtrs& e, const int K, const int64_t o,
                                            const bool runs, double* smem, Ctl& ctl)
{
    using C = Cfg<N, Tab>;
    const Lane<N, Tab> ln;
    const int lane = threadIdx.x % 32, wv = threadIdx.x / 32 - 1;
    const Vectors<N, Tab> vec{smem + 2 * C::STIFF * 32, 2 * wv, K - 2 * wv < 2 ? K - 2 * wv : 2};
    vec.load(ln, e, o, runs);
    for (int64_t it = 0;; ++it) {
        const int b = (int)(it & 1) ^ 1;  // the buffer of the previous iteration's step
        const double h = it > 0 ? ctl.h[b][lane] : 0.0;
        if (__any_sync(kFull, h != 0.0))
            vec.step(ln, a, dp::StepH{h, 0.0, ctl.rh[b][lane]}, smem + b * C::STIFF * 32, ctl.check[b][lane] != 0, K, wv,
                     ctl);
        __syncthreads();
        if (!ctl.more[it & 1]) break;
    }
    if (runs) vec.store(ln, e, o);
}

// The whole block.  The checks after a step, in this order: escape (sum_i q_i^2 >
// escape_r2, every step); then at health-check steps: non-finite state or vector
// -> NONFINITE, dh_max <- max(dh_max, |H - H0|), |H - h0| > dh_limit ->
// ENERGY_DRIFT, with early_exit SALI(w_1, w_2) < sali_threshold -> EARLY_CHAOTIC,
// the clock budget.  Health checks: fixed steps at absolute steps, adaptive runs at
// accepted-step counts divisible by sample_every.
template <int N, class Tab, bool ADAPT, bool PIPE>
__device__ __forceinline__ void ensemble_block(const StepArgs& a, const AdaptArgs& ad, const SysPar& sp, const int K,
                                               const EnsPtrs& e, const AdaptPtrs& ap, double* smem, Ctl& ctl)
{
    using C = Cfg<N, Tab>;
    constexpr int L = C::L, R = C::R;
    const int lane = threadIdx.x % 32;
    const int64_t o = (int64_t)blockIdx.x * C::OPW + lane / L;
    const bool runs = o < e.n && e.status[o] == CHS_ORBIT_OK;
    if (PIPE && threadIdx.x >= 32) {
        vector_warp<N, Tab>(a, e, K, o, runs, smem, ctl);
        return;
    }
    const Lane<N, Tab> ln;
    const Vectors<N, Tab> vec{smem + C::STIFF * 32, 0, K};  // one warp alone
    if (!PIPE) vec.load(ln, e, o, runs);
    const double inf = __longlong_as_double(0x7ff0000000000000LL);
    double q[R], p[R], nq[R], np[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        q[k] = runs ? e.x[ln.comp(0, k) * e.n + o] : 0.0;
        p[k] = runs ? e.x[ln.comp(1, k) * e.n + o] : 0.0;
    }
    int32_t st = runs ? CHS_ORBIT_OK : CHS_ORBIT_FORBIDDEN;
    const double h0 = runs ? e.h0[o] : 0.0;
    double dhm = runs ? e.dh_max[o] : 0.0;
    const int64_t exec0 = runs ? e.n_exec[o] : 0;
    int64_t todo = a.n_steps;
    if (!ADAPT && runs && e.t_end) {
        const int64_t rem = e.t_end[o] - exec0;
        if (rem < todo) todo = rem > 0 ? rem : 0;
    }
    double tt = 0.0, hnext = 0.0, el = 0.0, em = 0.0;
    int64_t rej = 0;
    if (ADAPT && runs) {
        tt = ap.t[o];
        hnext = ap.h[o];
        el = ap.err_last ? ap.err_last[o] : 0.0;
        em = ap.err_max ? ap.err_max[o] : 0.0;
        rej = ap.n_rej ? ap.n_rej[o] : 0;
    }
    const int64_t count0 = ADAPT ? exec0 : a.step0;  // the step count that health checks go by
    int64_t done = 0;
    int wait = 0;  // 2: at a health check, the vectors are under way; 1: they have arrived
    bool rejected = false;  // the current step has had a rejected trial
    const dp::StepH fixed = dp::step_h(a.dt);
    const long long t_start = clock64();

    // One iteration = one step (trial) of every orbit that is running and not at a
    // health check.  Each rejection shrinks the step by at least 0.9 until it drops
    // below 10 ulp(t), and accepted steps are capped, so every orbit leaves after
    // finitely many iterations.
    for (int64_t it = 0;; ++it) {
        const int b = it & 1;
        const bool at_check = wait > 0 && --wait == 0;
        if (__any_sync(kFull, at_check)) {
            bool fin = true;
#pragma unroll
            for (int k = 0; k < R; ++k) fin = fin && isfinite(q[k]) && isfinite(p[k]);
            const bool bad = (__ballot_sync(kFull, !fin) & ln.mates) != 0;
            const double H = ln.energy(sp, q, p);
            const bool over = (__ballot_sync(kFull, budget_spent(a, t_start)) & ln.mates) != 0;
            if (at_check) {
                bool vec_bad = false;
                for (int j = 0; PIPE ? 2 * j < K : j < (K > 0); ++j) vec_bad = vec_bad || ctl.bad[j][lane];
                if (bad || vec_bad) {
                    st = CHS_ORBIT_NONFINITE;
                } else {
                    const double dH = fabs(H - h0);
                    if (dH > dhm) dhm = dH;
                    if (a.dh_limit > 0.0 && dH > a.dh_limit)
                        st = CHS_ORBIT_ENERGY_DRIFT;
                    else if (a.early_exit && K >= 2 && ctl.aligned[lane])
                        st = CHS_ORBIT_EARLY_CHAOTIC;
                    else if (over)
                        st = CHS_ORBIT_STEP_BUDGET;
                }
            }
        }
        bool active = wait == 0 && st == CHS_ORBIT_OK && done < todo && (!ADAPT || tt < ad.t_final);
        double hh = active ? a.dt : 0.0, tn = tt;
        if (ADAPT && active) {
            const double min_step = 10.0 * (nextafter(tt, inf) - tt);
            if (!rejected) {
                if (ad.h_max > 0.0 && hnext > ad.h_max) hnext = ad.h_max;
                if (hnext < min_step) hnext = min_step;
            }
            if (hnext < min_step) {
                st = CHS_ORBIT_STEP_FAIL;
                active = false;
                hh = 0.0;
            } else {
                tn = tt + hnext;
                if (tn > ad.t_final) tn = ad.t_final;
                hh = tn - tt;
            }
        }
        bool accept = false, check = false;
        if (__any_sync(kFull, active)) {
            const dp::StepH sh = ADAPT ? dp::step_h(hh) : active ? fixed : dp::StepH{0.0, 0.0, 0.0};
            double s5 = 0.0, s3 = 0.0;
            ln.template orbit_step<ADAPT>(q, p, sh, sp, PIPE ? smem + b * C::STIFF * 32 : smem, nq, np, ad.atol, ad.rtol, s5, s3);
            accept = active;
            if constexpr (ADAPT) {
                const double err = dp::err_of<C::D>(lane_sum<L>(s5), lane_sum<L>(s3));
                const double r8 = (active && err > 0.0) ? inv_root8(err) : 0.0;
                accept = active && err < 1.0;
                if (accept) {
                    double fac = (err == 0.0) ? 10.0 : fmin(10.0, 0.9 * r8);
                    if (rejected) fac = fmin(fac, 1.0);
                    hnext = hh * fac;
                    tt = tn;
                    el = err;
                    em = fmax(em, err);
                    rejected = false;
                } else if (active) {
                    double fac = 0.9 * r8;
                    if (!(fac >= 0.2)) fac = 0.2;  // also for a non-finite error
                    hnext = hh * fac;
                    rejected = true;
                    ++rej;
                }
            }
            if (accept) {
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    q[k] = nq[k];
                    p[k] = np[k];
                }
                ++done;
            }
            if (a.escape_r2 > 0.0) {
                double r2 = 0.0;
#pragma unroll
                for (int k = 0; k < R; ++k) r2 = fma(q[k], q[k], r2);
                r2 = lane_sum<L>(r2);
                if (accept && r2 > a.escape_r2) st = CHS_ORBIT_ESCAPED;
            }
            check = accept && st == CHS_ORBIT_OK && a.sample_every > 0 && (count0 + done) % a.sample_every == 0;
            if (check) wait = PIPE ? 2 : 1;
            if (PIPE)
                ctl.rh[b][lane] = sh.rh;
            else if (__any_sync(kFull, accept))
                vec.step(ln, a, accept ? sh : dp::StepH{0.0, 0.0, 0.0}, smem, check, K, 0, ctl);
        }
        const bool more = __any_sync(kFull, active || wait > 0);
        if (PIPE) {
            ctl.h[b][lane] = accept ? hh : 0.0;
            ctl.check[b][lane] = check;
            if (lane == 0) ctl.more[b] = more;
            __syncthreads();
        }
        if (!more) break;
    }
    if (!runs) return;
    if (!PIPE) vec.store(ln, e, o);
#pragma unroll
    for (int k = 0; k < R; ++k) {
        e.x[ln.comp(0, k) * e.n + o] = q[k];
        e.x[ln.comp(1, k) * e.n + o] = p[k];
    }
    if (ln.first) {
        e.dh_max[o] = dhm;
        e.n_exec[o] = exec0 + done;
        e.status[o] = st;
        if constexpr (ADAPT) {
            ap.t[o] = tt;
            ap.h[o] = hnext;
            if (ap.err_last) ap.err_last[o] = el;
            if (ap.err_max) ap.err_max[o] = em;
            if (ap.n_rej) ap.n_rej[o] = rej;
        }
    }
}

}  // namespace fe
}  // namespace chs
