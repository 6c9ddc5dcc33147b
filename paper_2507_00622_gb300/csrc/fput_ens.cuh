// fput_ens.cuh -- shared pieces of the FPUT ensemble kernels (k_fput_ens.cu:
// fixed steps; k_fput_ens_adapt.cu: adaptive DOP 8(5)): an orbit's lanes, its
// step and the checks that follow a completed step.
//
// An ensemble orbit carries its state and k <= 6 deviation vectors.  One warp
// works 32 / L orbits, L = min(N, 32) lanes each, R = N / L adjacent masses per
// lane, and nothing is shared between warps: neighbours pass by shuffles, what
// a lane keeps for later (the stage stiffnesses around its masses, its rows of
// the deviation vectors) lies in its own column of shared memory, and there is
// no barrier.  The FP64 pipe bounds these kernels, a warp instruction costs the
// same whatever its active lanes, so every lane carries masses in both phases; a
// thread per component of the state (2N threads, half of them waiting in turn)
// took 1.6 times the FP64 instructions (1000 orbits of N = 32, GALI_4, adaptive to
// t = 50: 22.0 ms so, 14.8 ms now, the Nystrom form of fput_stages.cuh included).  A mass computes both of its bonds: the
// chain has one bond more than masses, so one of them needs a second evaluation
// in any case.
#pragma once

#include "fput_stages.cuh"

namespace chs {
namespace fe {

constexpr unsigned kFull = 0xffffffffu;

template <int N, class Tab>
struct Cfg {
    static constexpr int D = 2 * N;
    static constexpr int L = fs::ColShape<N>::L, R = fs::ColShape<N>::R;
    static constexpr int OPW = 32 / L;                  // orbits per warp and block
    static constexpr int STIFF = Tab::S * (2 * R + 1);  // a lane's stage stiffnesses: R + 1 bonds, R sums
    // shared bytes of a block (one warp) with K vectors
    static size_t smem(int K) { return (size_t)(STIFF + K * 2 * R) * 32 * sizeof(double); }
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

// One lane's part of an orbit: masses R * lane .. R * lane + R - 1.
template <int N, class Tab>
struct Lane {
    using C = Cfg<N, Tab>;
    static constexpr int L = C::L, R = C::R, S = Tab::S;
    double* sm;  // the lane's column of the block's shared array: entry e at sm[e * 32]
    int r0;      // lane of the orbit
    bool first, last;

    __device__ __forceinline__ explicit Lane(double* smem)
        : sm(smem + threadIdx.x % 32), r0(threadIdx.x % L), first(r0 == 0), last(r0 == L - 1)
    {
    }
    __device__ __forceinline__ double& stiff(int s, int k) const { return sm[(s * (2 * R + 1) + k) * 32]; }
    __device__ __forceinline__ double& diag(int s, int k) const { return sm[(s * (2 * R + 1) + R + 1 + k) * 32]; }
    __device__ __forceinline__ double& u(int j, int k) const { return sm[(C::STIFF + j * 2 * R + k) * 32]; }
    __device__ __forceinline__ double& v(int j, int k) const { return sm[(C::STIFF + j * 2 * R + R + k) * 32]; }
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

    // Phase 1: (nq, np) <- the end of the step of size sh.h from (q, p), the stage
    // stiffnesses into the lane's column; with ERR the lane's part of the error
    // norm's sums in s5 and s3.
    template <bool ERR>
    __device__ __forceinline__ void orbit_step(const double* q, const double* p, const dp::StepH sh, const SysPar& sp,
                                               double* nq, double* np, const double atol, const double rtol,
                                               double& s5, double& s3) const
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
                stiff(s, b) = c[b];
            }
#pragma unroll
            for (int k = 0; k < R; ++k) {
                diag(s, k) = -(c[k] + c[k + 1]);
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

    // Phase 2: the K vectors through the same step, scaled to unit length with
    // renorm; a step of 0 leaves them untouched, and a warp whose orbits all have
    // step 0 (rejected trials, frozen orbits) skips the work.
    __device__ __forceinline__ void vectors_step(const int K, const dp::StepH sh, const int renorm) const
    {
        if (!__any_sync(kFull, sh.h != 0.0)) return;
#pragma unroll 1
        for (int j = 0; j < K; ++j) {
            double a[R], b[R];
#pragma unroll
            for (int k = 0; k < R; ++k) {
                a[k] = u(j, k);
                b[k] = v(j, k);
            }
            fs::column_step<N, Tab>(a, b, sh, first, last, [&](int s, int k) { return stiff(s, k); },
                                    [&](int s, int k) { return diag(s, k); });
            double inv = 1.0;
            if (renorm) {
                double n2 = 0.0;
#pragma unroll
                for (int k = 0; k < R; ++k) n2 = fma(a[k], a[k], fma(b[k], b[k], n2));
                inv = rsqrt(lane_sum<L>(n2));
            }
            if (sh.h != 0.0) {
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    u(j, k) = a[k] * inv;
                    v(j, k) = b[k] * inv;
                }
            }
        }
    }

    // The checks after a step, in this order: escape (sum_i q_i^2 > escape_r2,
    // every step); then at health-check steps: non-finite state or vector ->
    // NONFINITE, dh_max <- max(dh_max, |H - h0|), |H - h0| > dh_limit ->
    // ENERGY_DRIFT, with early_exit SALI(w_1, w_2) < sali_threshold ->
    // EARLY_CHAOTIC.  stepped and check are per orbit (the same in all of its
    // lanes), any_check is warp-uniform.  Every lane of the warp calls this.
    __device__ __forceinline__ int32_t post_step(const StepArgs& a, const SysPar& sp, const int K, const double* q,
                                                 const double* p, const bool stepped, const bool check,
                                                 const bool any_check, const double h0, double& dhm,
                                                 int32_t st) const
    {
        if (a.escape_r2 > 0.0) {
            double r2 = 0.0;
#pragma unroll
            for (int k = 0; k < R; ++k) r2 = fma(q[k], q[k], r2);
            r2 = lane_sum<L>(r2);
            if (stepped && st == CHS_ORBIT_OK && r2 > a.escape_r2) st = CHS_ORBIT_ESCAPED;
        }
        if (!any_check) return st;
        bool fin = true;
#pragma unroll
        for (int k = 0; k < R; ++k) fin = fin && isfinite(q[k]) && isfinite(p[k]);
        for (int j = 0; j < K; ++j)
#pragma unroll
            for (int k = 0; k < R; ++k) fin = fin && isfinite(u(j, k)) && isfinite(v(j, k));
        const double nbad = lane_sum<L>(fin ? 0.0 : 1.0);
        double w[R + 2], term = 0.0;
#pragma unroll
        for (int k = 0; k < R; ++k) w[k + 1] = q[k];
        neighbours(w + 1, w[0], w[R + 1]);
#pragma unroll
        for (int k = 0; k < R; ++k) term += fma(0.5 * p[k], p[k], bond_v(sp, w[k + 1] - w[k]));
        if (last) term += bond_v(sp, -w[R]);  // the bond to the right wall
        const double H = lane_sum<L>(term);
        double sali = __longlong_as_double(0x7ff0000000000000LL);
        if (a.early_exit && K >= 2) {
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
            sali = sqrt(fmin(lane_sum<L>(s2), lane_sum<L>(d2)));
        }
        if (check && stepped && st == CHS_ORBIT_OK) {
            if (nbad > 0.0) {
                st = CHS_ORBIT_NONFINITE;
            } else {
                const double dH = fabs(H - h0);
                if (dH > dhm) dhm = dH;
                if (a.dh_limit > 0.0 && dH > a.dh_limit)
                    st = CHS_ORBIT_ENERGY_DRIFT;
                else if (a.early_exit && K >= 2 && sali < a.sali_threshold)
                    st = CHS_ORBIT_EARLY_CHAOTIC;
            }
        }
        return st;
    }

    // The orbit's state and vectors between global memory ([2N][n] and [K 2N][n])
    // and the lane.
    __device__ __forceinline__ void load(const EnsPtrs& e, const int64_t o, const int K, const bool valid, double* q,
                                         double* p) const
    {
        const double* wg = static_cast<const double*>(e.w);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            q[k] = valid ? e.x[comp(0, k) * e.n + o] : 0.0;
            p[k] = valid ? e.x[comp(1, k) * e.n + o] : 0.0;
            for (int j = 0; j < K; ++j) {
                u(j, k) = valid ? wg[(j * 2 * N + comp(0, k)) * e.n + o] : 0.0;
                v(j, k) = valid ? wg[(j * 2 * N + comp(1, k)) * e.n + o] : 0.0;
            }
        }
    }
    __device__ __forceinline__ void store(const EnsPtrs& e, const int64_t o, const int K, const double* q,
                                          const double* p) const
    {
        double* wg = static_cast<double*>(e.w);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            e.x[comp(0, k) * e.n + o] = q[k];
            e.x[comp(1, k) * e.n + o] = p[k];
            for (int j = 0; j < K; ++j) {
                wg[(j * 2 * N + comp(0, k)) * e.n + o] = u(j, k);
                wg[(j * 2 * N + comp(1, k)) * e.n + o] = v(j, k);
            }
        }
    }
};

}  // namespace fe
}  // namespace chs
