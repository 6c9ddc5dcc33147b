// fput_stages.cuh -- building blocks of the FPUT kernels that run explicit
// Runge-Kutta stages on the chain (k_fput_dp.cu: Lyapunov spectra with DOP853;
// fput_chain.cuh: ensembles with k deviation vectors, RK4 or DOP853).
//
// A step runs in two phases:
//   phase 1  the orbit through its stages; every stage leaves h^2 V''(D_b) of the
//            N + 1 bonds and minus the sum of its two bonds for every mass;
//   phase 2  the deviation vectors (columns), one at a time per warp segment:
//            L = min(N, 32) lanes split the column's N (q, p) row pairs, keep
//            the column's stage values in registers and exchange the
//            tridiagonal neighbours q_{i-1}, q_{i+1} by warp shuffles.  No
//            barrier and no stage storage in memory.
// Both run the tableau in Nystrom form (dop853.cuh): with q' = p, p' = F(q),
// one stage sum per mass instead of one for q and one for p.  Per mass and
// step of a column that is 59 + 17 FP64 instructions of sums and 36 of Hessian
// products with DOP853, against 140 + 48 with the sums of q and p kept apart
// (Lyapunov spectra of 2047 chains of N = 16, 40 steps, QR every 10: 18.1 ms so,
// 11.9 ms now).
// Bonds: D_b = q_b - q_{b-1}, b = 0..N, with walls q_{-1} = q_N = 0.
#pragma once

#include "dop853.cuh"

namespace chs {
namespace fs {

// Butcher tableaus as compile-time coefficients: weights B and the Nystrom
// coefficients Na = A A, Nc = A 1, Nb = b A, with the error weights of the pair.
struct TabRk4 {  // classic RK4
    static constexpr int S = 4;
    template <int s>
    static constexpr double B = (s == 0 || s == 3) ? 1.0 / 6.0 : 1.0 / 3.0;
    template <int s, int k>
    static constexpr double Na = (s == 2 && k == 0) ? 0.25 : (s == 3 && k == 1) ? 0.5 : 0.0;
    template <int s>
    static constexpr double Nc = s == 0 ? 0.0 : s == 3 ? 1.0 : 0.5;
    template <int s>
    static constexpr double Nb = s < 3 ? 1.0 / 6.0 : 0.0;
};

struct TabDop853 {  // the DOP853 pair (dop853.cuh), with its error weights
    static constexpr int S = 12;
    template <int s>
    static constexpr double B = dp::kB[s];
    template <int s, int k>
    static constexpr double Na = dp::kNa<s, k>;
    template <int s>
    static constexpr double Nc = dp::kNc<s>;
    template <int s>
    static constexpr double Nb = dp::kNb<s>;
    template <int s>
    static constexpr double E5 = dp::kE5[s];
    template <int s>
    static constexpr double E3 = dp::kB[s] - dp::kB3[s];
    template <int s>
    static constexpr double N5 = dp::kN5<s>;
    template <int s>
    static constexpr double N3 = dp::kN3<s>;
};

// Force and stiffness of a bond scaled by h^2: V'(r) = r (k + r (alpha + beta r)),
// V''(r) = k + r (2 alpha + 3 beta r).
struct Coef {
    double k, alpha, beta, a2, b3;
};

__device__ __forceinline__ Coef coef_of(const SysPar& sp, const double h2)
{
    const double al = h2 * sp.alpha, be = h2 * sp.beta;
    return Coef{h2 * sp.kk, al, be, 2.0 * al, 3.0 * be};
}

__device__ __forceinline__ double dv(const Coef& fc, double r)
{
    return r * fma(r, fma(fc.beta, r, fc.alpha), fc.k);
}

__device__ __forceinline__ double d2v(const Coef& fc, double r)
{
    return fma(r, fma(fc.b3, r, fc.a2), fc.k);
}

// acc + sum_{j < s} Na_sj G[j][k], the stage sum of mass k.
template <int s, class Tab, int R>
__device__ __forceinline__ double stage_sum(double acc, const double (*G)[R], const int k)
{
    dp::static_for<0, s>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        constexpr double c = Tab::template Na<s, j>;
        if constexpr (c != 0.0) acc = fma(c, G[j][k], acc);
    });
    return acc;
}

// The sums a mass accumulates over the stages (h^2-scaled stage values g):
// sq -> q, sv -> p and, with ERR, the error sums of q and p.
template <class Tab, bool ERR, int s>
__device__ __forceinline__ void add_stage(const double g, double& sq, double& sv, double* err)
{
    constexpr double nb = Tab::template Nb<s>, b = Tab::template B<s>;
    if constexpr (nb != 0.0) sq = fma(nb, g, sq);
    if constexpr (b != 0.0) sv = fma(b, g, sv);
    if constexpr (ERR) {
        constexpr double n5 = Tab::template N5<s>, n3 = Tab::template N3<s>;
        constexpr double c5 = Tab::template E5<s>, c3 = Tab::template E3<s>;
        if constexpr (n5 != 0.0) err[0] = fma(n5, g, err[0]);
        if constexpr (n3 != 0.0) err[1] = fma(n3, g, err[1]);
        if constexpr (c5 != 0.0) err[2] = fma(c5, g, err[2]);
        if constexpr (c3 != 0.0) err[3] = fma(c3, g, err[3]);
    }
}

// Phase 1 with one thread per mass (threads l < N of the orbit; the others only
// meet the barriers, one per stage, or warp syncs where WARP says that the block
// is one warp).  xb: [2][N] stage positions; cs: [S][N + 1] bond stiffnesses
// h^2 V''; dg: [S][N], minus the sum of a mass's two bonds.  On return (nq, np)
// is the end point of the step of size sh.h from (q, p); with ERR, err holds
// the error sums times h: err5_q, err3_q, err5_p, err3_p.
template <int N, class Tab, bool ERR, bool WARP>
__device__ __forceinline__ void mass_stages(const double q, const double p, const dp::StepH sh, const int l,
                                            double* xb, double* cs, double* dg, const SysPar& sp, double& nq,
                                            double& np, double* err, const bool act)
{
    const Coef fc = coef_of(sp, -sh.nh2);
    const double hp = sh.h * p;
    double G[Tab::S][1], sq = 0.0, sv = 0.0;
    if constexpr (ERR) err[0] = err[1] = err[2] = err[3] = 0.0;
    dp::static_for<0, Tab::S>([&](auto sc) {
        constexpr int s = decltype(sc)::value;
        double* xs = xb + (s & 1) * N;
        double q0 = q;
        if (act) {
            if constexpr (s > 0) q0 = stage_sum<s, Tab, 1>(fma(Tab::template Nc<s>, hp, q), G, 0);
            xs[l] = q0;
        }
        if constexpr (WARP)
            __syncwarp();
        else
            __syncthreads();
        if (act) {
            const double rl = q0 - (l > 0 ? xs[l - 1] : 0.0), rr = (l < N - 1 ? xs[l + 1] : 0.0) - q0;
            const double cl = d2v(fc, rl), cr = d2v(fc, rr);
            cs[s * (N + 1) + l] = cl;
            if (l == N - 1) cs[s * (N + 1) + N] = cr;
            dg[s * N + l] = -(cl + cr);
            const double g = dv(fc, rr) - dv(fc, rl);
            G[s][0] = g;
            add_stage<Tab, ERR, s>(g, sq, sv, err);
        }
    });
    nq = q + (hp + sq);
    np = fma(sh.rh, sv, p);
    if constexpr (ERR) {
        err[2] *= sh.rh;
        err[3] *= sh.rh;
    }
}

// Adds a mass's part of the error norm (dp::err_norm) to s5 and s3.
__device__ __forceinline__ void mass_error(const double q, const double p, const double nq, const double np,
                                           const double* err, const double atol, const double rtol, double& s5,
                                           double& s3)
{
    const double rq = dp::err_scale(q, nq, atol, rtol), rp = dp::err_scale(p, np, atol, rtol);
    const double q5 = err[0] * rq, q3 = err[1] * rq, p5 = err[2] * rp, p3 = err[3] * rp;
    s5 = fma(q5, q5, fma(p5, p5, s5));
    s3 = fma(q3, q3, fma(p3, p3, s3));
}

// Sum over the orbit's D threads, the same value (bit for bit) in each of
// them: an xor butterfly inside a warp (a + b and b + a round alike), then the
// warp partials in a fixed order.  Every thread of the block must call it.
template <int D>
__device__ __forceinline__ double orbit_sum(double v, double* red, const int l)
{
    constexpr int LW = D < 32 ? D : 32;
#pragma unroll
    for (int off = LW / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off, LW);
    if constexpr (D > 32) {
        if ((l & 31) == 0) red[l >> 5] = v;
        __syncthreads();
        double s = red[0];
#pragma unroll
        for (int i = 1; i < D / 32; ++i) s += red[i];
        __syncthreads();
        return s;
    } else {
        return v;
    }
}

// Lanes per column and columns per warp of phase 2.
template <int N>
struct ColShape {
    static constexpr int L = N < 32 ? N : 32;  // lanes per column
    static constexpr int R = N / L;            // adjacent row pairs per lane
    static constexpr int CPW = 32 / L;         // columns per warp at a time
};

// One column segment through the stages of u' = v, v' = -H_s u: the lane's rows
// (u[k], v[k]), k < R, with stiff(s, k) the h^2-scaled stiffness of the bond left
// of row k (k = R: right of the last row) and diag(s, k) minus the sum of the
// row's two bonds.  first / last: the lane holds the chain's first / last row.
template <int N, class Tab, class Stiff, class Diag>
__device__ __forceinline__ void column_step(double* u, double* v, const dp::StepH sh, const bool first,
                                            const bool last, Stiff stiff, Diag diag)
{
    constexpr int L = ColShape<N>::L, R = ColShape<N>::R;
    double G[Tab::S][R], hv[R], sq[R], sv[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        hv[k] = sh.h * v[k];
        sq[k] = sv[k] = 0.0;
    }
    dp::static_for<0, Tab::S>([&](auto sc) {
        constexpr int s = decltype(sc)::value;
        double w[R];
#pragma unroll
        for (int k = 0; k < R; ++k)
            w[k] = s == 0 ? u[k] : stage_sum<s, Tab, R>(fma(Tab::template Nc<s>, hv[k], u[k]), G, k);
        double left = __shfl_up_sync(0xffffffffu, w[R - 1], 1, L);
        double right = __shfl_down_sync(0xffffffffu, w[0], 1, L);
        left = first ? 0.0 : left;
        right = last ? 0.0 : right;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const double wl = k > 0 ? w[k > 0 ? k - 1 : 0] : left, wr = k < R - 1 ? w[k < R - 1 ? k + 1 : 0] : right;
            const double g = fma(stiff(s, k + 1), wr, fma(stiff(s, k), wl, diag(s, k) * w[k]));
            G[s][k] = g;
            add_stage<Tab, false, s>(g, sq[k], sv[k], nullptr);
        }
    });
#pragma unroll
    for (int k = 0; k < R; ++k) {
        u[k] += hv[k] + sq[k];
        v[k] = fma(sh.rh, sv[k], v[k]);
    }
}

// Phase 2 of the Lyapunov kernels: the kc columns of every orbit of the block (G
// orbits, each orbit's slab at smem + g * PER, column c at + c * WS, stiffnesses
// at + CS, their diagonals at + DG) advance by the step step_of(g, slab); a step
// of 0 leaves the columns untouched, and with SKIP a warp whose segments all
// have step 0 skips the work (callers whose steps are never 0 leave SKIP off: the
// vote changes the register allocation of the stage loop).  Every lane of
// every warp must call this: the segments of a warp loop together (a segment
// past the last column computes on column 0 of orbit 0 with step 0), so the
// shuffles always run on full warps.
template <int N, class Tab, int G, int PER, int WS, int CS, int DG, bool SKIP, class StepOf>
__device__ __forceinline__ void columns(double* smem, const int kc, StepOf step_of)
{
    constexpr int L = ColShape<N>::L, R = ColShape<N>::R, CPW = ColShape<N>::CPW;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int nwarps = blockDim.x / 32;
    const int seg = lane / L, r0 = lane % L;
    const int total = G * kc;
    for (int base = warp * CPW; base < total; base += nwarps * CPW) {
        const int task = base + seg;
        const bool real = task < total;
        const int og = real ? task / kc : 0, col = real ? task % kc : 0;
        double* slab = smem + og * PER;
        const dp::StepH sh = real ? step_of(og, slab) : dp::StepH{0.0, 0.0, 0.0};
        if constexpr (SKIP) {
            if (!__any_sync(0xffffffffu, sh.h != 0.0)) continue;
        }
        double* Wc = slab + col * WS + R * r0;
        const double* c_s = slab + CS + R * r0;
        const double* d_s = slab + DG + R * r0;
        double u[R], v[R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            u[k] = Wc[k];
            v[k] = Wc[N + k];
        }
        column_step<N, Tab>(u, v, sh, r0 == 0, r0 == L - 1, [&](int s, int k) { return c_s[s * (N + 1) + k]; },
                            [&](int s, int k) { return d_s[s * N + k]; });
        if (sh.h != 0.0) {
#pragma unroll
            for (int k = 0; k < R; ++k) {
                Wc[k] = u[k];
                Wc[N + k] = v[k];
            }
        }
    }
}

}  // namespace fs
}  // namespace chs
