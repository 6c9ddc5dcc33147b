// rk4_common.cuh -- pieces of the classic RK4 step shared by the one-orbit-per-
// thread kernels: the orbit's four stages (with the LD quadrature and the stage
// Hessians recorded) and the exact one-step propagator of the variational
// equations.
#pragma once

#include "chs_internal.cuh"
#include "fastmath.cuh"
#include "systems.cuh"

namespace chs {

// sum_i q_i^2 > escape_r2 (escape_r2 > 0).  The sum is formed only when some |q_i|
// reaches a bound below sqrt(escape_r2 / N), compared by the high words of the
// doubles on the integer pipe: an orbit inside that box has not escaped, and the
// test costs no FP64 instruction there.  bound_hi is StepArgs::escape_hi.
template <int N>
__device__ __forceinline__ bool escaped(const double* q, const int bound_hi, const double escape_r2)
{
    bool far = false;
#pragma unroll
    for (int i = 0; i < N; ++i) far = far || (__double2hiint(q[i]) & 0x7fffffff) >= bound_hi;
    if (!far) return false;
    double r2 = q[0] * q[0];
#pragma unroll
    for (int i = 1; i < N; ++i) r2 = fma(q[i], q[i], r2);
    return r2 > escape_r2;
}

// LD integrand sum_i |f_i|^p in FP64 for a general exponent p (p = 1/2 takes
// the double-float route, ld_acc_sqrt).
template <int D>
__device__ __forceinline__ double ld_integrand_pow(const double* f, double p)
{
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < D; ++i) acc += pow(fabs(f[i]), p);
    return acc;
}

// One term of the LD integrand in FP32: the correctly rounded root (or power) of
// |f|, f a component already rounded to FP32.
__device__ __forceinline__ float ld_term_f32(const float f, const int ld_sqrt, const float p)
{
    return ld_sqrt ? sqrtf(fabsf(f)) : powf(fabsf(f), p);
}

// acc += w sum_i sqrt|f_i| in double-float (p = 1/2; w a power of two).
template <int D>
__device__ __forceinline__ void ld_acc_sqrt(FF& acc, const double* f, const float w)
{
#pragma unroll
    for (int i = 0; i < D; ++i) ff_acc(acc, ff_sqrt(ff_split(fabs(f[i]))), w);
}

// The FP64 LD of one RK4 step: stage st's terms (f the stage's derivative) with
// weight 1 or 2 into fL (p = 1/2) or aL, and the step's sum into L.  The LD grows
// with |t|: a backward run (h < 0) accumulates a positive M_p.
template <int D>
__device__ __forceinline__ void ld_add_stage(const int st, const double* f, const int ld_sqrt, const double ld_p,
                                             FF& fL, double& aL)
{
    const bool mid = st == 1 || st == 2;
    if (ld_sqrt)
        ld_acc_sqrt<D>(fL, f, mid ? 2.0f : 1.0f);
    else
        aL = fma(mid ? 2.0 : 1.0, ld_integrand_pow<D>(f, ld_p), aL);
}
__device__ __forceinline__ void ld_finish(double& L, const double h, const int ld_sqrt, const FF fL, const double aL)
{
    L = fma(fabs(h / 6.0), ld_sqrt ? ff_to_f64(fL) : aL, L);
}

// One RK4 step of the orbit x by the stage derivatives f of the whole state,
// handed out as rec(s, xs, f, H).
template <class Sys, class Rec>
__device__ __forceinline__ void rk4_stages_f(double* x, const double h, const SysPar& sp, Rec&& rec)
{
    constexpr int D = 2 * Sys::N;
    const double hh = 0.5 * h, h6 = h / 6.0;
    double ax[D], xs[D], f[D], Hs[Sys::NH];
    Sys::eval(x, f, Hs, sp);
    rec(0, x, f, Hs);
#pragma unroll
    for (int c = 0; c < D; ++c) {
        ax[c] = f[c];
        xs[c] = fma(hh, f[c], x[c]);
    }
#pragma unroll
    for (int s = 1; s < 3; ++s) {
        Sys::eval(xs, f, Hs, sp);
        rec(s, xs, f, Hs);
#pragma unroll
        for (int c = 0; c < D; ++c) {
            ax[c] = fma(2.0, f[c], ax[c]);
            xs[c] = fma(s == 1 ? hh : h, f[c], x[c]);
        }
    }
    Sys::eval(xs, f, Hs, sp);
    rec(3, xs, f, Hs);
#pragma unroll
    for (int c = 0; c < D; ++c) x[c] = fma(h6, ax[c] + f[c], x[c]);
}

// One classic RK4 step of the orbit x and its LD accumulator L,
//   k1 = f(x), k2 = f(x + h/2 k1), k3 = f(x + h/2 k2), k4 = f(x + h k3),
//   x <- x + h/6 (k1 + 2 k2 + 2 k3 + k4),  L <- L + |h|/6 (g1 + 2 g2 + 2 g3 + g4),
// handing each stage s its positions and Hess V there (packed upper triangle)
// as rec(s, xs, H); a recorder that ignores H leaves its arithmetic unused.
//
// FP64 LD (LD and not LD32), p = 1/2: the weighted sum of the sixteen square
// roots is formed in double-float arithmetic (relative error ~1e-13, off the
// FP64 pipe) and added to L with one FP64 FMA; other exponents use pow.
//
// Without the LD, and for the FP32-frame mode's LD (LD32) at two degrees of freedom,
// the step runs in Nystrom form: with q' = p and p' = F(q),
//   q2 = q + h/2 p,  q3 = q2 + h^2/4 F1,  q4 = q + (h p + h^2/2 F2),
//   q <- q + (h p + h^2/6 (F1 + F2 + F3)),  p <- p + h/6 (F1 + 2 F2 + 2 F3 + F4),
// the same step in exact arithmetic with 12 FP64 instructions per degree of
// freedom beside the forces instead of 14 (the FP64 pipe bounds both; 262,144
// orbits, 300 steps, FP32 frame: quartic k = 6 13.3 -> 12.5 ms, Henon-Heiles k = 2
// with the LD 7.0 -> 6.7 ms; the quartic with the LD ran slower so, 13.9 -> 16.7 ms).
// The LD32 integrand needs the stage momenta in FP32 only: p_s = p + c h F is
// formed in FP32 from p split into two floats, so that it carries the one
// rounding an FP64 value rounded to FP32 would; the stage's terms are summed in
// FP32, the four stage sums in double-float.
template <class Sys, bool LD, bool LD32, class Rec>
__device__ __forceinline__ void rk4_stages(double* x, double& L, const double h, const int ld_sqrt,
                                           const double ld_p, const SysPar& sp, Rec&& rec)
{
    constexpr int N = Sys::N, D = 2 * N;
    constexpr bool L32 = LD && LD32;
    if constexpr (!LD || (LD32 && N == 2)) {
        const double hh = 0.5 * h, h6 = h / 6.0;
        const double h22 = 0.5 * h * h, h24 = 0.25 * h * h, h26 = h * h / 6.0;
        double xs[D], f[D], Hs[Sys::NH], F1[N], F2[N], t[N], hp[N], q2[N];
        FF pf[N], fL{0.0f, 0.0f};
        const float hf = (float)h, hhf = (float)hh, pp = (float)ld_p;
        float g = 0.0f;
        // adds the stage's terms, F at the stage and the momenta p + c F_prev
        auto ld_stage = [&](const float w, const float c, const float* Fprev, float* Fs) {
            if constexpr (L32) {
                g = 0.0f;
#pragma unroll
                for (int i = 0; i < N; ++i)
                    g += ld_term_f32(Fprev ? pf[i].hi + fmaf(c, Fprev[i], pf[i].lo) : pf[i].hi, ld_sqrt, pp);
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    Fs[i] = f32_from_f64(f[N + i]);
                    g += ld_term_f32(Fs[i], ld_sqrt, pp);
                }
                ff_acc(fL, FF{g, 0.0f}, w);
            }
        };
        float Ff[4][N];
#pragma unroll
        for (int c = 0; c < D; ++c) xs[c] = x[c];
        if constexpr (L32) {
#pragma unroll
            for (int i = 0; i < N; ++i) pf[i] = ff_split_signed(x[N + i]);
        }
        Sys::eval(xs, f, Hs, sp);
        rec(0, xs, Hs);
        ld_stage(1.0f, 0.0f, nullptr, Ff[0]);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            F1[i] = f[N + i];
            hp[i] = h * x[N + i];
            xs[i] = q2[i] = fma(hh, x[N + i], x[i]);
        }
        Sys::eval(xs, f, Hs, sp);
        rec(1, xs, Hs);
        ld_stage(2.0f, hhf, Ff[0], Ff[1]);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            F2[i] = f[N + i];
            xs[i] = fma(h24, F1[i], q2[i]);
        }
        Sys::eval(xs, f, Hs, sp);
        rec(2, xs, Hs);
        ld_stage(2.0f, hhf, Ff[1], Ff[2]);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            t[i] = F2[i] + f[N + i];
            F1[i] += t[i];
            xs[i] = x[i] + fma(h22, F2[i], hp[i]);
        }
        Sys::eval(xs, f, Hs, sp);
        rec(3, xs, Hs);
        ld_stage(1.0f, hf, Ff[2], Ff[3]);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            x[i] += fma(h26, F1[i], hp[i]);
            x[N + i] = fma(h6, (F1[i] + t[i]) + f[N + i], x[N + i]);
        }
        // the LD grows with |t|: a backward run (h < 0) accumulates a positive M_p
        if constexpr (L32) L = fma(fabs(h6), ff_to_f64(fL), L);
    } else {
        double aL = 0.0;
        FF fL{0.0f, 0.0f};
        rk4_stages_f<Sys>(x, h, sp, [&](int st, const double* xs, const double* f, const double* Hs) {
            rec(st, xs, Hs);
            if constexpr (L32) {
                float g = 0.0f;
#pragma unroll
                for (int c = 0; c < D; ++c) g += ld_term_f32(f32_from_f64(f[c]), ld_sqrt, (float)ld_p);
                ff_acc(fL, FF{g, 0.0f}, (st == 1 || st == 2) ? 2.0f : 1.0f);
            } else if constexpr (LD) {
                ld_add_stage<D>(st, f, ld_sqrt, ld_p, fL, aL);
            }
        });
        if constexpr (L32)
            L = fma(fabs(h / 6.0), ff_to_f64(fL), L);
        else if constexpr (LD)
            ld_finish(L, h, ld_sqrt, fL, aL);
    }
}

// The RK4 step recording Hess V at the four stage states in H[s].
template <class Sys, bool LD, bool LD32 = false>
__device__ __forceinline__ void rk4_state_capture(double* x, double& L, const double h,
                                                  const int ld_sqrt, const double ld_p,
                                                  const SysPar& sp, double (*H)[Sys::NH])
{
    rk4_stages<Sys, LD, LD32>(x, L, h, ld_sqrt, ld_p, sp, [&](int s, const double*, const double* Hs) {
#pragma unroll
        for (int i = 0; i < Sys::NH; ++i) H[s][i] = Hs[i];
    });
}

// The RK4 step recording the stage positions q rounded to FP32 (integer pipe)
// in qf[s]; the FP64 Hessians are not formed.
template <class Sys, bool LD, bool LD32 = false>
__device__ __forceinline__ void rk4_state_positions(double* x, double& L, const double h,
                                                    const int ld_sqrt, const double ld_p,
                                                    const SysPar& sp, float (*qf)[Sys::N])
{
    rk4_stages<Sys, LD, LD32>(x, L, h, ld_sqrt, ld_p, sp, [&](int s, const double* xs, const double*) {
#pragma unroll
        for (int i = 0; i < Sys::N; ++i) qf[s][i] = f32_from_f64(xs[i]);
    });
}

// Exact one-step propagator of RK4 on the linear variational equation
// w' = J_s w, J_s = [[0, I], [-H_s, 0]] (H_s = Hess V at stage s):
//   Phi = I + h/6 (J1 + 2J2 + 2J3 + J4) + h^2/6 (J2J1 + J3J2 + J4J3)
//           + h^3/12 (J3J2J1 + J4J3J2) + h^4/24 J4J3J2J1
//       = [[A, B], [C, D]] with
//   A = I - h^2/6 (H1+H2+H3) + h^4/24 H3H1,   B = h I - h^3/12 (H2+H3),
//   C = -h/6 (H1+2H2+2H3+H4) + h^3/12 (H3H1 + H4H2),
//   D = I - h^2/6 (H2+H3+H4) + h^4/24 H4H2.
// Applying Phi equals RK4 on the joint system in exact arithmetic.
template <int N, typename T>
struct PhiBlocks {
    T A[N][N], B[N][N], C[N][N], D[N][N];
};

template <int N, int NH, typename T>
__device__ __forceinline__ void phi_build(const T (*Hs)[NH], const double h, PhiBlocks<N, T>& P)
{
    const T hv = (T)h, c1 = (T)(h / 6.0), c2 = (T)(h * h / 6.0), c3 = (T)(h * h * h / 12.0),
            c4 = (T)(h * h * h * h / 24.0);
#pragma unroll
    for (int i = 0; i < N; ++i) {
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const T s1 = Hs[0][hidx<N>(i, j)], s2 = Hs[1][hidx<N>(i, j)];
            const T s3 = Hs[2][hidx<N>(i, j)], s4 = Hs[3][hidx<N>(i, j)];
            T p31 = Hs[2][hidx<N>(i, 0)] * Hs[0][hidx<N>(0, j)];
            T p42 = Hs[3][hidx<N>(i, 0)] * Hs[1][hidx<N>(0, j)];
#pragma unroll
            for (int m = 1; m < N; ++m) {
                p31 = fma(Hs[2][hidx<N>(i, m)], Hs[0][hidx<N>(m, j)], p31);
                p42 = fma(Hs[3][hidx<N>(i, m)], Hs[1][hidx<N>(m, j)], p42);
            }
            const T s23 = s2 + s3;
            const T id = (i == j) ? (T)1 : (T)0;
            P.A[i][j] = fma(c4, p31, fma(-c2, s1 + s23, id));
            P.B[i][j] = (i == j) ? fma(-c3, s23, hv) : -c3 * s23;
            P.C[i][j] = fma(c3, p31 + p42, -c1 * (fma((T)2, s23, s1) + s4));
            P.D[i][j] = fma(c4, p42, fma(-c2, s23 + s4, id));
        }
    }
}

// Henon-Heiles: Hess V = I + 2 M(q) with M(q) = [[q2, q1], [q1, -q2]] (from
// Eq. ham_eqs_HH), M linear in q, and M(a) M(b) = [[p, r], [-r, p]] with
// p = a1 b1 + a2 b2, r = a2 b1 - a1 b2.  The blocks of Phi from the four stage
// positions q_s, with c1 = h/6, c2 = h^2/6, c3 = h^3/12, c4 = h^4/24:
//   A = (1 - 3 c2 + c4) I + 2 M(c4 (q1 + q3) - c2 (q1 + q2 + q3)) + 4 c4 M(q3) M(q1)
//   B = (h - 2 c3) I - 2 c3 M(q2 + q3)
//   C = (2 c3 - 6 c1) I + 2 M(c3 (q1 + q2 + q3 + q4) - c1 (q1 + 2 q2 + 2 q3 + q4))
//       + 4 c3 (M(q3) M(q1) + M(q4) M(q2))
//   D = (1 - 3 c2 + c4) I + 2 M(c4 (q2 + q4) - c2 (q2 + q3 + q4)) + 4 c4 M(q4) M(q2)
// (the general blocks above with H_s = I + 2 M(q_s)); no Hessian is formed.
// 49 instructions: the M parts are 2 M of
//   A: (c4 - c2)(q1 + q3) - c2 q2,   D: (c4 - c2)(q2 + q4) - c2 q3,
//   C: (c3 - c1)(q1 + q2 + q3 + q4) - c1 (q2 + q3),
// and each block's diagonal part is formed once for its two entries.
template <typename T>
__device__ __forceinline__ void phi_build_hh(const T (*q)[2], const double h, PhiBlocks<2, T>& P)
{
    const double c1 = h / 6.0, c2 = h * h / 6.0, c3 = h * h * h / 12.0, c4 = h * h * h * h / 24.0;
    const T aAD = (T)(1.0 - 3.0 * c2 + c4), aB = (T)(h - 2.0 * c3), aC = (T)(2.0 * c3 - 6.0 * c1);
    const T n1 = (T)(-2.0 * c1), n2 = (T)(-2.0 * c2), n3 = (T)(-2.0 * c3), cc = (T)(2.0 * c4 - 2.0 * c2),
            cs = (T)(2.0 * c3 - 2.0 * c1), k4 = (T)(4.0 * c4), k3 = (T)(4.0 * c3);
    T mA[2], s23[2], mC[2], mD[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const T s13 = q[0][i] + q[2][i], s24 = q[1][i] + q[3][i];
        s23[i] = q[1][i] + q[2][i];
        mA[i] = fma(cc, s13, n2 * q[1][i]);
        mD[i] = fma(cc, s24, n2 * q[2][i]);
        mC[i] = fma(cs, s13 + s24, n1 * s23[i]);
    }
    const T p31 = fma(q[2][0], q[0][0], q[2][1] * q[0][1]), r31 = fma(q[2][1], q[0][0], -q[2][0] * q[0][1]);
    const T p42 = fma(q[3][0], q[1][0], q[3][1] * q[1][1]), r42 = fma(q[3][1], q[1][0], -q[3][0] * q[1][1]);
    const T dA = fma(k4, p31, aAD), dD = fma(k4, p42, aAD), dC = fma(k3, p31 + p42, aC), rc = r31 + r42;
    P.A[0][0] = dA + mA[1];
    P.A[1][1] = dA - mA[1];
    P.A[0][1] = fma(k4, r31, mA[0]);
    P.A[1][0] = fma(-k4, r31, mA[0]);
    P.B[0][0] = fma(n3, s23[1], aB);
    P.B[1][1] = fma(-n3, s23[1], aB);
    P.B[0][1] = P.B[1][0] = n3 * s23[0];
    P.C[0][0] = dC + mC[1];
    P.C[1][1] = dC - mC[1];
    P.C[0][1] = fma(k3, rc, mC[0]);
    P.C[1][0] = fma(-k3, rc, mC[0]);
    P.D[0][0] = dD + mD[1];
    P.D[1][1] = dD - mD[1];
    P.D[0][1] = fma(k4, r42, mD[0]);
    P.D[1][0] = fma(-k4, r42, mD[0]);
}

// w <- Phi w for one vector w = (u, v).
template <int N, typename T>
__device__ __forceinline__ void phi_apply(const PhiBlocks<N, T>& P, T* w)
{
    T nw[2 * N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        T u = P.A[i][0] * w[0], v = P.C[i][0] * w[0];
#pragma unroll
        for (int m = 1; m < N; ++m) {
            u = fma(P.A[i][m], w[m], u);
            v = fma(P.C[i][m], w[m], v);
        }
#pragma unroll
        for (int m = 0; m < N; ++m) {
            u = fma(P.B[i][m], w[N + m], u);
            v = fma(P.D[i][m], w[N + m], v);
        }
        nw[i] = u;
        nw[N + i] = v;
    }
#pragma unroll
    for (int c = 0; c < 2 * N; ++c) w[c] = nw[c];
}

// w scaled to unit length (relative error of the length ~2^-43).
template <int D>
__device__ __forceinline__ void unit_vector(double* w)
{
    double n2 = w[0] * w[0];
#pragma unroll
    for (int c = 1; c < D; ++c) n2 = fma(w[c], w[c], n2);
    const double inv = rsqrt_ff(n2);
#pragma unroll
    for (int c = 0; c < D; ++c) w[c] *= inv;
}

// SALI of two vectors (each normalised first): min(|u + v|, |u - v|).
template <int D>
__device__ __forceinline__ double sali_of(const double* a, const double* b)
{
    double na = a[0] * a[0], nb = b[0] * b[0];
#pragma unroll
    for (int c = 1; c < D; ++c) {
        na = fma(a[c], a[c], na);
        nb = fma(b[c], b[c], nb);
    }
    const double ia = rsqrt_nr(na), ib = rsqrt_nr(nb);
    double sp = 0.0, sm = 0.0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const double u = a[c] * ia, v = b[c] * ib;
        sp = fma(u + v, u + v, sp);
        sm = fma(u - v, u - v, sm);
    }
    return sqrt(fmin(sp, sm));
}

// One step of the modified Gram-Schmidt: w loses its component along the unit
// vector q.
template <int D>
__device__ __forceinline__ void remove_component(const double* q, double* w)
{
    double r = 0.0;
#pragma unroll
    for (int c = 0; c < D; ++c) r = fma(q[c], w[c], r);
#pragma unroll
    for (int c = 0; c < D; ++c) w[c] = fma(-r, q[c], w[c]);
}

// w scaled to unit length, S += ln |w|.
template <int D>
__device__ __forceinline__ void normalise_log(double* w, double& S)
{
    double n2 = 0.0;
#pragma unroll
    for (int c = 0; c < D; ++c) n2 = fma(w[c], w[c], n2);
    S += 0.5 * log(n2);
    const double inv = rsqrt_nr(n2);
#pragma unroll
    for (int c = 0; c < D; ++c) w[c] *= inv;
}

}  // namespace chs
