// dop853.cuh -- device building blocks of the DOP853 kernels (k_dop853.cu,
// k_dop853_adapt.cu): the tableau, one orbit step and one deviation-vector step,
// the error norm of the adaptive pair, and the per-step checks.
//
// Design.  A step runs in two phases.  Phase 1 takes the orbit (and the LD
// integrand) through the twelve stages and records each stage's Hessian;
// phase 2 takes each deviation vector through the twelve stages of the linear
// variational equation w' = J_s w with those Hessians.  The vectors never act
// on the orbit, so this is DOP853 on the joint system (x, w_1..w_k, M_p), and an
// adaptive trial that is rejected costs only phase 1.  Both phases run the
// pair in Nystrom form (below), which needs one stage sum per degree of freedom
// instead of two.  The stage Hessians live in a per-thread column of shared
// memory: on GB300 a warp's FP64 FMA occupies its sub-partition's FP64 unit for
// 64 cycles while a 64-bit shared-memory access costs about 2 cycles of the SM's
// shared-memory bandwidth, so re-reading them for every vector is cheap next to
// the arithmetic.  The LD integrand is evaluated only at the eight stages with
// b_s != 0 (the LD never feeds back into a stage).  Every coefficient is a
// compile-time constant: the zero entries generate no instructions.
#pragma once

#include <math.h>

#include <type_traits>

#include "k_dop853.cuh"
#include "rk4_common.cuh"

namespace chs {
namespace dp {

constexpr int kBlock = 32;  // threads per block (one warp: the shared slab sets occupancy)

// The DOP853 pair of Dormand and Prince as published in Hairer, Norsett and
// Wanner, Solving Ordinary Differential Equations I (2nd ed., Springer 1993),
// Sec. II.10.  Stages are numbered from 0.  kA: the strictly lower-triangular
// Runge-Kutta matrix (nodes c_s = sum_j a_sj); kB: the 8th-order weights;
// kE5: the 5th-order error weights b - bhat; kB3: the 3rd-order weights (on
// stages 0, 8 and 11), whose error weights are b - b3.
constexpr double kA[12][12] = {
    {0},
    {5.26001519587677318785587544488e-2},
    {1.97250569845378994544595329183e-2, 5.91751709536136983633785987549e-2},
    {2.95875854768068491816892993775e-2, 0.0, 8.87627564304205475450678981324e-2},
    {2.41365134159266685502369798665e-1, 0.0, -8.84549479328286085344864962717e-1,
     9.24834003261792003115737966543e-1},
    {3.7037037037037037037037037037e-2, 0.0, 0.0, 1.70828608729473871279604482173e-1,
     1.25467687566822425016691814123e-1},
    {3.7109375e-2, 0.0, 0.0, 1.70252211019544039314978060272e-1,
     6.02165389804559606850219397283e-2, -1.7578125e-2},
    {3.70920001185047927108779319836e-2, 0.0, 0.0, 1.70383925712239993810214054705e-1,
     1.07262030446373284651809199168e-1, -1.53194377486244017527936158236e-2,
     8.27378916381402288758473766002e-3},
    {6.24110958716075717114429577812e-1, 0.0, 0.0, -3.36089262944694129406857109825e0,
     -8.68219346841726006818189891453e-1, 2.75920996994467083049415600797e1,
     2.01540675504778934086186788979e1, -4.34898841810699588477366255144e1},
    {4.77662536438264365890433908527e-1, 0.0, 0.0, -2.48811461997166764192642586468e0,
     -5.90290826836842996371446475743e-1, 2.12300514481811942347288949897e1,
     1.52792336328824235832596922938e1, -3.32882109689848629194453265587e1,
     -2.03312017085086261358222928593e-2},
    {-9.3714243008598732571704021658e-1, 0.0, 0.0, 5.18637242884406370830023853209e0,
     1.09143734899672957818500254654e0, -8.14978701074692612513997267357e0,
     -1.85200656599969598641566180701e1, 2.27394870993505042818970056734e1,
     2.49360555267965238987089396762e0, -3.0467644718982195003823669022e0},
    {2.27331014751653820792359768449e0, 0.0, 0.0, -1.05344954667372501984066689879e1,
     -2.00087205822486249909675718444e0, -1.79589318631187989172765950534e1,
     2.79488845294199600508499808837e1, -2.85899827713502369474065508674e0,
     -8.87285693353062954433549289258e0, 1.23605671757943030647266201528e1,
     6.43392746015763530355970484046e-1},
};
constexpr double kB[12] = {
    5.42937341165687622380535766363e-2, 0.0, 0.0, 0.0, 0.0, 4.45031289275240888144113950566e0,
    1.89151789931450038304281599044e0, -5.8012039600105847814672114227e0,
    3.1116436695781989440891606237e-1, -1.52160949662516078556178806805e-1,
    2.01365400804030348374776537501e-1, 4.47106157277725905176885569043e-2};
constexpr double kE5[12] = {
    1.312004499419488073250102996e-2, 0.0, 0.0, 0.0, 0.0, -1.225156446376204440720569753e0,
    -4.957589496572501915214079952e-1, 1.664377182454986536961530415e0,
    -3.503288487499736816886487290e-1, 3.341791187130174790297318841e-1,
    8.192320648511571246570742613e-2, -2.235530786388629525884427845e-2};
constexpr double kB3[12] = {
    2.44094488188976377952755905512e-1, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0,
    7.33846688281611857341361741547e-1, 0.0, 0.0, 2.20588235294117647058823529412e-2};

// Compile-time loop: f(integral_constant<int, I>) for I = B .. E-1.
template <int B, int E, class F>
__device__ __forceinline__ void static_for(F&& f)
{
    if constexpr (B < E) {
        f(std::integral_constant<int, B>{});
        static_for<B + 1, E>(f);
    }
}

// The pair in Nystrom form.  Every system here is q' = p, p' = F(q), and its
// variational equation u' = v, v' = -H(q) u, so a stage's momentum derivative
// depends on the stage's position alone and the position derivatives p_s can be
// eliminated: with G_s = h^2 F(q_s),
//   q_s = q + c_s h p + sum_k abar_sk G_k,         abar = A A,  c_s = sum_j a_sj,
//   q'  = q + h p + sum_k bbar_k G_k,              bbar = b A,
//   p'  = p + (1/h) sum_s b_s G_s,
// the same step in exact arithmetic (Hairer, Norsett and Wanner, Sec. II.14)
// with one sum per degree of freedom and stage instead of two.  The products
// are formed here in double-double arithmetic from the tableau above, so each
// coefficient is the correctly rounded one; the pair's order conditions make
// some of them vanish (abar_s1 for s >= 5, bbar_1..4, bbar_11), which leaves
// rounding residues of the decimal tableau below 1e-13 that are set to zero.
struct Dd {
    double hi, lo;
};
constexpr Dd dd_add_prod(Dd s, double a, double b)
{
    // exact product a b = p + e (Veltkamp splitting, Dekker's product)
    const double ca = 134217729.0 * a, ah = ca - (ca - a), al = a - ah;
    const double cb = 134217729.0 * b, bh = cb - (cb - b), bl = b - bh;
    const double p = a * b, e = ((ah * bh - p) + ah * bl + al * bh) + al * bl;
    // s + (p + e): Knuth's two-sum of the high parts, then renormalise
    const double t = s.hi + p, bb = t - s.hi, err = (s.hi - (t - bb)) + (p - bb);
    const double lo = err + s.lo + e, hi = t + lo;
    return Dd{hi, lo - (hi - t)};
}
constexpr double dd_value(Dd s)
{
    return (s.hi < 1e-13 && s.hi > -1e-13) ? 0.0 : s.hi;
}
struct Nystrom {
    double a[12][12], c[12], b[12], e5[12], e3[12];
};
constexpr Nystrom make_nystrom()
{
    Nystrom n{};
    for (int k = 0; k < 12; ++k) {
        Dd sb{0, 0}, s5{0, 0}, s3{0, 0}, sc{0, 0};
        for (int j = 0; j < 12; ++j) {
            sc = dd_add_prod(sc, kA[k][j], 1.0);
            sb = dd_add_prod(sb, kB[j], kA[j][k]);
            s5 = dd_add_prod(s5, kE5[j], kA[j][k]);
            s3 = dd_add_prod(dd_add_prod(s3, kB[j], kA[j][k]), -kB3[j], kA[j][k]);
        }
        n.c[k] = sc.hi;
        n.b[k] = dd_value(sb);
        n.e5[k] = dd_value(s5);
        n.e3[k] = dd_value(s3);
        for (int s = 0; s < 12; ++s) {
            Dd sa{0, 0};
            for (int j = 0; j < 12; ++j) sa = dd_add_prod(sa, kA[s][j], kA[j][k]);
            n.a[s][k] = dd_value(sa);
        }
    }
    return n;
}
constexpr Nystrom kNys = make_nystrom();
constexpr int nys_terms()
{
    int n = 0;
    for (int s = 0; s < 12; ++s)
        for (int k = 0; k < 12; ++k) n += kNys.a[s][k] != 0.0;
    return n;
}
template <int S, int K>
constexpr double kNa = kNys.a[S][K];
template <int S>
constexpr double kNc = kNys.c[S];
template <int S>
constexpr double kNb = kNys.b[S];
template <int S>
constexpr double kN5 = kNys.e5[S];
template <int S>
constexpr double kN3 = kNys.e3[S];
static_assert(nys_terms() == 48, "the vanishing products of the pair are recognised");

// sum_{j<S} abar_Sj G_j[i] added to acc.
template <int S, int N>
__device__ __forceinline__ double nys_sum(double acc, const double (*G)[N], const int i)
{
    static_for<0, S>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        constexpr double c = kNa<S, j>;
        if constexpr (c != 0.0) acc = fma(c, G[j][i], acc);
    });
    return acc;
}

// Constants of a step of size h.  Steps too small for 1/h (a first guess far
// below the rounding of the state) leave the momenta as they are.
struct StepH {
    double h, nh2, rh;  // h, -h^2, 1/h
};
__device__ __forceinline__ StepH step_h(const double h)
{
    return StepH{h, -h * h, fabs(h) > 1e-290 ? 1.0 / h : 0.0};
}

// A thread's column of the block's shared array: -h^2 Hess V of the twelve
// stages (packed upper triangle), then the orbit's deviation vectors, entry e
// at base[e * kBlock].  The vectors are worked one after another in a loop that
// is not unrolled: held in registers they and the unrolled loop took 255
// registers with spills at k = 4, and the code did not fit the instruction
// cache.  Accesses are volatile so that the Hessians are re-read by each vector
// instead of being kept in registers; the stage values G_s of the vector in
// hand (at most ten live, N doubles each) stay in registers.
template <class Sys>
struct Slab {
    static constexpr int D = 2 * Sys::N, NH = Sys::NH;
    volatile double* base;
    __device__ __forceinline__ volatile double& H(int s, int t) const { return base[(s * NH + t) * kBlock]; }
    __device__ __forceinline__ volatile double& W(int j, int c) const { return base[(12 * NH + j * D + c) * kBlock]; }
};

template <class Sys>
__device__ __forceinline__ Slab<Sys> my_slab()
{
    extern __shared__ double dsm[];
    return Slab<Sys>{dsm + threadIdx.x};
}

// Shared bytes of a block whose threads keep K deviation vectors in the slab.
template <class Sys, int K>
constexpr size_t slab_bytes()
{
    return (size_t)(12 * Sys::NH + K * 2 * Sys::N) * kBlock * sizeof(double);
}

// The LD of a step, dL = |h| sum_s b_s g_s with g the LD integrand of f_s = (p_s, F_s)
// (the LD grows with |t|): stage s's part, from h p and the stages' G, with h p_s = h p
// + sum_j a_sj G_j formed only at the stages with b_s != 0.  p = 1/2: sums of
// sqrt|h p_s| and of sqrt|h^2 F_s| in double-float, widened once per stage; their
// factors |h|^(-1/2) and 1/|h| are applied at the end of the step (ld_total).
struct LdSum {
    double g = 0.0, gq = 0.0;
};
template <class Sys, int s>
__device__ __forceinline__ void ld_stage(const double* hp, const double (*G)[Sys::N], const StepH sh,
                                         const int ld_sqrt, const double ld_p, LdSum& sum)
{
    constexpr int N = Sys::N;
    constexpr double cb = kB[s];
    if constexpr (cb != 0.0) {
        double hps[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            hps[i] = hp[i];
            static_for<0, s>([&](auto jc) {
                constexpr int j = decltype(jc)::value;
                constexpr double c = kA[s][j];
                if constexpr (c != 0.0) hps[i] = fma(c, G[j][i], hps[i]);
            });
        }
        if (ld_sqrt) {
            sum.gq = fma(cb, ff_to_f64(ff_sum_sqrt_abs<N>(hps)), sum.gq);
            sum.g = fma(cb, ff_to_f64(ff_sum_sqrt_abs<N>(G[s])), sum.g);
        } else {
            double f[2 * N];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                f[i] = sh.rh * hps[i];
                f[N + i] = sh.rh * (sh.rh * G[s][i]);
            }
            sum.g = fma(cb, ld_integrand_pow<2 * N>(f, ld_p), sum.g);
        }
    }
}
__device__ __forceinline__ double ld_total(const StepH sh, const int ld_sqrt, const LdSum& sum)
{
    return ld_sqrt ? fma(sqrt(fabs(sh.h)), sum.gq, sum.g) : fabs(sh.h) * sum.g;
}

// For callers of orbit_step that have no use for the stages' G.
struct KeepNothing {
    template <class... T>
    __device__ __forceinline__ void operator()(T...) const
    {
    }
};

// Phase 1, the orbit's twelve stages from x = (q, p) in Nystrom form: xn = the
// step's end point, dL the LD of the step, the stage matrices -h^2 Hess V into the
// slab, and with ERR the error sums times h: h err5_q = sum_k (e5 A)_k G_k, h err5_p =
// (1/h) sum_s e5_s G_s, and err3 likewise.  The small terms are summed first and
// added to the state last.  keep(s, G_s) is called for every stage.
template <class Sys, bool LD, bool ERR, class Keep = KeepNothing>
__device__ __forceinline__ void orbit_step(const Slab<Sys>& sl, const double* x, const StepH sh,
                                           const int ld_sqrt, const double ld_p, const SysPar& sp,
                                           double* xn, double& dL, double* e5, double* e3, Keep keep = Keep{})
{
    constexpr int N = Sys::N, NH = Sys::NH;
    double G[12][N], hp[N], sq[N], sv[N], q5[N], q3[N], p5[N], p3[N];
    LdSum ld;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        hp[i] = __dmul_rn(sh.h, x[N + i]);
        sq[i] = sv[i] = q5[i] = q3[i] = p5[i] = p3[i] = 0.0;
    }
    static_for<0, 12>([&](auto sc) {
        constexpr int s = decltype(sc)::value;
        double qs[N], H[NH];
#pragma unroll
        for (int i = 0; i < N; ++i)
            qs[i] = (s == 0) ? x[i] : nys_sum<s, N>(fma(kNc<s>, hp[i], x[i]), G, i);
        Sys::eval_scaled(qs, sh.nh2, G[s], H, sp);
#pragma unroll
        for (int t = 0; t < NH; ++t) sl.H(s, t) = H[t];
        keep(s, G[s]);
        constexpr double cb = kB[s], nb = kNb<s>;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if constexpr (nb != 0.0) sq[i] = fma(nb, G[s][i], sq[i]);
            if constexpr (cb != 0.0) sv[i] = fma(cb, G[s][i], sv[i]);
            if constexpr (ERR) {
                if constexpr (kN5<s> != 0.0) q5[i] = fma(kN5<s>, G[s][i], q5[i]);
                if constexpr (kN3<s> != 0.0) q3[i] = fma(kN3<s>, G[s][i], q3[i]);
                constexpr double c5 = kE5[s], c3 = kB[s] - kB3[s];
                if constexpr (c5 != 0.0) p5[i] = fma(c5, G[s][i], p5[i]);
                if constexpr (c3 != 0.0) p3[i] = fma(c3, G[s][i], p3[i]);
            }
        }
        if constexpr (LD) ld_stage<Sys, s>(hp, G, sh, ld_sqrt, ld_p, ld);
    });
#pragma unroll
    for (int i = 0; i < N; ++i) {
        xn[i] = x[i] + (hp[i] + sq[i]);
        xn[N + i] = fma(sh.rh, sv[i], x[N + i]);
        if constexpr (ERR) {
            e5[i] = q5[i];
            e3[i] = q3[i];
            e5[N + i] = sh.rh * p5[i];
            e3[N + i] = sh.rh * p3[i];
        }
    }
    if constexpr (LD) dL = ld_total(sh, ld_sqrt, ld);
}

// Phase 2, one deviation vector w = (u, v) through the twelve stages of
// u' = v, v' = -H_s u in Nystrom form with the matrices of phase 1:
// G_s = -h^2 H_s u_s.  204 FP64 instructions for 2 DOF (328 with the stage sums
// of u and v kept apart): the 256 x 256 Henon-Heiles grid with k = 4 and the LD, 60
// steps, took 16.3 ms so and takes 10.6 ms.
template <class Sys>
__device__ __forceinline__ void vector_step(const Slab<Sys>& sl, double* w, const StepH sh)
{
    constexpr int N = Sys::N, NH = Sys::NH;
    double G[12][N], hv[N], sq[N], sv[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        hv[i] = __dmul_rn(sh.h, w[N + i]);
        sq[i] = sv[i] = 0.0;
    }
    static_for<0, 12>([&](auto sc) {
        constexpr int s = decltype(sc)::value;
        double us[N], H[NH];
#pragma unroll
        for (int i = 0; i < N; ++i)
            us[i] = (s == 0) ? w[i] : nys_sum<s, N>(fma(kNc<s>, hv[i], w[i]), G, i);
#pragma unroll
        for (int t = 0; t < NH; ++t) H[t] = sl.H(s, t);
        constexpr double cb = kB[s], nb = kNb<s>;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            double acc = H[hidx<N>(i, 0)] * us[0];
#pragma unroll
            for (int m = 1; m < N; ++m) acc = fma(H[hidx<N>(i, m)], us[m], acc);
            G[s][i] = acc;
            if constexpr (nb != 0.0) sq[i] = fma(nb, acc, sq[i]);
            if constexpr (cb != 0.0) sv[i] = fma(cb, acc, sv[i]);
        }
    });
#pragma unroll
    for (int i = 0; i < N; ++i) {
        w[i] = w[i] + (hv[i] + sq[i]);
        w[N + i] = fma(sh.rh, sv[i], w[N + i]);
    }
}

// 1 / (atol + rtol max(|x|, |xn|)), the weight of a component in the error norm.
__device__ __forceinline__ double err_scale(const double x, const double xn, const double atol, const double rtol)
{
    return rcp_nr(fma(rtol, fmax(fabs(x), fabs(xn)), atol));
}

// The error of a trial from the weighted sums of squares over the D components
// of h err5 and h err3: |h| E5 / sqrt(D (E5 + 0.01 E3)), 0 when both vanish.
template <int D>
__device__ __forceinline__ double err_of(const double E5, const double E3)
{
    if (E5 == 0.0 && E3 == 0.0) return 0.0;
    return E5 * rsqrt_nr((double)D * fma(0.01, E3, E5));
}

// Error norm of a trial over the orbit components:
//   scale_i = atol + rtol max(|x_i|, |xn_i|),  E5 = sum (err5_i / scale_i)^2,
//   E3 likewise, err = |h| E5 / sqrt(D (E5 + 0.01 E3));
// e5 and e3 are h err5 and h err3, which absorbs the factor |h|.
template <int D>
__device__ __forceinline__ double err_norm(const double* x, const double* xn, const double* e5,
                                           const double* e3, const double atol, const double rtol)
{
    double E5 = 0.0, E3 = 0.0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const double rsc = err_scale(x[i], xn[i], atol, rtol);
        const double q5 = e5[i] * rsc, q3 = e3[i] * rsc;
        E5 = fma(q5, q5, E5);
        E3 = fma(q3, q3, E3);
    }
    return err_of<D>(E5, E3);
}

// SALI of two vectors (each normalised first): min(|u + v|, |u - v|).
template <int D>
__device__ __forceinline__ double sali2(const double* a, const double* b)
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

// The K deviation vectors of the slab through one step, scaled to unit length
// with renorm.
template <class Sys, int K>
__device__ __forceinline__ void vectors_step(const Slab<Sys>& sl, const StepH sh, const int renorm)
{
    constexpr int D = 2 * Sys::N;
#pragma unroll 1
    for (int j = 0; j < K; ++j) {
        double w[D];
#pragma unroll
        for (int c = 0; c < D; ++c) w[c] = sl.W(j, c);
        vector_step<Sys>(sl, w, sh);
        if (renorm) unit_vector<D>(w);
#pragma unroll
        for (int c = 0; c < D; ++c) sl.W(j, c) = w[c];
    }
}

// What follows every completed step and its renormalisation (the
// chs_integrate_batch contract): escape, and at health checks finiteness,
// energy drift and the early exit.  Returns the orbit status.
template <class Sys, int K>
__device__ __forceinline__ int32_t post_step(const double* x, const Slab<Sys>& sl, const double L,
                                             const StepArgs& a, const SysPar& sp, const bool check,
                                             const double h0, double& dhm)
{
    constexpr int N = Sys::N, D = 2 * N;
    if (a.escape_r2 > 0.0) {
        double r2 = x[0] * x[0];
#pragma unroll
        for (int i = 1; i < N; ++i) r2 = fma(x[i], x[i], r2);
        if (r2 > a.escape_r2) return CHS_ORBIT_ESCAPED;
    }
    if (check) {
        bool fin = isfinite(L);
#pragma unroll
        for (int c = 0; c < D; ++c) fin = fin && isfinite(x[c]);
#pragma unroll 1
        for (int i = 0; i < K * D; ++i) fin = fin && isfinite((double)sl.W(0, i));
        if (!fin) return CHS_ORBIT_NONFINITE;
        const double dH = fabs(Sys::energy(x, sp) - h0);
        dhm = fmax(dhm, dH);
        if (a.dh_limit > 0.0 && dH > a.dh_limit) return CHS_ORBIT_ENERGY_DRIFT;
        if constexpr (K >= 2) {
            if (a.early_exit) {
                double u[D], v[D];
#pragma unroll
                for (int c = 0; c < D; ++c) {
                    u[c] = sl.W(0, c);
                    v[c] = sl.W(1, c);
                }
                if (sali2<D>(u, v) < a.sali_threshold) return CHS_ORBIT_EARLY_CHAOTIC;
            }
        }
    }
    return CHS_ORBIT_OK;
}

// Calls f(integral_constant<int, K>) for the runtime vector count k, within
// the counts the system supports (k <= 4 for 2 DOF, k <= 6 for 3 DOF).
template <class Sys, class F>
cudaError_t with_k(int k, F&& f)
{
    switch (k) {
    case 0: f(std::integral_constant<int, 0>{}); break;
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5:
        if constexpr (Sys::N >= 3) {
            f(std::integral_constant<int, 5>{});
            break;
        }
        return cudaErrorInvalidValue;
    case 6:
        if constexpr (Sys::N >= 3) {
            f(std::integral_constant<int, 6>{});
            break;
        }
        return cudaErrorInvalidValue;
    default:
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace dp
}  // namespace chs
