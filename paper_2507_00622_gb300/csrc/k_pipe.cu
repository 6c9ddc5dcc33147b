// k_pipe.cu -- Henon-Heiles RK4 on ensembles too small to fill the GPU: the step
// of 32 orbits spread over the warps of one block.
//
// An FP64 warp instruction occupies its sub-partition's FP64 unit for 64 cycles,
// and one warp carries 32 orbits through ~150 (two vectors, LD) to ~210 of them
// per step, one after another: with fewer than 608 warps (19,456 orbits) most of
// the GPU's 608 FP64 units idle while the others decide the time.  Here each
// group of 32 orbits is a pipeline of warps in one block, lane = orbit:
//   warp O   the orbit's four stages (44 FP64 instructions; 40 without the LD);
//   warp P   the one-step propagator Phi from O's stage positions (49);
//   warps V  two deviation vectors each: w <- Phi w, renormalisation (48);
//   warp L   the LD's sixteen square roots (FP32 double-float, 2 FP64).
// Iteration i works step i in O, step i - 1 in P and L, step i - 2 in V; the data
// of a step pass through double-buffered shared memory (a lane reads only its own
// orbit's column), with one block barrier per iteration.  The pipeline is
// drained at the health checks, where the step's state, vectors and LD meet.
// Every quantity is computed by the functions of the one-thread form (k_small.cu)
// in the same order, so the results are the same bit for bit.
//
// 32 x 32 grid, k = 2, LD, 2000 steps on GB300: 4.32 ms, 14.5 ms with one thread
// per orbit (2.2 against 7.2 us a step).
#include <math.h>

#include "k_pipe.cuh"
#include "rk4_common.cuh"

namespace chs {
namespace {

using Sys = SysHenonHeiles;
constexpr int N = 2, D = 4;

// Warps of the pipeline: O, P, one V per two vectors, L.
template <int K, bool LD>
struct PipeCfg {
    static constexpr int NV = (K + 1) / 2;
    static constexpr int WARPS = 2 + NV + (LD ? 1 : 0);
};

struct PipeSmem {
    double q[2][8][32];     // stage positions of a step
    double f[2][16][32];    // its stage derivatives (LD)
    double phi[2][16][32];  // its propagator
    int32_t live[4][32];    // 1: the lane's orbit took the step
    int32_t bad[4][32];     // at a health check, per V warp and L: a non-finite value
    int32_t aligned[32];    // at a health check: SALI < threshold
    int32_t seg;            // steps until the next health check or the end; 0: done
};

__device__ __forceinline__ void store_phi(const PhiBlocks<N, double>& P, double (*to)[32], const int lane)
{
#pragma unroll
    for (int r = 0; r < N; ++r)
#pragma unroll
        for (int c = 0; c < N; ++c) {
            to[2 * r + c][lane] = P.A[r][c];
            to[4 + 2 * r + c][lane] = P.B[r][c];
            to[8 + 2 * r + c][lane] = P.C[r][c];
            to[12 + 2 * r + c][lane] = P.D[r][c];
        }
}

__device__ __forceinline__ void load_phi(PhiBlocks<N, double>& P, const double (*from)[32], const int lane)
{
#pragma unroll
    for (int r = 0; r < N; ++r)
#pragma unroll
        for (int c = 0; c < N; ++c) {
            P.A[r][c] = from[2 * r + c][lane];
            P.B[r][c] = from[4 + 2 * r + c][lane];
            P.C[r][c] = from[8 + 2 * r + c][lane];
            P.D[r][c] = from[12 + 2 * r + c][lane];
        }
}

template <int K, bool LD, int MODE>
__global__ void __launch_bounds__(32 * PipeCfg<K, LD>::WARPS)
k_integrate_pipe(const StepArgs a, const SysPar sp, const EnsPtrs e, const OrbitList ol)
{
    constexpr int NV = PipeCfg<K, LD>::NV;
    __shared__ PipeSmem sm;
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
    const bool is_o = warp == 0, is_p = warp == 1, is_v = warp >= 2 && warp < 2 + NV, is_l = LD && warp == 2 + NV;
    const int64_t n = e.n, t = (int64_t)blockIdx.x * 32 + lane;
    int64_t o = t;
    bool mine = t < n;
    if (MODE == kModeList) {
        mine = t < *ol.count;
        o = mine ? ol.list[t] : 0;
    }
    mine = mine && e.status[o] == CHS_ORBIT_OK;

    // each warp's part of the orbit's state
    double x[D], w[2][D], L = 0.0, h0 = 0.0, dhm = 0.0;
    int64_t exec0 = 0, todo = 0, s = 0;
    int64_t until = a.sample_every > 0 ? a.sample_every - (a.step0 % a.sample_every) : -1;
    int32_t st = CHS_ORBIT_OK;
    const int j0 = 2 * (warp - 2);  // a V warp's first vector
    const int nvec = is_v ? (K - j0 < 2 ? K - j0 : 2) : 0;
    double* wg = static_cast<double*>(e.w);
    const long long t_start = clock64();
    if (is_o) {
#pragma unroll
        for (int c = 0; c < D; ++c) x[c] = mine ? e.x[c * n + o] : 0.0;
        if (mine) {
            h0 = e.h0[o];
            dhm = e.dh_max[o];
            exec0 = e.n_exec[o];
            todo = a.n_steps;
            if (e.t_end) todo = min(todo, max(e.t_end[o] - exec0, (int64_t)0));
        }
    }
    if (is_v) {
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
            for (int c = 0; c < D; ++c) w[v][c] = (mine && v < nvec) ? wg[((j0 + v) * D + c) * n + o] : 0.0;
    }
    if (is_l && mine) L = e.ld[o];

    for (;;) {
        // the segment: to the next health check or the last step of any lane
        if (is_o) {
            const int64_t left = st == CHS_ORBIT_OK ? todo - s : 0;
            int seg = (int)(left < (1 << 20) ? left : (1 << 20));
            seg = __reduce_max_sync(0xffffffffu, seg);
            if (until > 0 && until < seg) seg = (int)until;
            if (lane == 0) sm.seg = seg;
        }
        __syncthreads();
        const int seg = sm.seg;
        if (seg == 0) break;
        bool last_live = false;
        for (int i = 0; i < seg + 2; ++i) {
            if (is_o && i < seg) {
                const int b = i & 1;
                const bool live = st == CHS_ORBIT_OK && s < todo;
                sm.live[i & 3][lane] = live;
                last_live = live;
                if (live) {
                    ++s;
                    if constexpr (LD) {
                        rk4_stages_f<Sys>(x, a.dt, sp, [&](int k, const double* xs, const double* f, const double*) {
#pragma unroll
                            for (int c = 0; c < N; ++c) sm.q[b][2 * k + c][lane] = xs[c];
#pragma unroll
                            for (int c = 0; c < D; ++c) sm.f[b][4 * k + c][lane] = f[c];
                        });
                    } else {
                        double none = 0.0;
                        rk4_stages<Sys, false, false>(x, none, a.dt, 0, 0.0, sp,
                                                      [&](int k, const double* xs, const double*) {
#pragma unroll
                                                          for (int c = 0; c < N; ++c) sm.q[b][2 * k + c][lane] = xs[c];
                                                      });
                    }
                    if (escaped<N>(x, a.escape_hi, a.escape_r2)) st = CHS_ORBIT_ESCAPED;
                }
            } else if (is_p && i >= 1 && i <= seg && sm.live[(i - 1) & 3][lane]) {
                const int b = (i - 1) & 1;
                double q[4][2];
#pragma unroll
                for (int k = 0; k < 4; ++k)
#pragma unroll
                    for (int c = 0; c < N; ++c) q[k][c] = sm.q[b][2 * k + c][lane];
                PhiBlocks<N, double> P;
                phi_build_hh<double>(q, a.dt, P);
                store_phi(P, sm.phi[b], lane);
            } else if (is_l && i >= 1 && i <= seg && sm.live[(i - 1) & 3][lane]) {
                const int b = (i - 1) & 1;
                FF fL{0.0f, 0.0f};
                double aL = 0.0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    double f[D];
#pragma unroll
                    for (int c = 0; c < D; ++c) f[c] = sm.f[b][4 * k + c][lane];
                    ld_add_stage<D>(k, f, a.ld_sqrt, a.ld_p, fL, aL);
                }
                ld_finish(L, a.dt, a.ld_sqrt, fL, aL);
            } else if (is_v && i >= 2 && sm.live[(i - 2) & 3][lane]) {
                const int b = i & 1;
                PhiBlocks<N, double> P;
                load_phi(P, sm.phi[b], lane);
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    if (v >= nvec) break;
                    phi_apply<N, double>(P, w[v]);
                    if (a.renorm) unit_vector<D>(w[v]);
                }
            }
            __syncthreads();
        }
        if (until > 0) {
            until -= seg;
            if (until == 0) {
                // health check: what the orbit's owner does not hold comes through flags
                until = a.sample_every;
                if (is_v) {
                    bool fin = true;
#pragma unroll
                    for (int v = 0; v < 2; ++v)
#pragma unroll
                        for (int c = 0; c < D; ++c) fin = fin && (v >= nvec || isfinite(w[v][c]));
                    sm.bad[warp - 2][lane] = !fin;
                    if (warp == 2) sm.aligned[lane] = a.early_exit && sali_of<D>(w[0], w[1]) < a.sali_threshold;
                }
                if (is_l) sm.bad[NV][lane] = !isfinite(L);
                __syncthreads();
                if (is_o && last_live && st == CHS_ORBIT_OK) {
                    bool fin = true;
#pragma unroll
                    for (int c = 0; c < D; ++c) fin = fin && isfinite(x[c]);
#pragma unroll
                    for (int v = 0; v < NV + (LD ? 1 : 0); ++v) fin = fin && !sm.bad[v][lane];
                    if (!fin) {
                        st = CHS_ORBIT_NONFINITE;
                    } else {
                        const double dH = fabs(Sys::energy(x, sp) - h0);
                        dhm = fmax(dhm, dH);
                        if (a.dh_limit > 0.0 && dH > a.dh_limit)
                            st = CHS_ORBIT_ENERGY_DRIFT;
                        else if (sm.aligned[lane])
                            st = CHS_ORBIT_EARLY_CHAOTIC;
                        else if (budget_spent(a, t_start))
                            st = CHS_ORBIT_STEP_BUDGET;
                    }
                }
            }
        }
    }
    if (!mine) return;
    if (is_o) {
#pragma unroll
        for (int c = 0; c < D; ++c) e.x[c * n + o] = x[c];
        e.dh_max[o] = dhm;
        const int64_t exec = exec0 + s;
        const bool keep = st == CHS_ORBIT_OK && (!e.t_end || exec < e.t_end[o]);
        e.n_exec[o] = exec;
        e.status[o] = st;
        if (MODE == kModeList) list_append(ol, keep, (int32_t)o);
    }
    if (is_v) {
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
            for (int c = 0; c < D; ++c)
                if (v < nvec) wg[((j0 + v) * D + c) * n + o] = w[v][c];
    }
    if (is_l) e.ld[o] = L;
}

// The Lyapunov spectrum by QR (chs_lyapunov_spectrum) as the same pipeline: warp O
// the orbit, warp P the propagator, warp V0 the vectors 0 and 1, warp V1 the
// vectors 2 and 3 one iteration behind V0.  At a QR step V0 orthonormalises its two
// vectors and hands them to V1, which removes their components from its own: the
// modified Gram-Schmidt of k_lyap_small in the same order, the same results.
// 500 steps, QR every 10 on GB300, at 4864, 9728 and 14,592 orbits: 1.31, 1.84 and 2.37
// ms, 3.07 ms with one thread per orbit; 3.12 against 3.07 ms at 19,456.
//
// DENSE: a section grid's FORBIDDEN cells (a quarter of it) would leave lanes empty in
// most groups, so block b takes the OK orbits with ranks 32 b ... 32 b + 31, which every
// block counts for itself from ic_status (a few us); blocks past the last one end.
// A 128 x 128 section grid, 500 steps: 3.05 -> 2.35 ms.
struct LyapSmem {
    double q[2][8][32];     // stage positions of a step
    double phi[4][16][32];  // its propagator (read by V0 and, an iteration later, V1)
    double q01[2][8][32];   // V0's unit vectors of a QR step
    int32_t bad[2][32];     // at a health check: V0's, V1's exponent sums are not finite
    int32_t live[32];       // the orbit is running
    uint32_t ok[kLyapDenseOrbits / 32];  // DENSE: the OK orbits, a bit each
    int32_t sums[4], pick[32];           // their number per warp's part, the block's orbits
};

// DENSE: the lane's orbit, or n; the block writes the outputs of the other orbits of
// its own 32.
__device__ __forceinline__ int64_t pick_orbit(LyapSmem& sm, const int64_t n, const int32_t* __restrict__ ic_status,
                                              double* __restrict__ lambda, int32_t* __restrict__ status_out)
{
    constexpr int PER = (kLyapDenseOrbits / 32 + 127) / 128;
    const int t = threadIdx.x, warp = t / 32, lane = t & 31, tiles = (int)((n + 127) / 128), words = 4 * tiles;
#pragma unroll 8
    for (int i = 0; i < tiles; ++i) {
        const int64_t o = i * 128 + t;
        const uint32_t m = __ballot_sync(0xffffffffu, o < n && ic_status[o < n ? o : 0] == CHS_ORBIT_OK);
        if (lane == 0) sm.ok[i * 4 + warp] = m;
    }
    if (t < 32) sm.pick[t] = -1;
    const int64_t own = (int64_t)blockIdx.x * 32 + lane;
    if (own < n && ic_status[own] != CHS_ORBIT_OK) {
        if (warp == 0) status_out[own] = ic_status[own];
        lambda[warp * n + own] = __longlong_as_double(0x7ff8000000000000LL);
    }
    __syncthreads();
    int mine = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (t * PER + i < words) mine += __popc(sm.ok[t * PER + i]);
    int rank = mine;  // inclusive prefix over the block's threads
#pragma unroll
    for (int d = 1; d < 32; d *= 2) {
        const int v = __shfl_up_sync(0xffffffffu, rank, d);
        if (lane >= d) rank += v;
    }
    if (lane == 31) sm.sums[warp] = rank;
    __syncthreads();
    for (int i = 0; i < warp; ++i) rank += sm.sums[i];
    rank -= mine + (int)blockIdx.x * 32;  // of the thread's first orbit, from the block's first
    if (rank < 32 && rank + mine > 0) {
        for (int i = 0; i < PER; ++i) {
            if (t * PER + i >= words) break;
            for (uint32_t m = sm.ok[t * PER + i]; m; m &= m - 1, ++rank)
                if (rank >= 0 && rank < 32) sm.pick[rank] = (t * PER + i) * 32 + __ffs(m) - 1;
        }
    }
    __syncthreads();
    return sm.pick[lane] < 0 ? n : sm.pick[lane];
}

template <bool DENSE>
__global__ void __launch_bounds__(128)
k_lyap_pipe(const StepArgs a, const SysPar sp, const int64_t n, const double* __restrict__ ics,
            const int32_t* __restrict__ ic_status, double* __restrict__ lambda, int32_t* __restrict__ status_out)
{
    __shared__ LyapSmem sm;
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
    const int64_t o = DENSE ? pick_orbit(sm, n, ic_status, lambda, status_out) : (int64_t)blockIdx.x * 32 + lane;
    const bool valid = o < n;
    if (DENSE && !__syncthreads_or(valid)) return;
    double x[D], w[2][D], S[2] = {0.0, 0.0};
    int32_t st = valid ? (ic_status ? ic_status[o] : CHS_ORBIT_OK) : CHS_ORBIT_FORBIDDEN;
    bool fin = true;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        x[c] = valid ? ics[c * n + o] : 0.0;
        fin = fin && isfinite(x[c]);
    }
    if (st == CHS_ORBIT_OK && !fin) st = CHS_ORBIT_NONFINITE;
    const int j0 = 2 * (warp - 2);  // a V warp's first vector
#pragma unroll
    for (int v = 0; v < 2; ++v)
#pragma unroll
        for (int c = 0; c < D; ++c) w[v][c] = (j0 + v == c) ? 1.0 : 0.0;
    if (warp == 0) sm.live[lane] = st == CHS_ORBIT_OK;
    const long long t_start = clock64();
    int64_t until_qr = a.qr_every;  // V warps
    int64_t s = 0;                  // steps taken before the segment
    const int64_t every = a.sample_every > 0 ? a.sample_every : a.n_steps;
    while (s < a.n_steps) {
        const int64_t seg = a.n_steps - s < every ? a.n_steps - s : every;
        __syncthreads();  // live is written
        const bool live = sm.live[lane] != 0;
        if (!__syncthreads_or(live)) break;
        for (int64_t i = 0; i < seg + 3; ++i) {
            if (warp == 0) {
                if (live && i < seg) {
                    const int b = (int)(i & 1);
                    double none = 0.0;
                    rk4_stages<Sys, false, false>(x, none, a.dt, 0, 0.0, sp, [&](int k, const double* xs, const double*) {
#pragma unroll
                        for (int c = 0; c < N; ++c) sm.q[b][2 * k + c][lane] = xs[c];
                    });
                }
            } else if (warp == 1) {
                if (live && i >= 1 && i <= seg) {
                    const int b = (int)((i - 1) & 1), f = (int)((i - 1) & 3);
                    double q[4][2];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
#pragma unroll
                        for (int c = 0; c < N; ++c) q[k][c] = sm.q[b][2 * k + c][lane];
                    PhiBlocks<N, double> P;
                    phi_build_hh<double>(q, a.dt, P);
                    store_phi(P, sm.phi[f], lane);
                }
            } else {
                const int64_t k = i - warp;  // the step this warp works
                if (live && k >= 0 && k < seg) {
                    PhiBlocks<N, double> P;
                    load_phi(P, sm.phi[k & 3], lane);
                    phi_apply<N, double>(P, w[0]);
                    phi_apply<N, double>(P, w[1]);
                    if (--until_qr == 0 || s + k + 1 == a.n_steps) {
                        until_qr = a.qr_every;
                        const int b = (int)(k & 1);
                        if (warp == 3) {
                            double q[2][D];
#pragma unroll
                            for (int c = 0; c < D; ++c) {
                                q[0][c] = sm.q01[b][c][lane];
                                q[1][c] = sm.q01[b][D + c][lane];
                            }
#pragma unroll
                            for (int v = 0; v < 2; ++v) {
                                remove_component<D>(q[0], w[v]);
                                remove_component<D>(q[1], w[v]);
                            }
                        }
                        normalise_log<D>(w[0], S[0]);
                        remove_component<D>(w[0], w[1]);
                        normalise_log<D>(w[1], S[1]);
                        if (warp == 2) {
#pragma unroll
                            for (int c = 0; c < D; ++c) {
                                sm.q01[b][c][lane] = w[0][c];
                                sm.q01[b][D + c][lane] = w[1][c];
                            }
                        }
                    }
                }
            }
            __syncthreads();
        }
        s += seg;
        if (a.sample_every > 0 && seg == every) {
            if (warp >= 2) sm.bad[warp - 2][lane] = !(isfinite(S[0]) && isfinite(S[1]));
            __syncthreads();
            if (warp == 0 && live) {
                bool f2 = !sm.bad[0][lane] && !sm.bad[1][lane];
#pragma unroll
                for (int c = 0; c < D; ++c) f2 = f2 && isfinite(x[c]);
                if (!f2)
                    st = CHS_ORBIT_NONFINITE;
                else if (budget_spent(a, t_start))
                    st = CHS_ORBIT_STEP_BUDGET;
                sm.live[lane] = st == CHS_ORBIT_OK;
            }
        }
    }
    __syncthreads();
    if (!valid) return;
    if (warp == 0) status_out[o] = st;
    if (warp >= 2) {
        const double T = (double)a.n_steps * a.dt;
        const bool good = sm.live[lane] != 0;
#pragma unroll
        for (int v = 0; v < 2; ++v)
            lambda[(j0 + v) * n + o] = good ? S[v] / T : __longlong_as_double(0x7ff8000000000000LL);
    }
}

template <int K, bool LD>
cudaError_t pipe_k(const StepArgs& a, const SysPar& sp, const EnsPtrs& e, const OrbitList* ol, cudaStream_t st)
{
    const unsigned g = blocks_for(e.n, 32);
    constexpr int threads = 32 * PipeCfg<K, LD>::WARPS;
    if (ol && ol->list)
        k_integrate_pipe<K, LD, kModeList><<<g, threads, 0, st>>>(a, sp, e, *ol);
    else
        k_integrate_pipe<K, LD, kModeAll><<<g, threads, 0, st>>>(a, sp, e, OrbitList{});
    return cudaGetLastError();
}

template <bool LD>
cudaError_t pipe_ld(int k, const StepArgs& a, const SysPar& sp, const EnsPtrs& e, const OrbitList* ol, cudaStream_t st)
{
    switch (k) {
    case 2: return pipe_k<2, LD>(a, sp, e, ol, st);
    case 3: return pipe_k<3, LD>(a, sp, e, ol, st);
    case 4: return pipe_k<4, LD>(a, sp, e, ol, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

// The pipeline pays while groups of 32 orbits leave FP64 units idle.  us per step
// (one thread per orbit in brackets) at 4864, 9728 and 14,592 orbits, one, two and
// three groups per SM: k = 2 without the LD 2.1, 2.8 and 4.1 (4.7); k = 3 with the LD
// 2.2, 3.4 and 4.9 (7.3); k = 4 with the LD 2.3, 3.8 and 5.5 (8.1).  At four groups per
// SM the GPU is full either way.
// It is drained at every health check (two of its iterations), which at
// intervals below 16 steps costs more than an eighth.  A block size that the
// caller asked for runs the one-thread form.  A queue launch of so few orbits, which
// hold every warp at once anyway, runs it without the queue.
bool pipe_applies(const SysPar& sp, int k, const StepArgs& a, int64_t n)
{
    return sp.model == CHS_HENON_HEILES && k >= 2 && k <= 4 && a.block == 0 &&
           (a.sample_every == 0 || a.sample_every >= 16) && n <= kPipeOrbits;
}

cudaError_t launch_integrate_pipe(const SysPar& sp, int k, bool ld, const StepArgs& a, const EnsPtrs& e,
                                  const OrbitList* ol, cudaStream_t st)
{
    return ld ? pipe_ld<true>(k, a, sp, e, ol, st) : pipe_ld<false>(k, a, sp, e, ol, st);
}

// The DENSE form: the caller's status array may be the output array, which one block
// would write before another has counted; then the groups stay as they lie, as they do
// where one group per SM holds every cell.
static bool lyap_dense(int64_t n, const int32_t* ic_status, const int32_t* status)
{
    const uintptr_t i = (uintptr_t)ic_status, o = (uintptr_t)status, bytes = (uintptr_t)n * sizeof(int32_t);
    return ic_status && n > kLyapDenseFrom && n <= kLyapDenseOrbits && (i + bytes <= o || o + bytes <= i);
}

// Up to three groups of 32 orbits per SM (figures at k_lyap_pipe): 14,592 orbits, or
// 18,432 cells of a grid, of which up to 79 % are orbits (17,000 cells, 75 % and all of
// them OK: 2.36 and 3.13 ms, 3.08 with one thread per orbit); health checks as above.
bool lyap_pipe_applies(const SysPar& sp, const StepArgs& a, int64_t n, const int32_t* ic_status, const int32_t* status)
{
    return sp.model == CHS_HENON_HEILES && a.block == 0 && (a.sample_every == 0 || a.sample_every >= 16) &&
           (n <= kLyapPipeOrbits || lyap_dense(n, ic_status, status));
}

cudaError_t launch_lyap_pipe(const SysPar& sp, const StepArgs& a, int64_t n, const double* ics,
                             const int32_t* ic_status, double* lambda, int32_t* status, cudaStream_t st)
{
    if (lyap_dense(n, ic_status, status))
        k_lyap_pipe<true><<<blocks_for(n, 32), 128, 0, st>>>(a, sp, n, ics, ic_status, lambda, status);
    else
        k_lyap_pipe<false><<<blocks_for(n, 32), 128, 0, st>>>(a, sp, n, ics, ic_status, lambda, status);
    return cudaGetLastError();
}

}  // namespace chs
