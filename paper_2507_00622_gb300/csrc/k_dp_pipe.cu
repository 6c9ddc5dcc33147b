// k_dp_pipe.cu -- fixed-step DOP853 on Henon-Heiles ensembles too small to fill the
// GPU: the step of 32 orbits spread over the warps of one block, as k_pipe.cu does
// for RK4 (lane = orbit, one block barrier per iteration):
//   warp O    the orbit's twelve stages (252 FP64 instructions);
//   warps V   one deviation vector each through the stages of the step before (213);
//   warp L    the LD of that step (119).
// One thread per orbit runs them one after another.  Stage matrices, and for the LD
// the stage values G, pass through double-buffered shared memory.  The functions are
// those of the one-thread form (dop853.cuh), in the same order: the results are the
// same bit for bit.
//
// One thread per orbit leaves an ensemble of a few thousand orbits at one warp or none
// per sub-partition, so the step takes the time of its whole serial stream of FP64
// instructions (797 at k = 2 with the LD) whatever the ensemble's size.  Here the
// longest warp's 252 remain and the block's other warps use the SM's other FP64
// units: 800 orbits, k = 2 with the LD, 29.7 -> 9.1 us per step; k = 4, 43.7 -> 12.5.
#include "dop853.cuh"
#include "k_dp_pipe.cuh"

namespace chs {
namespace {

using Sys = SysHenonHeiles;
constexpr int N = 2, D = 4, NH = 3;

template <int K, bool LD>
struct DpSmem {
    double H[2][12 * NH * 32];                    // a step's stage matrices (dp::Slab's layout)
    double G[2][LD ? 24 : 1][32], hp[2][N][32];   // its stage values and h p (LD)
    double w[K < 2 ? 1 : 2][D][32];               // at a health check with early exit: w_0 and w_1
    int32_t live[2][32];                          // 1: the lane's orbit took the step
    int32_t bad[K + 1][32];                       // at a health check, per V warp and L: a non-finite value
    int32_t seg;                                  // steps until the next health check or the end; 0: done
};

template <int K, bool LD, int MODE>
__global__ void __launch_bounds__(dp_pipe_warps(K, LD) * 32, dp_pipe_blocks(K, LD))
k_dp_pipe(const StepArgs a, const SysPar sp, const EnsPtrs e, const OrbitList ol)
{
    __shared__ DpSmem<K, LD> sm;
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
    const bool is_o = warp == 0, is_v = warp >= 1 && warp <= K, is_l = LD && warp == 1 + K;
    const int64_t n = e.n, t = (int64_t)blockIdx.x * 32 + lane;
    int64_t o = t;
    bool mine = t < n;
    if (MODE == kModeList) {
        mine = t < *ol.count;
        o = mine ? ol.list[t] : 0;
    }
    mine = mine && e.status[o] == CHS_ORBIT_OK;

    const int j = warp - 1;  // a V warp's vector
    double* wg = static_cast<double*>(e.w);
    double x[D], w[D], L = 0.0, h0 = 0.0, dhm = 0.0;
    int64_t exec0 = 0, todo = 0, s = 0;
    int64_t until = a.sample_every > 0 ? a.sample_every - (a.step0 % a.sample_every) : -1;
    int32_t st = CHS_ORBIT_OK;
    const long long t_start = clock64();
#pragma unroll
    for (int c = 0; c < D; ++c) {
        x[c] = (is_o && mine) ? e.x[c * n + o] : 0.0;
        w[c] = (is_v && mine) ? wg[(j * D + c) * n + o] : 0.0;
    }
    if (is_o && mine) {
        h0 = e.h0[o];
        dhm = e.dh_max[o];
        exec0 = e.n_exec[o];
        todo = a.n_steps;
        if (e.t_end) todo = min(todo, max(e.t_end[o] - exec0, (int64_t)0));
    }
    if (is_l && mine) L = e.ld[o];
    const dp::StepH sh = dp::step_h(a.dt);

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
        for (int i = 0; i < seg + 1; ++i) {
            const int b = is_o ? i & 1 : (i & 1) ^ 1;  // O's buffer; the others work the one before
            const dp::Slab<Sys> sl{sm.H[b] + lane};
            if (is_o && i < seg) {
                const bool live = st == CHS_ORBIT_OK && s < todo;
                sm.live[b][lane] = live;
                last_live = live;
                if (live) {
                    ++s;
                    if constexpr (LD) {
#pragma unroll
                        for (int c = 0; c < N; ++c) sm.hp[b][c][lane] = __dmul_rn(sh.h, x[N + c]);
                    }
                    double xn[D], none = 0.0;
                    dp::orbit_step<Sys, false, false>(sl, x, sh, 0, 0.0, sp, xn, none, nullptr, nullptr,
                                                      [&](int k, const double* g) {
                                                          if constexpr (LD) {
#pragma unroll
                                                              for (int c = 0; c < N; ++c) sm.G[b][2 * k + c][lane] = g[c];
                                                          }
                                                      });
#pragma unroll
                    for (int c = 0; c < D; ++c) x[c] = xn[c];
                    if (a.escape_r2 > 0.0) {
                        double r2 = x[0] * x[0];
#pragma unroll
                        for (int c = 1; c < N; ++c) r2 = fma(x[c], x[c], r2);
                        if (r2 > a.escape_r2) st = CHS_ORBIT_ESCAPED;
                    }
                }
            } else if (is_v && i >= 1 && sm.live[b][lane]) {
                dp::vector_step<Sys>(sl, w, sh);
                if (a.renorm) unit_vector<D>(w);
            } else if (is_l && i >= 1 && sm.live[b][lane]) {
                double G[12][N], hp[N];
                dp::LdSum ld;
#pragma unroll
                for (int c = 0; c < N; ++c) hp[c] = sm.hp[b][c][lane];
                dp::static_for<0, 12>([&](auto kc) {
                    constexpr int k = decltype(kc)::value;
#pragma unroll
                    for (int c = 0; c < N; ++c) G[k][c] = sm.G[b][LD ? 2 * k + c : 0][lane];
                    dp::ld_stage<Sys, k>(hp, G, sh, a.ld_sqrt, a.ld_p, ld);
                });
                L += dp::ld_total(sh, a.ld_sqrt, ld);
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
                    for (int c = 0; c < D; ++c) fin = fin && isfinite(w[c]);
                    sm.bad[j][lane] = !fin;
                    if (K >= 2 && j < 2 && a.early_exit) {
#pragma unroll
                        for (int c = 0; c < D; ++c) sm.w[K >= 2 ? j : 0][c][lane] = w[c];
                    }
                }
                if (is_l) sm.bad[K][lane] = !isfinite(L);
                __syncthreads();
                if (is_o && last_live && st == CHS_ORBIT_OK) {
                    bool fin = true;
#pragma unroll
                    for (int c = 0; c < D; ++c) fin = fin && isfinite(x[c]);
#pragma unroll
                    for (int v = 0; v < K + (LD ? 1 : 0); ++v) fin = fin && !sm.bad[v][lane];
                    if (!fin) {
                        st = CHS_ORBIT_NONFINITE;
                    } else {
                        const double dH = fabs(Sys::energy(x, sp) - h0);
                        dhm = fmax(dhm, dH);
                        bool aligned = false;
                        if constexpr (K >= 2) {
                            if (a.early_exit) {
                                double y[2][D];
#pragma unroll
                                for (int v = 0; v < 2; ++v)
#pragma unroll
                                    for (int c = 0; c < D; ++c) y[v][c] = sm.w[v][c][lane];
                                aligned = dp::sali2<D>(y[0], y[1]) < a.sali_threshold;
                            }
                        }
                        if (a.dh_limit > 0.0 && dH > a.dh_limit)
                            st = CHS_ORBIT_ENERGY_DRIFT;
                        else if (aligned)
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
        for (int c = 0; c < D; ++c) wg[(j * D + c) * n + o] = w[c];
    }
    if (is_l) e.ld[o] = L;
}

template <int K, bool LD>
cudaError_t dp_pipe_k(const StepArgs& a, const SysPar& sp, const EnsPtrs& e, const OrbitList* ol, cudaStream_t st)
{
    const unsigned g = blocks_for(e.n, 32);
    constexpr int threads = 32 * dp_pipe_warps(K, LD);
    if (ol && ol->list)
        k_dp_pipe<K, LD, kModeList><<<g, threads, 0, st>>>(a, sp, e, *ol);
    else
        k_dp_pipe<K, LD, kModeAll><<<g, threads, 0, st>>>(a, sp, e, OrbitList{});
    return cudaGetLastError();
}

}  // namespace

// The pipeline pays while it fits in one wave.  us per step (one thread per orbit in
// brackets) at 4864, 9728 and 14,592 orbits: k = 1 without the LD 8.8, 9.8 and 13.4
// (16.1); k = 2 with the LD 9.1, 16.2 and 24.8 (29.7); k = 4 without the LD 12.6, 20.6 and
// 30.8 (36.8); k = 4 with the LD 12.5 and 23.3 (43.7), then a second wave.  It is drained
// at every health check (one of its iterations); at intervals below 8 steps the
// one-thread form runs.  A queue launch of so few orbits, which hold every warp at
// once anyway, runs without the queue.
bool dp_pipe_applies(const SysPar& sp, int k, bool ld, const StepArgs& a, int64_t n)
{
    return sp.model == CHS_HENON_HEILES && k >= 1 && k <= 4 &&
           (a.sample_every == 0 || a.sample_every >= 8) && n <= dp_pipe_orbits(k, ld);
}

cudaError_t launch_dp_pipe(const SysPar& sp, int k, bool ld, const StepArgs& a, const EnsPtrs& e, const OrbitList* ol,
                           cudaStream_t st)
{
    switch (k) {
    case 1: return ld ? dp_pipe_k<1, true>(a, sp, e, ol, st) : dp_pipe_k<1, false>(a, sp, e, ol, st);
    case 2: return ld ? dp_pipe_k<2, true>(a, sp, e, ol, st) : dp_pipe_k<2, false>(a, sp, e, ol, st);
    case 3: return ld ? dp_pipe_k<3, true>(a, sp, e, ol, st) : dp_pipe_k<3, false>(a, sp, e, ol, st);
    case 4: return ld ? dp_pipe_k<4, true>(a, sp, e, ol, st) : dp_pipe_k<4, false>(a, sp, e, ol, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace chs
