// dense.cuh -- an ensemble's running orbits dealt out evenly over the SMs.
//
// With thread t on orbit t, the FORBIDDEN cells of a section grid (a quarter of it)
// leave warps empty or partly filled, and the sub-partitions, each with its own FP64
// unit, unequal numbers of warps: on a 256 x 256 grid under DOP853 the fullest executed 1.75
// times the mean, and it sets the time.  Here 152 blocks of twelve warps, one block
// filling an SM (blocks of four warps did not spread evenly over the SMs: 0.8 of the
// plain form's speed at 18,200 cells), read the statuses once, build the bit mask of OK
// orbits, and their warps take groups of 32 consecutive OK orbits: group w * 152 + i
// belongs to warp w of block i, so every sub-partition gets the same number of groups
// within one.
//
// The status array has to stay as it was until the last block has read it: an
// orbit that freezes leaves its status in the top byte of its n_exec (step counts stay
// far below 2^56), and a second small kernel moves it to its place.
#pragma once

#include "chs_internal.cuh"

namespace chs {

constexpr int kDenseBlocks = 152, kDenseWarps = 12, kDenseThreads = 32 * kDenseWarps;  // 168 registers a thread
constexpr int64_t kDenseOrbits = 1 << 20;
constexpr size_t kDenseSmemLimit = 227 * 1024;

// In dynamic shared memory: the mask of OK orbits, the number of OK orbits before each
// chunk of 32 words (padded to whole warps), the warps' picks, the total.
struct DenseSmem {
    int chunks, heads;  // chunks, padded
    uint32_t* ok;
    int32_t *before, *pick, *total;
    __host__ __device__ DenseSmem(void* base, const int64_t n)
    {
        chunks = (int)((n + 1023) / 1024);
        heads = (chunks + 31) / 32 * 32;
        ok = static_cast<uint32_t*>(base);
        before = reinterpret_cast<int32_t*>(ok + 32 * chunks);
        pick = before + heads;
        total = pick + 32 * kDenseWarps;
    }
    static size_t bytes(const int64_t n)
    {
        const int chunks = (int)((n + 1023) / 1024);
        return sizeof(int32_t) * (32 * chunks + (chunks + 31) / 32 * 32 + 32 * kDenseWarps + 1);
    }
};

// The mask of OK orbits and its prefix sums; returns their number.  All threads.
__device__ __forceinline__ int dense_scan(const DenseSmem& sm, const int64_t n, const int32_t* __restrict__ status)
{
    const int t = threadIdx.x, warp = t / 32, lane = t & 31;
    const int words = (int)((n + 31) / 32);
#pragma unroll 16
    for (int i = warp; i < words; i += kDenseWarps) {
        const int64_t o = (int64_t)i * 32 + lane;
        const uint32_t m = __ballot_sync(0xffffffffu, o < n && status[o < n ? o : 0] == CHS_ORBIT_OK);
        if (lane == 0) sm.ok[i] = m;
    }
    if (words + t < 32 * sm.chunks) sm.ok[words + t] = 0;
    __syncthreads();
    for (int c = warp; c < sm.heads; c += kDenseWarps) {
        const int p = c < sm.chunks ? __popc(sm.ok[32 * c + lane]) : 0;
        const int sum = __reduce_add_sync(0xffffffffu, p);
        if (lane == 0) sm.before[c] = sum;
    }
    __syncthreads();
    if (warp == 0) {
        int total = 0;
        for (int c = lane; c < sm.heads; c += 32) {
            const int own = sm.before[c];
            int upto = own;
#pragma unroll
            for (int d = 1; d < 32; d *= 2) {
                const int u = __shfl_up_sync(0xffffffffu, upto, d);
                if (lane >= d) upto += u;
            }
            sm.before[c] = total + upto - own;
            total += __shfl_sync(0xffffffffu, upto, 31);
        }
        if (lane == 0) *sm.total = total;
    }
    __syncthreads();
    return *sm.total;
}

// The lane's orbit of group g (a whole warp calls this), or -1.
__device__ __forceinline__ int dense_pick(const DenseSmem& sm, const int g)
{
    const int lane = threadIdx.x & 31, lo = 32 * g;
    int32_t* pick = sm.pick + (threadIdx.x - lane);
    __syncwarp();
    pick[lane] = -1;
    __syncwarp();
    int c = -1;  // the last chunk that starts at or before rank lo
    for (int q = lane; q < sm.heads; q += 32) c += __popc(__ballot_sync(0xffffffffu, sm.before[q] <= lo));
    if (c >= sm.chunks) c = sm.chunks - 1;
    for (; c < sm.chunks && sm.before[c] < lo + 32; ++c) {
        uint32_t m = sm.ok[32 * c + lane];
        const int p = __popc(m);
        int r = p;
#pragma unroll
        for (int d = 1; d < 32; d *= 2) {
            const int u = __shfl_up_sync(0xffffffffu, r, d);
            if (lane >= d) r += u;
        }
        r += sm.before[c] - p - lo;  // rank of the word's first orbit within the group
        for (; m; m &= m - 1, ++r)
            if (r >= 0 && r < 32) pick[r] = (32 * c + lane) * 32 + __ffs(m) - 1;
    }
    __syncwarp();
    return pick[lane];
}

// Runs work(o) on the block's share of the OK orbits.
template <class Work>
__device__ __forceinline__ void dense_run(void* smem, const EnsPtrs& e, Work work)
{
    const DenseSmem sm(smem, e.n);
    const int groups = (dense_scan(sm, e.n, e.status) + 31) / 32;
    for (int g = threadIdx.x / 32 * kDenseBlocks + blockIdx.x; g < groups; g += kDenseWarps * kDenseBlocks) {
        const int o = dense_pick(sm, g);
        if (o >= 0) work((int64_t)o);
    }
}

// An orbit's step count and status, as store() of the one-thread forms writes them
// (DENSE: the status waits in the top byte).
template <bool DENSE>
__device__ __forceinline__ void store_exec(const EnsPtrs& e, const int64_t o, const int64_t exec, const int32_t st)
{
    constexpr uint64_t low = ((uint64_t)1 << 56) - 1;
    if (DENSE) {
        e.n_exec[o] = st == CHS_ORBIT_OK ? exec : (int64_t)(((uint64_t)st << 56) | ((uint64_t)exec & low));
    } else {
        e.n_exec[o] = exec;
        e.status[o] = st;
    }
}

// The calls it takes: a plain launch without per-orbit end steps (a warp's groups then
// take equally long), long enough that reading the statuses (~10 us) does
// not show.  Up to 2^20 orbits, whose mask is 128 KB of shared memory (reading 4 MB of
// statuses then takes a block ~0.2 ms of at least 20).
inline bool dense_applies(const StepArgs& a, const EnsPtrs& e, const OrbitList* ol, int64_t least_steps)
{
    return !ol && !e.t_end && e.n <= kDenseOrbits && a.n_steps >= least_steps;
}

// The second kernel: statuses to their places.
cudaError_t launch_dense_status(const EnsPtrs& e, cudaStream_t st);

// Launches a dense kernel whose blocks need `slabs` bytes of shared memory before the
// mask; false, with nothing launched, when they do not fit.
template <class Kernel>
inline bool launch_dense(Kernel kernel, const size_t slabs, const StepArgs& a, const SysPar& sp, const EnsPtrs& e,
                         cudaStream_t st)
{
    const size_t bytes = slabs + DenseSmem::bytes(e.n);
    if (bytes > kDenseSmemLimit) return false;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    kernel<<<kDenseBlocks, kDenseThreads, bytes, st>>>(a, sp, e);
    if (cudaPeekAtLastError() == cudaSuccess) launch_dense_status(e, st);
    return true;
}

}  // namespace chs
