// k_mlp.cu -- the early-stop surrogate: a 12 -> 128 -> 128 -> 128 -> 2 ReLU
// multilayer perceptron with BF16 weights and activations and FP32
// accumulation, its training kernels (loss gradient, backward pass, Adam) and
// the fused decision kernel used during integration.
//
// Inputs (features) of an orbit still running at the decision time t:
//   f_i = log10(max(SALI(t_i), 1e-20)) / 8,  t_i = (i + 1) t / S, i < S (S = 10)
//   f_10 = LD(t) / t - 1            (the mean LD rate, centred)
//   f_11 = (E_o - 0.133) / 0.033    (the orbit's energy, centred)
// Outputs: y_0 = logit of "chaotic at the final time", y_1 = final log10(SALI) / 8.
//
// Parameter layout (one flat array, row-major out x in):
//   W1 [128][12], b1 [128], W2 [128][128], b2 [128], W3 [128][128], b3 [128],
//   W4 [2][128], b4 [2]   -- 34,946 values.
//
// The hidden layers of the forward pass run on the tensor cores (below), the
// training kernels on the FP32 pipe; weights and activations are stored in BF16.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <math.h>

#include "chs_internal.cuh"

namespace chs {

namespace cg = cooperative_groups;

constexpr int kF = 12, kH = 128, kO = 2, kS = 10;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kF, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH * kH, kOffW4 = kOffB3 + kH,
              kOffB4 = kOffW4 + kO * kH, kParams = kOffB4 + kO;

size_t mlp_param_count() { return (size_t)kParams; }

__device__ __forceinline__ float bf(const __nv_bfloat16 v) { return __bfloat162float(v); }

// Features of orbit o (see the file comment); non-finite SALI samples count as 1e-20.
__device__ __forceinline__ void features(const double* __restrict__ series, const int S, const double* ld,
                                         const double t, const double* E, const int64_t n, const int64_t o,
                                         float* f)
{
    for (int i = 0; i < kS; ++i) {
        double s = i < S ? series[(int64_t)i * n + o] : 1e-20;
        s = (s > 1e-20 && isfinite(s)) ? s : 1e-20;
        f[i] = (float)(log10(s) / 8.0);
    }
    f[10] = (float)(ld[o] / t - 1.0);
    f[11] = (float)((E[o] - 0.133) / 0.033);
}

__global__ void k_mlp_features(const double* __restrict__ series, const int S, const double* __restrict__ ld,
                               const double t, const double* __restrict__ E, const int64_t n, float* __restrict__ X)
{
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= n) return;
    float f[kF];
    features(series, S, ld, t, E, n, o, f);
#pragma unroll
    for (int i = 0; i < kF; ++i) X[(int64_t)i * n + o] = f[i];
}

// ---------------------------------------------------------------------------
// Forward pass
//
// A persistent grid (one block of kFwdWarps warps per SM); a warp takes tiles of
// 32 samples, as two halves of 16 rows (16 samples where 32 would leave SMs
// without a tile: a batch of 4096 then has two warps at work on most SMs), through
// all layers without leaving its own shared memory:
//   features / X   FP32, 32 samples at a time;
//   layer 1        FP32 FMA chains (K = 12, FP32 inputs);
//   layers 2, 3    mma.sync m16n8k16 (BF16 operands, FP32 accumulators), weights
//                  resident in shared memory, operands by ldmatrix;
//   layer 4        FP32 FMA chains (2 x 128 per sample).
// The products of layers 2 and 3 are a fifth of the kernel's time here, behind the
// FP64 features and the FP32 layers, and M = 16 rows per warp keep a batch of a
// few thousand samples on all SMs, so the wider tcgen05 tiles would gain nothing.
//
// The activations are BF16, so the order of a layer's FP32 sum decides the
// result only where the sum lies within rounding of a BF16 rounding boundary
// (or of zero, for the ReLU).  The definition is the sequential chain
// acc = fma(w_k, a_k, acc), k ascending, plus the bias; the tensor cores sum in
// another order.  Every output whose BF16 value would change within
//   delta = 2^-20 (|w_u|_2 |a|_2 + |b_u|)
// of the tensor-core sum (16 times the rounding unit of a bound on every partial
// sum; about 0.3 % of the outputs) is computed again by the chain itself, so the
// activations are those of the chain and the result does not depend on the
// tensor cores' summation order.
//
// chs_surrogate_decide on 524,288 samples (GB300): 0.36 ms, 5.80 ms with FP32 register
// tiles for all layers and the library's log10; 100 TFLOP/s of 2 x 34,560 flops a
// sample.  Instruction issue bounds it (half of the slots; ALU and FP64 pipes a third
// busy each, tensor pipe 15 %).
// ---------------------------------------------------------------------------

constexpr int kFwdWarps = 14;  // as many as shared memory holds
constexpr int kQueue = 64;      // outputs of a half layer that its lanes share out for the chain
constexpr int kWS = kH + 8;  // padded row of a BF16 matrix in shared memory (ldmatrix without conflicts)
constexpr float kDelta = 9.5367431640625e-07f;  // 2^-20
constexpr int kLogTab = 64;

struct alignas(16) FwdWarp {
    __nv_bfloat16 a[2][16 * kWS];  // activations of one half: layer input and output
    float x[kF][32];
    float y[2][32];
    uint16_t queue[kQueue];        // outputs to compute by the chain: 128 row + unit
};
struct alignas(16) FwdSmem {
    __nv_bfloat16 w2[kH * kWS], w3[kH * kWS];
    float w1[kF][kH];  // transposed
    float w4[kO][kH];
    float b[3][kH], b4[kO];
    float wn[2][kH], bn[2][kH];  // delta's factors |w_u| and |b_u| of layers 2 and 3, times 2^-20
    double2 lt[kLogTab];         // (1 / c, log10(c) / 8), c the middle of a mantissa interval
    FwdWarp warp[kFwdWarps];
};

// log10(s) / 8 for a positive normal s, absolute error below 5e-16: s =
// 2^e m, log10(m) = log10(c) + log10(1 + r) with c from the table and r = m / c -
// 1, |r| <= 2^-7 (Tang, ACM TOMS 16, 1990), six terms of the series.  10 FP64
// instructions against the library's ~30; rounded to FP32 the two differ once in
// a million values.
__device__ __forceinline__ double log10_8(const double s, const double2* __restrict__ lt)
{
    const int hi = __double2hiint(s);
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(s));
    const double2 c = lt[(hi >> 14) & (kLogTab - 1)];
    const double r = fma(m, c.x, -1.0);
    constexpr double q = 0.43429448190325182765 / 8.0;  // log10(e) / 8
    double p = -q / 6.0;
    p = fma(p, r, q / 5.0);
    p = fma(p, r, -q / 4.0);
    p = fma(p, r, q / 3.0);
    p = fma(p, r, -q / 2.0);
    p = fma(p, r, q);
    // the exponent as a double by its bits (2^52 + 2^31 + e, e > -2^31)
    const double e = __hiloint2double(0x43300000, (int)(0x80000000u + (unsigned)((hi >> 20) - 1023))) -
                     (4503599627370496.0 + 2147483648.0);
    return fma(p, r, fma(e, 0.30102999566398119521 / 8.0, c.y));
}

__device__ __forceinline__ void ldmatrix4(unsigned (&r)[4], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}

__device__ __forceinline__ void ldmatrix4_trans(unsigned (&r)[4], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], const unsigned b0, const unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The chain of one output over K = 128 inputs: rows of W and of the activations
// (16-byte aligned), k ascending.
__device__ __forceinline__ float chain128(const __nv_bfloat16* __restrict__ w, const __nv_bfloat16* __restrict__ a)
{
    float acc = 0.0f;
#pragma unroll 4
    for (int k = 0; k < kH; k += 8) {
        const uint4 wv = *reinterpret_cast<const uint4*>(w + k), av = *reinterpret_cast<const uint4*>(a + k);
        const unsigned wu[4] = {wv.x, wv.y, wv.z, wv.w}, au[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc = fmaf(__uint_as_float(wu[i] << 16), __uint_as_float(au[i] << 16), acc);
            acc = fmaf(__uint_as_float(wu[i] & 0xffff0000u), __uint_as_float(au[i] & 0xffff0000u), acc);
        }
    }
    return acc;
}

__device__ __forceinline__ unsigned pack_relu(const float lo, const float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(fmaxf(lo, 0.0f), fmaxf(hi, 0.0f));
    return *reinterpret_cast<const unsigned*>(&v);
}

// The squares of the packed pair added to s (the norm of a row of activations).
__device__ __forceinline__ float add_squares(const unsigned v, float s)
{
    const float lo = __uint_as_float(v << 16), hi = __uint_as_float(v & 0xffff0000u);
    return fmaf(hi, hi, fmaf(lo, lo, s));
}

// |a|_2 of rows g and g + 8 from the quad's partial sums.
__device__ __forceinline__ void row_norms(float (&n2)[2])
{
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        n2[r] += __shfl_xor_sync(0xffffffffu, n2[r], 1);
        n2[r] += __shfl_xor_sync(0xffffffffu, n2[r], 2);
        n2[r] = sqrtf(n2[r]);
    }
}

// Layer 1 on one half (rows = samples 16 half .. + 15 of wp.x): FP32 chains over
// the 12 inputs, outputs where an mma accumulator would have them.
__device__ __forceinline__ void layer1(const FwdSmem& sm, FwdWarp& wp, const int half, float (&norm)[2])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    float xa[kF], xb[kF];
#pragma unroll
    for (int k = 0; k < kF; ++k) {
        xa[k] = wp.x[k][16 * half + g];
        xb[k] = wp.x[k][16 * half + g + 8];
    }
    norm[0] = norm[1] = 0.0f;
#pragma unroll 4
    for (int nt = 0; nt < kH / 8; ++nt) {
        const int u = 8 * nt + 2 * t;
        float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int k = 0; k < kF; ++k) {
            const float2 w = *reinterpret_cast<const float2*>(&sm.w1[k][u]);
            c[0] = fmaf(w.x, xa[k], c[0]);
            c[1] = fmaf(w.y, xa[k], c[1]);
            c[2] = fmaf(w.x, xb[k], c[2]);
            c[3] = fmaf(w.y, xb[k], c[3]);
        }
        const float2 bu = *reinterpret_cast<const float2*>(&sm.b[0][u]);
        const unsigned va = pack_relu(c[0] + bu.x, c[1] + bu.y), vb = pack_relu(c[2] + bu.x, c[3] + bu.y);
        *reinterpret_cast<unsigned*>(&wp.a[0][g * kWS + u]) = va;
        *reinterpret_cast<unsigned*>(&wp.a[0][(g + 8) * kWS + u]) = vb;
        norm[0] = add_squares(va, norm[0]);
        norm[1] = add_squares(vb, norm[1]);
    }
    row_norms(norm);
    __syncwarp();
}

// A hidden layer of 128 x 128 on one half: in -> out (16 rows each), norm the
// row norms of in, replaced by those of out.
__device__ __forceinline__ void layer_mma(const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                                          const float* __restrict__ wn, const float* __restrict__ bn,
                                          const __nv_bfloat16* in, __nv_bfloat16* out, uint16_t* queue,
                                          float (&norm)[2])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    unsigned A[8][4];
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) ldmatrix4(A[ks], in + (lane & 15) * kWS + 16 * ks + 8 * (lane >> 4));
    uint64_t again = 0;  // outputs to compute by the chain, bit 4 nt + e
    float n2[2] = {0.0f, 0.0f};
#pragma unroll 1
    for (int nt = 0; nt < kH / 8; nt += 2) {
        float c[2][4] = {};
        const __nv_bfloat16* wr = W + (8 * nt + (lane & 7)) * kWS + 8 * (lane >> 3);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) {  // two k-steps of 16 per ldmatrix
            unsigned B0[4], B1[4];
            ldmatrix4(B0, wr + 32 * k2);
            ldmatrix4(B1, wr + 8 * kWS + 32 * k2);
            mma_bf16(c[0], A[2 * k2], B0[0], B0[1]);
            mma_bf16(c[1], A[2 * k2], B1[0], B1[1]);
            mma_bf16(c[0], A[2 * k2 + 1], B0[2], B0[3]);
            mma_bf16(c[1], A[2 * k2 + 1], B1[2], B1[3]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int u = 8 * (nt + h) + 2 * t;
            const float2 bu = *reinterpret_cast<const float2*>(bias + u);
            const float2 wu = *reinterpret_cast<const float2*>(wn + u), bb = *reinterpret_cast<const float2*>(bn + u);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float v0 = c[h][2 * r] + bu.x, v1 = c[h][2 * r + 1] + bu.y;
                const float d0 = fmaf(wu.x, norm[r], bb.x), d1 = fmaf(wu.y, norm[r], bb.y);
                const unsigned lo = pack_relu(v0 - d0, v1 - d1), up = pack_relu(v0 + d0, v1 + d1);
                const unsigned diff = lo ^ up;
                again |= (uint64_t)(((diff & 0xffffu) ? 1u : 0u) | ((diff & 0xffff0000u) ? 2u : 0u))
                         << (4 * (nt + h) + 2 * r);
                *reinterpret_cast<unsigned*>(&out[(g + 8 * r) * kWS + u]) = up;
                n2[r] = add_squares(up, n2[r]);
            }
        }
    }
    // The flagged outputs (about six) are shared out over the lanes, so that the warp
    // runs the chain once; where they are more than the queue holds (saturated or
    // non-finite inputs) every lane works off its own.
    const int mine = __popcll(again);
    int before = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, before, off);
        if (lane >= off) before += up;
    }
    const int total = __shfl_sync(0xffffffffu, before, 31);
    before -= mine;
    auto output = [&](const int i) { return 128 * (g + 8 * ((i >> 1) & 1)) + 8 * (i >> 2) + 2 * t + (i & 1); };
    auto chain = [&](const int at) {
        const int row = at >> 7, u = at & 127;
        const float v = chain128(W + u * kWS, in + row * kWS) + bias[u];
        out[row * kWS + u] = __float2bfloat16_rn(fmaxf(v, 0.0f));
    };
    if (total <= kQueue) {
        for (int q = before; again; ++q) {
            queue[q] = (uint16_t)output(__ffsll((long long)again) - 1);
            again &= again - 1;
        }
        __syncwarp();  // the queue and the lanes' outputs are written
        for (int q = lane; q < total; q += 32) chain(queue[q]);
    } else {
        while (again) {
            chain(output(__ffsll((long long)again) - 1));
            again &= again - 1;
        }
    }
    row_norms(n2);
    norm[0] = n2[0];
    norm[1] = n2[1];
    __syncwarp();
}

// One layer's activations of a half to act [128][n]: pairs of samples by
// transposed ldmatrix.
__device__ __forceinline__ void store_act(const __nv_bfloat16* in, __nv_bfloat16* __restrict__ act, const int64_t s0,
                                          const int64_t n)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const bool pair = (n & 1) == 0 && (reinterpret_cast<uintptr_t>(act) & 3) == 0;  // s0 is a multiple of 16
#pragma unroll 1
    for (int u0 = 0; u0 < kH; u0 += 16) {
        unsigned r[4];  // (samples 0-7, units 0-7), (8-15, 0-7), (0-7, 8-15), (8-15, 8-15), transposed
        ldmatrix4_trans(r, in + (lane & 15) * kWS + u0 + 8 * (lane >> 4));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t o = s0 + 8 * (i & 1) + 2 * t;
            __nv_bfloat16* to = act + (int64_t)(u0 + 8 * (i >> 1) + g) * n + o;
            if (pair && o + 1 < n) {
                *reinterpret_cast<unsigned*>(to) = r[i];
            } else {
                const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&r[i]);
                if (o < n) to[0] = v.x;
                if (o + 1 < n) to[1] = v.y;
            }
        }
    }
}

// Forward pass over the features X [12][n] (or, when series != NULL, over the
// features built on the fly); writes Y [2][n] and, when act != NULL, the three
// hidden activations [3][128][n] (BF16) for the backward pass.  With decide:
// orbits whose status is OK take status EARLY_CHAOTIC when sigmoid(y0) >= conf
// and PREDICTED_REGULAR when sigmoid(y0) <= 1 - conf, and t_end is not touched.
template <bool FROM_SERIES>
__global__ void __launch_bounds__(32 * kFwdWarps, 1)
k_mlp_forward(const __nv_bfloat16* __restrict__ P, const float* __restrict__ X, const double* __restrict__ series,
              const int S, const double* __restrict__ ld, const double t, const double* __restrict__ E, const int64_t n,
              float* __restrict__ Y, __nv_bfloat16* __restrict__ act, int32_t* __restrict__ status,
              const double conf, float* __restrict__ prob, const int halves)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FwdSmem& sm = *reinterpret_cast<FwdSmem*>(smem_raw);
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
    // the parameters: weights of layers 2 and 3 as BF16, the others widened
    if ((reinterpret_cast<uintptr_t>(P) & 15) == 0) {  // rows of 256 bytes at multiples of 16
        static_assert(kOffW2 % 8 == 0 && kOffW3 % 8 == 0, "16-byte rows");
#pragma unroll 4
        for (int i = threadIdx.x; i < kH * kH / 8; i += blockDim.x) {
            const int to = (i / (kH / 8)) * kWS + 8 * (i % (kH / 8));
            *reinterpret_cast<uint4*>(sm.w2 + to) = *reinterpret_cast<const uint4*>(P + kOffW2 + 8 * i);
            *reinterpret_cast<uint4*>(sm.w3 + to) = *reinterpret_cast<const uint4*>(P + kOffW3 + 8 * i);
        }
    } else {
        for (int i = threadIdx.x; i < kH * kH; i += blockDim.x) {
            const int u = i / kH, k = i % kH;
            sm.w2[u * kWS + k] = P[kOffW2 + i];
            sm.w3[u * kWS + k] = P[kOffW3 + i];
        }
    }
    for (int i = threadIdx.x; i < kH * kF; i += blockDim.x) sm.w1[i % kF][i / kF] = bf(P[kOffW1 + i]);
    for (int i = threadIdx.x; i < kO * kH; i += blockDim.x) sm.w4[i / kH][i % kH] = bf(P[kOffW4 + i]);
    for (int u = threadIdx.x; u < kH; u += blockDim.x) {
        sm.b[0][u] = bf(P[kOffB1 + u]);
        sm.b[1][u] = bf(P[kOffB2 + u]);
        sm.b[2][u] = bf(P[kOffB3 + u]);
        if (u < kO) sm.b4[u] = bf(P[kOffB4 + u]);
    }
    if (FROM_SERIES && threadIdx.x < kLogTab) {
        const double c = 1.0 + (threadIdx.x + 0.5) / kLogTab;
        sm.lt[threadIdx.x] = make_double2(1.0 / c, log10(c) / 8.0);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * kH; i += blockDim.x) {
        const int l = i / kH, u = i % kH;
        const __nv_bfloat16* w = (l ? sm.w3 : sm.w2) + u * kWS;
        float s = 0.0f;
#pragma unroll 4
        for (int k = 0; k < kH; k += 8) {
            const uint4 v = *reinterpret_cast<const uint4*>(w + k);
            s = add_squares(v.w, add_squares(v.z, add_squares(v.y, add_squares(v.x, s))));
        }
        sm.wn[l][u] = kDelta * sqrtf(s);
        sm.bn[l][u] = kDelta * fabsf(sm.b[1 + l][u]);
    }
    __syncthreads();

    FwdWarp& wp = sm.warp[warp];
    const double rt = 1.0 / t;
    const int rows = 16 * halves;  // samples per tile
    const int64_t tiles = (n + rows - 1) / rows;
    for (int64_t tile = blockIdx.x + (int64_t)gridDim.x * warp; tile < tiles; tile += (int64_t)gridDim.x * kFwdWarps) {
        const int64_t o = tile * rows + lane;  // this lane's sample
        const bool valid = lane < rows && o < n;
        if (FROM_SERIES) {
#pragma unroll 2
            for (int i = 0; i < kS; ++i) {
                double s = (valid && i < S) ? series[(int64_t)i * n + o] : 1e-20;
                s = (s > 1e-20 && isfinite(s)) ? s : 1e-20;
                wp.x[i][lane] = (float)log10_8(s, sm.lt);
            }
            wp.x[10][lane] = valid ? (float)fma(ld[o], rt, -1.0) : 0.0f;
            wp.x[11][lane] = valid ? (float)((E[o] - 0.133) * (1.0 / 0.033)) : 0.0f;
        } else {
#pragma unroll
            for (int k = 0; k < kF; ++k) wp.x[k][lane] = valid ? X[(int64_t)k * n + o] : 0.0f;
        }
        __syncwarp();
#pragma unroll 1
        for (int half = 0; half < halves; ++half) {
            const int64_t s0 = tile * rows + 16 * half;
            float norm[2];
            layer1(sm, wp, half, norm);
            if (act) store_act(wp.a[0], act, s0, n);
            layer_mma(sm.w2, sm.b[1], sm.wn[0], sm.bn[0], wp.a[0], wp.a[1], wp.queue, norm);
            if (act) store_act(wp.a[1], act + (int64_t)kH * n, s0, n);
            layer_mma(sm.w3, sm.b[2], sm.wn[1], sm.bn[1], wp.a[1], wp.a[0], wp.queue, norm);
            if (act) store_act(wp.a[0], act + (int64_t)2 * kH * n, s0, n);
            // layer 4: lane (output, row), the chain over k
            const int row = lane & 15, out = lane >> 4;
            const __nv_bfloat16* a = wp.a[0] + row * kWS;
            const float* w = sm.w4[out];
            float acc = 0.0f;
#pragma unroll 4
            for (int k = 0; k < kH; k += 8) {
                const uint4 av = *reinterpret_cast<const uint4*>(a + k);
                const unsigned au[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc = fmaf(w[k + 2 * i], __uint_as_float(au[i] << 16), acc);
                    acc = fmaf(w[k + 2 * i + 1], __uint_as_float(au[i] & 0xffff0000u), acc);
                }
            }
            wp.y[out][16 * half + row] = acc + sm.b4[out];
            __syncwarp();  // the half's buffers are free
        }
        if (valid) {
            const float y0 = wp.y[0][lane], y1 = wp.y[1][lane];
            if (Y) {
                Y[o] = y0;
                Y[n + o] = y1;
            }
            if (status) {
                const double pc = 1.0 / (1.0 + exp(-(double)y0));
                if (prob) prob[o] = (float)pc;
                if (status[o] == CHS_ORBIT_OK) {
                    if (pc >= conf)
                        status[o] = CHS_ORBIT_EARLY_CHAOTIC;
                    else if (pc <= 1.0 - conf)
                        status[o] = CHS_ORBIT_PREDICTED_REGULAR;
                }
            }
        }
        __syncwarp();  // y and x are read before the next tile writes them
    }
}

// Loss and its gradient w.r.t. the outputs, averaged over n:
//   L = BCE(sigmoid(y0), label) + w_reg (y1 - target)^2,
//   dL/dy0 = (sigmoid(y0) - label) / n,  dL/dy1 = 2 w_reg (y1 - target) / n.
// Returns the sample's loss and writes its gradient.
__device__ __forceinline__ float sample_loss(const float* __restrict__ Y, const float* __restrict__ label,
                                             const float* __restrict__ target, const int64_t n, const int64_t o,
                                             const float w_reg, float* __restrict__ dY)
{
    const float y0 = Y[o], y1 = Y[n + o], lb = label[o], tg = target[o];
    const float p = 1.0f / (1.0f + expf(-y0));
    dY[o] = (p - lb) / (float)n;
    dY[n + o] = 2.0f * w_reg * (y1 - tg) / (float)n;
    // log(1 + exp(-|y|)) form of the cross entropy
    return fmaxf(y0, 0.0f) - y0 * lb + log1pf(expf(-fabsf(y0))) + w_reg * (y1 - tg) * (y1 - tg);
}

__device__ __forceinline__ float warp_sum_f32(float l)
{
    for (int off = 16; off > 0; off >>= 1) l += __shfl_down_sync(0xffffffffu, l, off);
    return l;
}

// loss_out (one float) accumulates the batch loss (atomicAdd; zero it first).
__global__ void k_mlp_loss_grad(const float* __restrict__ Y, const float* __restrict__ label,
                                const float* __restrict__ target, const int64_t n, const float w_reg,
                                float* __restrict__ dY, float* __restrict__ loss_out)
{
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const float l = warp_sum_f32(o < n ? sample_loss(Y, label, target, n, o, w_reg, dY) : 0.0f);
    if ((threadIdx.x & 31) == 0 && o - (threadIdx.x & 31) < n) atomicAdd(loss_out, l / (float)n);
}

// The same for a training batch in one cluster of blocks: no zeroed accumulator (a
// memset launch less) and a loss summed in a fixed order.
constexpr int kLossBlock = 512, kLossCluster = 8;

__global__ void __cluster_dims__(kLossCluster, 1, 1) __launch_bounds__(kLossBlock)
k_mlp_loss_grad_cluster(const float* __restrict__ Y, const float* __restrict__ label,
                        const float* __restrict__ target, const int64_t n, const float w_reg, float* __restrict__ dY,
                        float* __restrict__ loss_out)
{
    __shared__ float part[kLossBlock / 32], total;
    cg::cluster_group cl = cg::this_cluster();
    float l = 0.0f;
    for (int64_t o = (int64_t)cl.block_rank() * kLossBlock + threadIdx.x; o < n; o += kLossCluster * kLossBlock)
        l += sample_loss(Y, label, target, n, o, w_reg, dY);
    l = warp_sum_f32(l);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x / 32] = l;
    __syncthreads();
    if (threadIdx.x < 32) {
        l = warp_sum_f32(threadIdx.x < kLossBlock / 32 ? part[threadIdx.x] : 0.0f);
        if (threadIdx.x == 0) total = l;
    }
    cl.sync();
    if (cl.block_rank() == 0 && threadIdx.x == 0) {
        l = 0.0f;
#pragma unroll
        for (int q = 0; q < kLossCluster; ++q) l += cl.map_shared_rank(&total, q)[0];
        *loss_out = l / (float)n;
    }
    cl.sync();  // no block leaves before its total is read
}

// Back-propagation of one sample tile: from dY [2][n] and the stored
// activations, the pre-activation gradients of every layer:
//   d4 = dY;  d3 = (W4^T d4) * [a3 > 0];  d2 = (W3^T d3) * [a2 > 0];  d1 = (W2^T d2) * [a1 > 0]
// written as FP32 [3][128][n] (d1, d2, d3).  FP32 chains over the units in
// ascending order; a thread owns 4 units x 2 samples, and tiles of 32 samples put a
// batch of 4096 on 128 SMs with 16 warps each.  chs_mlp_backward, batch 4096 (this kernel and k_mlp_wgrad): 43 us; 99 us
// while loads stood inside conditionals and so went out one at a time.
constexpr int kBTile = 32, kBRow = kBTile + 4;  // samples per block; padded row of a gradient tile
constexpr int kBThreads = 512;
struct BwdSmem {
    float w[kH * kH];         // a layer's weights, row = output unit
    float d[2][kH * kBRow];   // the gradient entering a layer and the one leaving it
    float w4[kO][kH];
};

// A layer's BF16 weights widened into shared memory.
__device__ __forceinline__ void stage_weights(const __nv_bfloat16* __restrict__ Wg, float* __restrict__ Ws)
{
    if ((reinterpret_cast<uintptr_t>(Wg) & 15) == 0) {
#pragma unroll
        for (int i = threadIdx.x; i < kH * kH / 8; i += kBThreads) {
            const uint4 v = *reinterpret_cast<const uint4*>(Wg + 8 * i);
            const unsigned p[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; q += 2)
                *reinterpret_cast<float4*>(Ws + 8 * i + 2 * q) =
                    make_float4(__uint_as_float(p[q] << 16), __uint_as_float(p[q] & 0xffff0000u),
                                __uint_as_float(p[q + 1] << 16), __uint_as_float(p[q + 1] & 0xffff0000u));
        }
    } else {
        for (int i = threadIdx.x; i < kH * kH; i += kBThreads) Ws[i] = bf(Wg[i]);
    }
}

__global__ void __launch_bounds__(kBThreads)
k_mlp_backprop(const __nv_bfloat16* __restrict__ P, const __nv_bfloat16* __restrict__ act,
               const float* __restrict__ dY, const int64_t n, float* __restrict__ delta)
{
    extern __shared__ __align__(16) unsigned char bsm[];
    BwdSmem& sm = *reinterpret_cast<BwdSmem*>(bsm);
    constexpr int J = kH * kBTile / kBThreads;  // units of a sample that a thread masks: warp + 16 j
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    const int64_t o = (int64_t)blockIdx.x * kBTile + lane, oc = o < n ? o : n - 1;
    const bool valid = o < n;
    // every activation this thread masks by is on its way before anything waits for one
    __nv_bfloat16 raw[3][J];
#pragma unroll
    for (int l = 2; l >= 0; --l)
#pragma unroll
        for (int j = 0; j < J; ++j) raw[l][j] = act[(int64_t)(l * kH + warp + 16 * j) * n + oc];
    const float y0 = valid ? dY[oc] : 0.0f, y1 = valid ? dY[n + oc] : 0.0f;
    for (int i = threadIdx.x; i < kO * kH; i += kBThreads) sm.w4[i / kH][i % kH] = bf(P[kOffW4 + i]);
    stage_weights(P + kOffW3, sm.w);
    unsigned on[3];  // bit j: activation above zero
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        on[l] = 0;
#pragma unroll
        for (int j = 0; j < J; ++j) on[l] |= (valid && bf(raw[l][j]) > 0.0f) ? 1u << j : 0u;
    }
    __syncthreads();
    // layer 4: d3 = W4^T dY masked by a3 > 0
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int k = warp + 16 * j;
        const float g = (on[2] >> j) & 1u ? sm.w4[0][k] * y0 + sm.w4[1][k] * y1 : 0.0f;
        sm.d[0][k * kBRow + lane] = g;
        if (valid) delta[(int64_t)(2 * kH + k) * n + o] = g;
    }
    // layers 3 and 2: d_{l-1}[k][s] = sum_u W_l[u][k] d_l[u][s], masked by a_{l-1} > 0
    const int tk = lane, ts = warp;  // units 4 tk .. + 3, samples 2 ts, 2 ts + 1
#pragma unroll 1
    for (int l = 0; l < 2; ++l) {
        if (l == 1) stage_weights(P + kOffW2, sm.w);
        __syncthreads();  // the weights and the incoming gradient are complete
        float acc[4][2] = {};
        const float* d = sm.d[l] + 2 * ts;
#pragma unroll 8
        for (int u = 0; u < kH; ++u) {
            const float4 w = *reinterpret_cast<const float4*>(sm.w + u * kH + 4 * tk);
            const float2 dv2 = *reinterpret_cast<const float2*>(d + u * kBRow);
            const float wv[4] = {w.x, w.y, w.z, w.w}, dv[2] = {dv2.x, dv2.y};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) acc[a][b] = fmaf(wv[a], dv[b], acc[a][b]);
        }
        // through shared memory (the tile this layer does not read), so that rows of samples leave together
        float* out = sm.d[1 - l];
#pragma unroll
        for (int a = 0; a < 4; ++a)
            *reinterpret_cast<float2*>(out + (4 * tk + a) * kBRow + 2 * ts) = make_float2(acc[a][0], acc[a][1]);
        __syncthreads();  // out is complete, the weights are free
        const int ai = 1 - l;  // activation a_{l-1}: layer 3 -> a2 (1), layer 2 -> a1 (0)
        const unsigned m = ai ? on[1] : on[0];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int k = warp + 16 * j;
            const float g = (m >> j) & 1u ? out[k * kBRow + lane] : 0.0f;
            out[k * kBRow + lane] = g;
            if (valid) delta[(int64_t)(ai * kH + k) * n + o] = g;
        }
    }
}

// Weight and bias gradients as batch reductions:
//   dW_l[u][k] = sum_s d_l[u][s] a_{l-1}[k][s],  db_l[u] = sum_s d_l[u][s]
// with a_0 = X, d_4 = dY.  A cluster of kSplit blocks (132 blocks in all, one wave)
// works one 32 x 64 tile of one
// layer's dW, each block a contiguous part of the batch, and the blocks' partial
// sums are joined through distributed shared memory in a fixed order (the sums do
// not depend on the run).  A single block per tile walked the batch alone: 40
// blocks for 152 SMs (a training step of batch 4096 took 394 us, 68 us now).
constexpr int kSplit = 6, kWU = 32, kWK = 64, kWS_ = 64;  // blocks per tile, tile, samples per chunk
constexpr int kWThreads = 256;  // two groups of 128, each half of a chunk's samples
constexpr int kWTiles = 4 + 2 * (kH / kWU) * (kH / kWK) + kH / kWK;  // layers 1; 2 and 3; 4

__global__ void __cluster_dims__(kSplit, 1, 1) __launch_bounds__(kWThreads)
k_mlp_wgrad(const float* __restrict__ X, const __nv_bfloat16* __restrict__ act, const float* __restrict__ delta,
            const float* __restrict__ dY, const int64_t n, float* __restrict__ G)
{
    __shared__ __align__(16) float Ds[kWS_][kWU + 4], As[kWS_][kWK + 4];
    __shared__ float part[2][kWU][kWK];  // the groups' sums
    __shared__ float bias[2][kWU];       // of the chunks' first and second 32 samples
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int b = blockIdx.x / kSplit;
    int layer, ut, kt;
    constexpr int per = (kH / kWU) * (kH / kWK);
    if (b < 4) { layer = 1; ut = b; kt = 0; }
    else if (b < 4 + 2 * per) { layer = 2 + (b - 4) / per; ut = (b - 4) % per / (kH / kWK); kt = (b - 4) % (kH / kWK); }
    else { layer = 4; ut = 0; kt = b - 4 - 2 * per; }
    const int U = layer == 4 ? kO : kH, K = layer == 1 ? kF : kH;
    const float* d = layer == 4 ? dY : delta + (int64_t)(layer - 1) * kH * n;
    const __nv_bfloat16* av = act + (int64_t)(layer > 1 ? layer - 2 : 0) * kH * n;  // layers 2 .. 4
    // chunks of samples, a contiguous range of them per block
    const int64_t chunks = (n + kWS_ - 1) / kWS_, each = (chunks + kSplit - 1) / kSplit;
    const int64_t c0 = rank * each, c1 = min(chunks, c0 + each);
    const int sl = threadIdx.x % kWS_, row = threadIdx.x / kWS_;  // sample and first row (of every 4th) to load
    const int grp = threadIdx.x / 128, tu = threadIdx.x % 128 / 16, tk = threadIdx.x % 16;
    float acc[4][4] = {}, accb[kWU / 4] = {};
    // the next chunk's loads (rows row + 4 i, sample sl), raw and unconditional at clamped indices, so
    // that all of them are in flight at once; what lies outside is zeroed on the way to shared memory
    float rd[kWU / 4], rx[kWK / 4];
    __nv_bfloat16 ra[kWK / 4];
    bool in = false;
    auto fetch = [&](const int64_t c) {
        const int64_t o = c * kWS_ + sl, oc = o < n ? o : n - 1;
        in = o < n;
#pragma unroll
        for (int i = 0; i < kWU / 4; ++i) {
            const int u = ut * kWU + row + 4 * i;
            rd[i] = d[(int64_t)(u < U ? u : U - 1) * n + oc];
        }
        if (layer == 1) {
#pragma unroll
            for (int i = 0; i < kWK / 4; ++i) {
                const int k = row + 4 * i;
                rx[i] = X[(int64_t)(k < K ? k : K - 1) * n + oc];
            }
        } else {
#pragma unroll
            for (int i = 0; i < kWK / 4; ++i) ra[i] = av[(int64_t)(kt * kWK + row + 4 * i) * n + oc];
        }
    };
    if (c0 < c1) fetch(c0);
    for (int64_t c = c0; c < c1; ++c) {
#pragma unroll
        for (int i = 0; i < kWU / 4; ++i) {
            const float v = (in && ut * kWU + row + 4 * i < U) ? rd[i] : 0.0f;
            Ds[sl][row + 4 * i] = v;
            accb[i] += v;
        }
#pragma unroll
        for (int i = 0; i < kWK / 4; ++i)
            As[sl][row + 4 * i] = !in ? 0.0f : layer != 1 ? bf(ra[i]) : row + 4 * i < K ? rx[i] : 0.0f;
        __syncthreads();
        if (c + 1 < c1) fetch(c + 1);
#pragma unroll 8
        for (int s = 0; s < kWS_ / 2; ++s) {
            const float4 dv = *reinterpret_cast<const float4*>(&Ds[2 * s + grp][4 * tu]);
            const float4 kv = *reinterpret_cast<const float4*>(&As[2 * s + grp][4 * tk]);
            const float dd[4] = {dv.x, dv.y, dv.z, dv.w}, kk[4] = {kv.x, kv.y, kv.z, kv.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(dd[i], kk[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) part[grp][4 * tu + i][4 * tk + j] = acc[i][j];
#pragma unroll
    for (int i = 0; i < kWU / 4; ++i) {  // a warp holds 32 samples of a row
        const float v = warp_sum_f32(accb[i]);
        if (sl % 32 == 0) bias[sl / 32][row + 4 * i] = v;
    }
    cl.sync();
    // the cluster's blocks share out the tile's sums and join each over the blocks, in order
    const int offW = layer == 1 ? kOffW1 : layer == 2 ? kOffW2 : layer == 3 ? kOffW3 : kOffW4;
    const int offB = layer == 1 ? kOffB1 : layer == 2 ? kOffB2 : layer == 3 ? kOffB3 : kOffB4;
    for (int i = rank * kWThreads + threadIdx.x; i < kWU * (kWK + 1); i += kSplit * kWThreads) {
        const bool weight = i < kWU * kWK;
        const int r = weight ? i / kWK : i - kWU * kWK, c = weight ? i % kWK : 0;
        const int u = ut * kWU + r, k = kt * kWK + c;
        float* p0 = weight ? &part[0][r][c] : &bias[0][r];
        float* p1 = weight ? &part[1][r][c] : &bias[1][r];
        float sum = 0.0f;
#pragma unroll
        for (int q = 0; q < kSplit; ++q) sum += cl.map_shared_rank(p0, q)[0] + cl.map_shared_rank(p1, q)[0];
        if (u < U && weight && k < K) G[offW + u * K + k] = sum;
        if (u < U && !weight && kt == 0) G[offB + u] = sum;
    }
    cl.sync();  // no block leaves while another reads its part
}

// Adam on FP32 master weights; writes the BF16 copy used by the kernels.
__global__ void k_mlp_adam(float* __restrict__ W, float* __restrict__ m, float* __restrict__ v,
                           const float* __restrict__ g, const int64_t P, const float lr, const float b1,
                           const float b2, const float eps, const float c1, const float c2,
                           __nv_bfloat16* __restrict__ Wb)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float w = W[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    W[i] = w;
    Wb[i] = __float2bfloat16_rn(w);
}

// ---------------------------------------------------------------------------

static_assert(sizeof(FwdSmem) <= 227 * 1024, "the forward kernel's shared memory");

static int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        sms = 1;
    return sms;
}

// Launches the forward kernel: tiles of 16 samples while tiles of 32 would give
// each SM fewer than four, and never more blocks than tiles.
template <bool FROM_SERIES>
static cudaError_t forward(const __nv_bfloat16* P, const float* X, const double* series, int S, const double* ld,
                           double t, const double* E, int64_t n, float* Y, __nv_bfloat16* act, int32_t* status,
                           double conf, float* prob, cudaStream_t st)
{
    cudaError_t e = cudaFuncSetAttribute(k_mlp_forward<FROM_SERIES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(FwdSmem));
    if (e != cudaSuccess) return e;
    const int sms = sm_count(), halves = n < (int64_t)4 * 32 * sms ? 1 : 2;
    const int64_t tiles = (n + 16 * halves - 1) / (16 * halves);
    k_mlp_forward<FROM_SERIES><<<(unsigned)(tiles < sms ? tiles : sms), 32 * kFwdWarps, sizeof(FwdSmem), st>>>(
        P, X, series, S, ld, t, E, n, Y, act, status, conf, prob, halves);
    return cudaGetLastError();
}

cudaError_t launch_mlp_features(const double* series, int S, const double* ld, double t, const double* E,
                                int64_t n, float* X, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    k_mlp_features<<<blocks_for(n, 256), 256, 0, st>>>(series, S, ld, t, E, n, X);
    return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const void* P, const float* X, int64_t n, float* Y, void* act,
                               cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    return forward<false>(static_cast<const __nv_bfloat16*>(P), X, nullptr, 0, nullptr, 1.0, nullptr, n, Y,
                          static_cast<__nv_bfloat16*>(act), nullptr, 0.0, nullptr, st);
}

cudaError_t launch_mlp_decide(const void* P, const double* series, int S, const double* ld, double t,
                              const double* E, int64_t n, double conf, int32_t* status, float* prob,
                              cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    return forward<true>(static_cast<const __nv_bfloat16*>(P), nullptr, series, S, ld, t, E, n, nullptr, nullptr,
                         status, conf, prob, st);
}

// Largest batch whose loss one cluster sums: up to there the call takes 8.6 to 9.2 us,
// the host's part of it; a single block took 16.5 us at 16,384.
constexpr int64_t kLossOneCluster = 32768;

cudaError_t launch_mlp_loss_grad(const float* Y, const float* label, const float* target, int64_t n,
                                 float w_reg, float* dY, float* loss, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    if (n <= kLossOneCluster) {
        k_mlp_loss_grad_cluster<<<kLossCluster, kLossBlock, 0, st>>>(Y, label, target, n, w_reg, dY, loss);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(loss, 0, sizeof(float), st);
    if (e != cudaSuccess) return e;
    k_mlp_loss_grad<<<blocks_for(n, 256), 256, 0, st>>>(Y, label, target, n, w_reg, dY, loss);
    return cudaGetLastError();
}

cudaError_t launch_mlp_backward(const void* P, const float* X, const void* act, const float* dY,
                                int64_t n, float* delta, float* G, cudaStream_t st)
{
    if (n == 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_mlp_backprop, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(BwdSmem));
    if (e != cudaSuccess) return e;
    k_mlp_backprop<<<blocks_for(n, kBTile), kBThreads, sizeof(BwdSmem), st>>>(
        static_cast<const __nv_bfloat16*>(P), static_cast<const __nv_bfloat16*>(act), dY, n, delta);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_mlp_wgrad<<<kWTiles * kSplit, kWThreads, 0, st>>>(X, static_cast<const __nv_bfloat16*>(act), delta, dY, n, G);
    return cudaGetLastError();
}

cudaError_t launch_mlp_adam(float* W, float* m, float* v, const float* g, float lr, float b1, float b2,
                            float eps, int step, void* Wb, cudaStream_t st)
{
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    k_mlp_adam<<<blocks_for(kParams, 256), 256, 0, st>>>(W, m, v, g, kParams, lr, b1, b2, eps, c1, c2,
                                                         static_cast<__nv_bfloat16*>(Wb));
    return cudaGetLastError();
}

}  // namespace chs
