// gs_narrow.cuh -- the modified Gram-Schmidt of the FPUT Lyapunov kernels where a
// warp has few columns left.
//
// In the "dot products first" order a warp owns 32 columns, one per lane, and at
// pivot j only the columns from j on have work; an idle lane costs an FP64 slot.
// Once at most WD = 16 (8) of its columns are left the warp therefore takes its
// rows in 32 / WD parts side by side, lane = part * WD + column, instead of letting
// half (three quarters) of its lanes idle through all of them; the parts of a dot
// product are joined by a butterfly, which gives the same sum in every part.  At d =
// 128, N = 64, QR every 10, 256 threads: 921 -> 861 us per step of 1064 orbits, the
// pivot's reciprocal (rcp_full) included.
#pragma once

#include "fastmath.cuh"

namespace chs {
namespace gs {

// w_j . w_c over ROWS rows (element (r, c) at W[r * RS + c * CS]) for c = c0 + lane %
// WD, the same in every part.  Every lane of the warp calls it.
template <int ROWS, int WD, int RS, int CS>
__device__ __forceinline__ double narrow_dot(const double* __restrict__ W, const int j, const int c0, const int lane)
{
    constexpr int PART = ROWS * WD / 32;  // rows per part
    const double* a = W + (lane / WD * PART) * RS;
    const int c = c0 + lane % WD;
    double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
    for (int i = 0; i < PART; i += 2) {
        s0 = fma(a[i * RS + j * CS], a[i * RS + c * CS], s0);
        s1 = fma(a[(i + 1) * RS + j * CS], a[(i + 1) * RS + c * CS], s1);
    }
    double s = s0 + s1;
#pragma unroll
    for (int off = WD; off < 32; off <<= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return s;
}

// w_c += f w_j on the same rows for the columns c > j.
template <int ROWS, int WD, int RS, int CS>
__device__ __forceinline__ void narrow_axpy(double* __restrict__ W, const int j, const int c0, const int lane,
                                            const double f)
{
    constexpr int PART = ROWS * WD / 32;
    double* a = W + (lane / WD * PART) * RS;
    const int c = c0 + lane % WD;
#pragma unroll 4
    for (int i = 0; i < PART; ++i) {
        const double v = fma(f, a[i * RS + j * CS], a[i * RS + c * CS]);
        if (c > j) a[i * RS + c * CS] = v;
    }
}

// The whole Gram-Schmidt of a D x D matrix by D threads (D = 32 or 64: one or two
// warps; thread l owns column l), without the final normalisation: returns the
// squared norm of column l.  nj: a shared double.  Every thread of the block calls
// it, with `mine` saying whether its orbit takes part (the same in a warp).
template <int D, int RS, int CS>
__device__ __forceinline__ double columns_mgs(double* W, double* nj, const int l, const bool mine)
{
    static_assert(D % 32 == 0, "whole warps of columns");
    const int lane = l % 32, c0 = l - lane;
    double n2 = 1.0;
    for (int j = 0; j < D; ++j) {
        const int left = mine ? c0 + 32 - j : 0;  // columns of this warp that are left (warp-uniform)
        double r = 0.0;
        if (left > 16) {
            if (l >= j) {
                double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
                for (int i = 0; i < D; i += 2) {
                    s0 = fma(W[i * RS + j * CS], W[i * RS + l * CS], s0);
                    s1 = fma(W[(i + 1) * RS + j * CS], W[(i + 1) * RS + l * CS], s1);
                }
                r = s0 + s1;
            }
            if (l == j) *nj = r;
        } else if (left > 8) {
            r = narrow_dot<D, 16, RS, CS>(W, j, c0 + 16, lane);
            if (c0 + 16 + lane == j) *nj = r;
        } else if (left > 0) {
            r = narrow_dot<D, 8, RS, CS>(W, j, c0 + 24, lane);
            if (c0 + 24 + lane == j) *nj = r;
        }
        __syncthreads();
        if (left > 0) {
            const double norm = *nj, f = -r * rcp_full(norm);
            if (l == j) n2 = norm;
            if (left > 16) {
                if (l > j) {
#pragma unroll 4
                    for (int i = 0; i < D; ++i) W[i * RS + l * CS] = fma(f, W[i * RS + j * CS], W[i * RS + l * CS]);
                }
            } else if (left > 8) {
                narrow_axpy<D, 16, RS, CS>(W, j, c0 + 16, lane, f);
            } else {
                narrow_axpy<D, 8, RS, CS>(W, j, c0 + 24, lane, f);
            }
        }
        __syncthreads();
    }
    return n2;
}

}  // namespace gs
}  // namespace chs
