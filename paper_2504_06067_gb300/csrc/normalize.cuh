// normalize.cuh -- device functions of the normalization step shared by its
// kernels (k_normalize.cu) and the one-cluster generation (k_small.cu).
#pragma once
#include "common.cuh"

namespace {

// Non-negative doubles order like their bit patterns; -0.0 is mapped to
// +0.0 so that the two zeros compare equal, as IEEE comparisons do.
__device__ __forceinline__ unsigned long long okey(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b << 1) == 0ull ? 0ull : b;  // integer test for +-0 (FP64 compares are slow)
}

__device__ __forceinline__ bool key_less(unsigned long long a, int ia, unsigned long long b, int ib)
{
    return a < b || (a == b && ia < ib);
}

// Gaussian elimination with partial pivoting (first maximal |pivot|) on
// E b = 1, a = 1 / b.  One warp: lane r holds row r of the
// (row-swapped) system, so each elimination step updates every row at once;
// every element sees the same _rn operations in the same order as a serial
// elimination (factor = A_rc / A_cc, A_rk -= factor * A_ck for k >= c,
// rhs_r -= factor * rhs_c; back substitution from the last unknown, each
// row's known terms subtracted from the highest column down).
// M <= NSGA3_FAST_M: m = M; M = NSGA3_WARP_M: any m <= 32 at run time
// (rows and columns >= m are never touched).  `ok` false: no valid system.
// Returns whether every intercept is usable, with lane r's in a.
template <int M>
__device__ __forceinline__ bool solve_rows(int m, double (&A)[M], bool ok, double& a)
{
    const int lane = lane_id();
    double rhs = 1.0;
#pragma unroll
    for (int col = 0; col < M; ++col) {
        if (!ok || col >= m) break;
        // pivot: first row >= col of maximal |A[.][col]| (rows in current order)
        int p = col;
        double best = fabs(__shfl_sync(0xffffffffu, A[col], col));
#pragma unroll
        for (int r = col + 1; r < M; ++r) {
            const double x = fabs(__shfl_sync(0xffffffffu, A[col], r));
            if (r < m && x > best) {
                best = x;
                p = r;
            }
        }
        if (best == 0.0) {
            ok = false;
            break;
        }
        if (p != col) {  // swap rows col and p
#pragma unroll
            for (int q = 0; q < M; ++q) {
                const double a_c = __shfl_sync(0xffffffffu, A[q], col);
                const double a_p = __shfl_sync(0xffffffffu, A[q], p);
                if (lane == col) A[q] = a_p;
                if (lane == p) A[q] = a_c;
            }
            const double r_c = __shfl_sync(0xffffffffu, rhs, col);
            const double r_p = __shfl_sync(0xffffffffu, rhs, p);
            if (lane == col) rhs = r_p;
            if (lane == p) rhs = r_c;
        }
        double piv[M];
#pragma unroll
        for (int q = 0; q < M; ++q) piv[q] = __shfl_sync(0xffffffffu, A[q], col);
        const double prhs = __shfl_sync(0xffffffffu, rhs, col);
        if (lane > col && lane < m) {
            const double factor = __ddiv_rn(A[col], piv[col]);
#pragma unroll
            for (int q = col; q < M; ++q)
                if (q < m) A[q] = __dsub_rn(A[q], __dmul_rn(factor, piv[q]));
            rhs = __dsub_rn(rhs, __dmul_rn(factor, prhs));
        }
    }
    a = 0.0;
    if (ok) {
        // back substitution column by column from the last unknown: every
        // lane subtracts A_ir b_r as soon as b_r is known, so row i meets its
        // terms from the highest column down, as the serial loop does
        double b = 0.0;  // lane r ends with b_r
#pragma unroll
        for (int r = M - 1; r >= 0; --r) {
            if (r >= m) continue;
            const double br = __shfl_sync(0xffffffffu, lane == r ? __ddiv_rn(rhs, A[r]) : 0.0, r);
            if (lane == r) b = br;
            if (lane < r) rhs = __dsub_rn(rhs, __dmul_rn(A[r], br));
        }
        a = lane < m ? __ddiv_rn(1.0, b) : 1.0;
        const bool bad = lane < m && (!isfinite(a) || a <= 1e-6);
        if (__any_sync(0xffffffffu, bad)) ok = false;
    }
    return ok;
}

}  // namespace
