// normalize.cuh -- device functions of the normalization step shared by its
// kernels (k_normalize.cu) and the one-cluster generation (k_small.cu).
#pragma once
#include "common.cuh"
#include "sf64.cuh"

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

// Whether the largest f~ = f - z* of an objective over T (as its key) says that
// some member of T, or the ideal point, is not finite: an infinity or a NaN
// there leaves one in f~, whose key is no finite value's.  The cosines of such
// a member are NaN, so it has no nearest direction: the selection ends with
// DEV_ENONFINITE before the association.
__device__ __forceinline__ bool not_finite_key(unsigned long long k) { return k >= 0x7ff0000000000000ull; }

// The quotients of a chain that runs once: one copy of the code (below).
__device__ __noinline__ double div_once(double a, double b) { return sf64::div(a, b); }

// Gaussian elimination with partial pivoting (first maximal |pivot|) on
// E b = 1, a = 1 / b, by one warp; m <= 32.  A: m rows of m + 1 values in
// shared memory, [E - z* | 1], overwritten.  Every element sees the same _rn
// operations in the same order as a serial elimination (factor = A_rc / A_cc,
// A_rk -= factor * A_ck for k > c, rhs_r -= factor * rhs_c; back substitution
// from the last unknown, each row's known terms subtracted from the highest
// column down).  `ok` false: no valid system.  Returns whether every
// intercept is usable, with lane r's in a.
// A chain that runs once per selection: what it costs is latency and fetching
// instructions, so the loops are not unrolled (a register form unrolled for
// each m took 8,300 cycles at m = 3 and, with row swaps, 25,000 at m = 8),
// pivots are compared as integers (|x| orders like its bits; an FP64 compare
// takes 110 cycles) and quotients formed on the integer pipes (sf64.cuh).
__device__ __noinline__ bool solve_rows(int m, double* A, bool ok, double& a)
{
    const int lane = lane_id(), ld = m + 1;
    a = 0.0;
    __syncwarp();
#pragma unroll 1
    for (int col = 0; col < m; ++col) {
        if (!ok) break;
        // pivot: first row >= col of maximal |A[.][col]| (rows in current order)
        const bool cand = lane >= col && lane < m;
        const unsigned long long k = cand ? sf64::bits(A[lane * ld + col]) << 1 : 0ull;  // |x|, twice
        const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(k >> 32));
        const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(k >> 32) == hi ? (uint32_t)k : 0u);
        if ((hi | lo) == 0u) {
            ok = false;
            break;
        }
        const unsigned who = __ballot_sync(0xffffffffu, cand && k == (((unsigned long long)hi << 32) | lo));
        const int p = __ffs(who) - 1;
        if (p != col) {  // swap rows col and p
#pragma unroll 1
            for (int q = col + lane; q <= m; q += 32) {
                const double x = A[col * ld + q];
                A[col * ld + q] = A[p * ld + q];
                A[p * ld + q] = x;
            }
            __syncwarp();
        }
        double f = 0.0;
        if (lane > col && lane < m) f = div_once(A[lane * ld + col], A[col * ld + col]);
        __syncwarp();
        // rows below, columns after col and the right side: a lane per element
        const int nq = m - col, ne = (m - 1 - col) * nq;
        const unsigned inv = 65536u / (unsigned)nq + 1u;  // e / nq = (e inv) >> 16 for e nq < 65,536
#pragma unroll 1
        for (int e0 = 0; e0 < ne; e0 += 32) {
            const int e = e0 + lane, dr = (int)(((unsigned)e * inv) >> 16);
            const int r = col + 1 + dr, q = col + 1 + e - dr * nq;
            const double fr = __shfl_sync(0xffffffffu, f, r & 31);
            if (e < ne) A[r * ld + q] = __dsub_rn(A[r * ld + q], __dmul_rn(fr, A[col * ld + q]));
        }
        __syncwarp();
    }
    if (ok) {
        // back substitution column by column from the last unknown: every
        // lane subtracts A_ir b_r as soon as b_r is known, so row i meets its
        // terms from the highest column down, as the serial loop does
        const int row = lane < m ? lane : 0;
        const double* Ar = A + row * ld;
        const sf64::Divisor dd = sf64::divisor(Ar[row]);
        double rhs = Ar[m], b = 0.0;  // lane r ends with b_r
#pragma unroll 1
        for (int r = m - 1; r >= 0; --r) {
            const double br = __shfl_sync(0xffffffffu, sf64::div(rhs, dd), r);
            if (lane == r) b = br;
            if (lane < r) rhs = __dsub_rn(rhs, __dmul_rn(Ar[r], br));
        }
        a = lane < m ? div_once(1.0, b) : 1.0;
        // not finite, or <= 1e-6: positive doubles order like their bits
        const unsigned long long ab = sf64::bits(a);
        const bool bad = lane < m && (ab >= 0x7ff0000000000000ull || ab <= sf64::bits(1e-6));
        if (__any_sync(0xffffffffu, bad)) ok = false;
    }
    return ok;
}

}  // namespace
