// associate.cuh -- the exact distance of the association (Eq. 2), shared by
// its kernels (k_associate.cu) and the one-cluster generation (k_small.cu).
#pragma once
#include "common.cuh"
#include "sf64.cuh"

namespace {

// Perpendicular distance of f' (norm nf) to direction Zj (norm nzj), FP64,
// one rounded operation after the other as a plain CPU evaluation (the
// quotient and the square root on the integer pipes: the same values).
__device__ __forceinline__ double perp_dist(const double* fp, double nf, const double* Zj, double nzj, int m)
{
    if (sf64::is_zero(nf)) return 0.0;
    double dot = 0.0;
    for (int q = 0; q < m; ++q) dot = __dadd_rn(dot, __dmul_rn(fp[q], Zj[q]));
    const double den = __dmul_rn(nf, nzj);
    const double cth = sf64::div(dot, den);
    double one_m = __dsub_rn(1.0, __dmul_rn(cth, cth));
    if (sf64::is_negative(one_m)) one_m = 0.0;
    return __dmul_rn(nf, sf64::sqrt_rn(one_m));
}

// FP32 unit vector of f' = (f - z) / a without FP64 (z* and f are FP32
// values; ia = 1 / a in FP32, two roundings).  Each component is within
// 6 2^-24 of the exact one relative to it, up to one factor common to all
// (the norm), which no comparison of cosines sees: cosines with an FP32
// direction (2^-24) summed by m FMAs of non-negative terms are within
// (m + 7) 2^-24 of the exact ones.  False, with u untouched, when a factor
// or the norm leaves the range in which those bounds hold (tiny or huge
// objectives: the caller takes the FP64 form).
template <int M>
__device__ __forceinline__ bool unit32(const float* f, const float* z, const float* ia, float* u)
{
    float x[M], s = 0.0f;
    bool ok = true;
#pragma unroll
    for (int q = 0; q < M; ++q) {
        x[q] = __fmul_rn(__fsub_rn(f[q], z[q]), ia[q]);
        s = fmaf(x[q], x[q], s);
        ok = ok && ia[q] >= 1e-30f && ia[q] <= 1e30f;
    }
    if (!ok || !(s >= 1e-25f && s <= 1e25f)) return false;
    const float n = rsqrtf(s);
#pragma unroll
    for (int q = 0; q < M; ++q) u[q] = __fmul_rn(x[q], n);
    return true;
}

// A direction whose FP32 cosine with unit32's vector (or the FP64 form's) is
// more than this below the best one cannot be the nearest, nor tie.
template <int M>
__device__ __forceinline__ constexpr float cos_band()
{
    return 2.0f * (float)(M + 7) * 5.9604644775390625e-08f + 1e-12f;
}

}  // namespace
