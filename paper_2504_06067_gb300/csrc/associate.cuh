// associate.cuh -- the exact distance of the association (Eq. 2), shared by
// its kernels (k_associate.cu) and the one-cluster generation (k_small.cu).
#pragma once
#include "common.cuh"

namespace {

// Perpendicular distance of f' (norm nf) to direction Zj (norm nzj), FP64,
// one rounded operation after the other as a plain CPU evaluation.
__device__ __forceinline__ double perp_dist(const double* fp, double nf, const double* Zj, double nzj,
                                            int m)
{
    if (nf == 0.0) return 0.0;
    double dot = 0.0;
    for (int q = 0; q < m; ++q) dot = __dadd_rn(dot, __dmul_rn(fp[q], Zj[q]));
    const double den = __dmul_rn(nf, nzj);
    const double cth = __ddiv_rn(dot, den);
    double one_m = __dsub_rn(1.0, __dmul_rn(cth, cth));
    if (one_m < 0.0) one_m = 0.0;
    return __dmul_rn(nf, __dsqrt_rn(one_m));
}

}  // namespace
