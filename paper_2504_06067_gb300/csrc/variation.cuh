// variation.cuh -- device functions of the variation (Alg. 1, crossover and
// mutation) and of the softmax-simplex objective, used by the variation
// kernels (k_problem.cu) and the one-cluster generation (k_small.cu).
#pragma once
#include "common.cuh"

namespace {

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Bounded polynomial mutation (Deb and Goyal): y + dq with
// dq = val^(1/(eta+1)) - 1 (lower branch) or 1 - val^(1/(eta+1)) (upper
// branch).  val^e - 1 is formed as expm1(e log val), which keeps dq
// accurate relative to itself; pow(val, e) - 1 would lose the bits of dq
// below the ulp of 1 when val is near 1.
__device__ __forceinline__ float pm_mutate(float y, float u, float eta_m)
{
    const float mp = 1.0f / (eta_m + 1.0f);
    // one powf, logf and expm1f on the chosen branch's operands (the same
    // values as calling them in each branch)
    const bool lo = u < 0.5f;
    const float xy = lo ? 1.0f - y : 1.0f - (1.0f - y);
    const float pw = powf(xy, eta_m + 1.0f);
    const float val = lo ? 2.0f * u + (1.0f - 2.0f * u) * pw : 2.0f * (1.0f - u) + 2.0f * (u - 0.5f) * pw;
    const float ex = expm1f(mp * logf(val));
    const float dq = lo ? ex : -ex;
    y = y + dq;
    return fminf(fmaxf(y, 0.0f), 1.0f);
}

// The pair's share of the state that the end of the generation overwrites:
// rows of the merged individuals and the parents' objectives.
__device__ __forceinline__ void merge_pair(const RunView& v, int q)
{
    const int lane = lane_id();
    if (lane < 2) {
        v.pold[2 * q + lane] = v.pcan[2 * q + lane];
        v.cslot[2 * q + lane] = v.fslot[2 * q + lane];
    }
    for (int e = lane; e < 2 * v.m; e += 32) v.F[(size_t)2 * q * v.m + e] = v.PF[(size_t)2 * q * v.m + e];
}

// Variation of one pair (one warp, lanes over the variables): binary
// tournament on rank (first drawn wins ties), SBX with per-variable
// crossover and child swap, polynomial mutation, clip to [0, 1].  Calls
// out(var, c1, c2) for every variable in lane order var = lane + 32 t (from
// v0 on and every `step`-th only, when several warps share the pair).
// SBX is written c1,2 = (y1 + y2)/2 -/+ (beta/2)(y2 - y1) with one FMA, the
// same value as ((1 + beta) y1 + (1 - beta) y2)/2 with fewer roundings.
// ROLL: one copy of the mutation's code for both children (a chain that runs
// once is bound by instruction fetch; a kernel that fills the GPU by issue: 8 %
// more instructions, 97 us instead of 92 at N = 50,000, d = 200).
template <bool ROLL, class Out>
__device__ __forceinline__ void vary_pair(const RunView& v, int q, uint32_t gen, Out out, int v0 = 0, int step = 32)
{
    const int lane = lane_id();
    const int N = v.N, d = v.d;
    // the pair's two blocks by odd and even lanes at once
    const U4 t = philox((uint32_t)q, gen, RNG_TOURNAMENT, (uint32_t)lane & 1u, v.seed);
    const uint32_t a1 = bounded(__shfl_sync(0xffffffffu, t.x, 0), N), b1 = bounded(__shfl_sync(0xffffffffu, t.y, 0), N);
    const uint32_t a2 = bounded(__shfl_sync(0xffffffffu, t.z, 0), N), b2 = bounded(__shfl_sync(0xffffffffu, t.w, 0), N);
    const uint32_t cx = __shfl_sync(0xffffffffu, t.x, 1);
    // the rows of all four drawn parents are read beside their ranks
    const int ra1 = v.pcan[a1], rb1 = v.pcan[b1], ra2 = v.pcan[a2], rb2 = v.pcan[b2];
    const size_t p1 = v.rank[b1] < v.rank[a1] ? rb1 : ra1;
    const size_t p2 = v.rank[b2] < v.rank[a2] ? rb2 : ra2;
    const bool cross = u01(cx) < v.p_c;
    const float e = 1.0f / (v.eta_c + 1.0f);
    for (int var = v0 + lane; var < d; var += step) {
        const float y1 = v.X[p1 * d + var], y2 = v.X[p2 * d + var];
        float c1 = y1, c2 = y2;
        const U4 sb = philox((uint32_t)q * (uint32_t)d + (uint32_t)var, gen, RNG_SBX, 0u, v.seed);
        if (cross && u01(sb.y) < 0.5f) {
            const float u = u01(sb.x);
            // one powf on the chosen base (the same value as either branch's call)
            const float base = (u <= 0.5f) ? 2.0f * u : 1.0f / (2.0f * (1.0f - u));
            const float beta = powf(base, e);
            const float mid = 0.5f * (y1 + y2), hb = 0.5f * beta, dy = y2 - y1;
            c1 = fmaf(-hb, dy, mid);
            c2 = fmaf(hb, dy, mid);
            if (u01(sb.z) < 0.5f) {
                const float tmp = c1;
                c1 = c2;
                c2 = tmp;
            }
            c1 = fminf(fmaxf(c1, 0.0f), 1.0f);
            c2 = fminf(fmaxf(c2, 0.0f), 1.0f);
        }
        const bool mut0 = u01(sb.w) < v.p_m;
        const U4 pm = philox((uint32_t)q * (uint32_t)d + (uint32_t)var, gen, RNG_PM, 0u, v.seed);
        const bool mut1 = u01(pm.y) < v.p_m;
        if constexpr (ROLL) {
#pragma unroll 1
            for (int h = 0; h < 2; ++h)
                if (h ? mut1 : mut0) {
                    const float y = pm_mutate(h ? c2 : c1, u01(h ? pm.z : pm.x), v.eta_m);
                    if (h)
                        c2 = y;
                    else
                        c1 = y;
                }
        } else {
            if (mut0) c1 = pm_mutate(c1, u01(pm.x), v.eta_m);
            if (mut1) c2 = pm_mutate(c2, u01(pm.z), v.eta_m);
        }
        out(var, c1, c2);
    }
}

// g term (x - 0.5)^2 of one variable added into a float-float sum (sh, sl):
// x - 0.5 by Fast2Sum (exact when x >= 0.25), the square's error by an FMA
__device__ __forceinline__ void g_add(float xv, float& sh, float& sl)
{
    const float th = __fsub_rn(xv, 0.5f);
    const float tl = xv < 0.25f ? __fsub_rn(xv, __fadd_rn(th, 0.5f)) : 0.0f;
    const float p = __fmul_rn(th, th);
    const float pl = __fmaf_rn(th, th, -p) + 2.0f * th * tl;
    float s1, e1;
    two_sum(sh, p, s1, e1);
    sh = s1;
    sl = sl + (e1 + pl);
}

// Variation of pair q fused with the softmax-simplex objective (m <= 10), one
// warp; each lane keeps its children's first m - 1 variables and its
// float-float partial sums of g while it writes the children, then the warp
// reduces g, lanes 0..m-1 (child 0) and 16..16+m-1 (child 1) form
// a_j = sum_e W_je x_e and e_j = exp(a_j), every lane adds e_0..e_{m-1} in
// order, and lane j writes f_j = (1 + g) e_j / den rounded to FP32.  The
// children are never read back.
//
// The arithmetic is FP32 with error-free transformations instead of FP64
// (1/64 of the FP32 rate on GB300): a_j as a compensated dot product
// (TwoProduct by FMA, TwoSum; Ogita, Rump and Oishi's Dot2) a_hi + a_lo;
// e_j = expf(a_hi) (1 + a_lo), so the rounding of a never reaches the
// exponential (an absolute error of a becomes a relative error of e_j);
// den and 1 + g as float-float sums; one correctly rounded division.  The
// result is within about 4 ulp (2.4e-7) of (1 + g) e_j / den: expf's 2 ulp,
// the division's and the last product's half ulp.
template <int M, bool ROLL>
__device__ __forceinline__ void vary_eval_pair(const RunView& v, int q, uint32_t gen)
{
    constexpr int K = M - 1;
    const int lane = lane_id();
    const int N = v.N;
    float* x0 = v.X + (size_t)v.fslot[2 * q] * v.d;
    float* x1 = v.X + (size_t)v.fslot[2 * q + 1] * v.d;
    merge_pair(v, q);
    float gh0 = 0.0f, gl0 = 0.0f, gh1 = 0.0f, gl1 = 0.0f;
    float xk0 = 0.0f, xk1 = 0.0f;
    vary_pair<ROLL>(v, q, gen, [&](int var, float c1, float c2) {
        x0[var] = c1;
        x1[var] = c2;
        if (var < K) {
            xk0 = c1;
            xk1 = c2;
        } else {
            g_add(c1, gh0, gl0);
            g_add(c2, gh1, gl1);
        }
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        float s1, e1;
        const float oh0 = __shfl_xor_sync(0xffffffffu, gh0, o), ol0 = __shfl_xor_sync(0xffffffffu, gl0, o);
        two_sum(gh0, oh0, s1, e1);
        gh0 = s1;
        gl0 = gl0 + (ol0 + e1);
        const float oh1 = __shfl_xor_sync(0xffffffffu, gh1, o), ol1 = __shfl_xor_sync(0xffffffffu, gl1, o);
        two_sum(gh1, oh1, s1, e1);
        gh1 = s1;
        gl1 = gl1 + (ol1 + e1);
    }
    const int j = lane & 15;
    const bool second = lane >= 16;
    float ah = 0.0f, al = 0.0f;
#pragma unroll
    for (int e = 0; e < K; ++e) {
        const float xe0 = __shfl_sync(0xffffffffu, xk0, e);
        const float xe1 = __shfl_sync(0xffffffffu, xk1, e);
        if (j < M) {
            const float w = v.Wobj[j * K + e], x = second ? xe1 : xe0;
            const float p = __fmul_rn(w, x);
            const float pe = __fmaf_rn(w, x, -p);
            float s1, e1;
            two_sum(ah, p, s1, e1);
            ah = s1;
            al = al + (e1 + pe);
        }
    }
    float ex = 0.0f;
    if (j < M) {
        const float E = expf(ah);
        ex = __fmaf_rn(E, al, E);
    }
    float dh0 = 0.0f, dl0 = 0.0f, dh1 = 0.0f, dl1 = 0.0f;
#pragma unroll
    for (int t = 0; t < M; ++t) {
        float s1, e1;
        two_sum(dh0, __shfl_sync(0xffffffffu, ex, t), s1, e1);
        dh0 = s1;
        dl0 += e1;
        two_sum(dh1, __shfl_sync(0xffffffffu, ex, 16 + t), s1, e1);
        dh1 = s1;
        dl1 += e1;
    }
    if (j < M) {
        const float dh = second ? dh1 : dh0, dl = second ? dl1 : dl0;
        float r = __fdiv_rn(ex, dh);
        r = __fmaf_rn(-r, __fdiv_rn(dl, dh), r);  // e / (dh + dl)
        const float gh = second ? gh1 : gh0, gl = second ? gl1 : gl0;
        float Gh, Ge;
        two_sum(1.0f, gh, Gh, Ge);
        const float Gl = Ge + gl;  // 1 + g = Gh + Gl
        v.F[(size_t)(N + 2 * q + (second ? 1 : 0)) * M + j] = __fmaf_rn(r, Gh, r * Gl);
    }
}

}  // namespace
