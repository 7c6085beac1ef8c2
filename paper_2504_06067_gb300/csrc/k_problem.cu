// k_problem.cu -- reference directions, initial population and the fused
// variation + objective kernel around the selection.
//
// Reference directions (Sec. II-C): Das-Dennis lattice {k/p : sum k = p} in
// lexicographic order of k, optional inner layer (1 - tau)/m + tau z; one
// thread unranks one composition.  FP64 with _rn intrinsics.
//
// Variation (Alg. 1, crossover and mutation; Sec. III-A), one warp per offspring pair q:
//   tournament: Philox(q, gen, 1, 0) -> a1, b1, a2, b2 in [0, N); the lower
//   front wins, ties keep the first drawn; Philox(q, gen, 1, 1) word 0 < p_c
//   lets the pair cross.  SBX per variable v (Philox(q*d+v, gen, 2, 0)):
//   word 1 < 0.5 crosses v with spread beta from word 0, word 2 < 0.5 swaps
//   the children; clip to [0,1].  Polynomial mutation of variable v: word 3
//   of that block < p_m mutates child 2q with u = word 0 of
//   Philox(q*d+v, gen, 3, 0); word 1 of that block < p_m mutates child 2q+1
//   with u = its word 2 (two Philox blocks per pair and variable).
//   Children 2q and 2q + 1 go to the rows fslot[2q], fslot[2q + 1].  FP32 arithmetic.
// Objective (the softmax-simplex family): k = m - 1,
//   g = sum_{v >= k} (x_v - 0.5)^2, f_j = (1 + g) softmax(W x[0:k])_j,
//   evaluated in FP64 (sums left to right) and rounded to FP32; for m > 10
//   the products W x are summed as compensated FP32 dot products.
#include "kernels.cuh"
#include "variation.cuh"

namespace {

__device__ long long binom_ll(int n, int k)
{
    if (k < 0 || k > n) return 0;
    long long r = 1;
    for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
    return r;
}

__global__ void k_refdirs(int m, int p1, int p2, double tau, int w1, int w, double* Zd, double* nz,
                          float* Zh, int M4)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= w) return;
    const bool inner = t >= w1;
    const int p = inner ? p2 : p1;
    long long idx = inner ? t - w1 : t;
    double* z = Zd + (size_t)t * m;  // first the composition k, then k / p
    int left = p;
    for (int q = 0; q < m - 1; ++q) {
        int val = 0;
        for (; val <= left; ++val) {
            const long long n = binom_ll(left - val + (m - q - 2), m - q - 2);
            if (idx < n) break;
            idx -= n;
        }
        z[q] = (double)val;
        left -= val;
    }
    z[m - 1] = (double)left;
    double s = 0.0;
    for (int q = 0; q < m; ++q) {
        double zq = __ddiv_rn(z[q], (double)p);
        if (inner) {
            const double a = __ddiv_rn(__dsub_rn(1.0, tau), (double)m);
            const double b = __dmul_rn(tau, zq);
            zq = __dadd_rn(a, b);
        }
        z[q] = zq;
        s = __dadd_rn(s, __dmul_rn(zq, zq));
    }
    const double n = __dsqrt_rn(s);
    nz[t] = n;
    for (int q = 0; q < M4; ++q) Zh[(size_t)t * M4 + q] = q < m ? __double2float_rn(__ddiv_rn(z[q], n)) : 0.0f;
}

// Objective of n rows of X into Fout: a block covers R = obj_rows(m) rows.
//   g = sum_{v >= m-1} (x_v - 0.5)^2: each term is formed exactly as a
//   float-float value (x - 0.5 by Fast2Sum, the square by an FMA product
//   error) and the terms are added in float-float (TwoSum) by a warp per row
//   with coalesced loads, then a warp reduction; the float-float sum is
//   within ~2^-44 relative of the exact sum, so (1 + g) in FP64 matches a
//   left-to-right FP64 sum to far below the final FP32 rounding.  This keeps
//   the sum off GB300's FP64 pipe (1/64 of the FP32 rate).
//   Thread (row, j) forms a_j = sum_v W_jv x_v in FP64 (left to right) and
//   e_j = exp(a_j); the row's denominator adds e_0..e_{m-1} in order once;
//   f_j = (1 + g) e_j / den, rounded to FP32.
constexpr int OR = 32;
constexpr int OT = 256;

// rows per block: 32 for m <= 10; above, about 256 (row, objective) pairs
// per block, one per thread, so that the FP64 dot products of many
// objectives spread over the whole GPU (R x m exponentials in shared memory)
inline int obj_rows(int m)
{
    if (m <= NSGA3_FAST_M) return OR;
    const int r = OT / m;
    return r < 1 ? 1 : r;
}
inline size_t obj_smem(int m) { return (size_t)obj_rows(m) * (m + 2) * sizeof(double); }

// m > NSGA3_FAST_M: a_j = sum_v W_jv x_v for RB rows x 128 objectives per
// CTA as compensated FP32 dot products (each product split exactly into
// p + e by an FMA, the sum carried as a float-float pair by TwoSum; Ogita,
// Rump and Oishi's Dot2), then e_j = exp(a_j) in FP64 into v.fprime (free
// during the variation).  Dot2's error, about (k 2^-24)^2 of sum |W x|, is
// far below the FP32 rounding of f: the FP64 evaluation of the m
// exponentials' products would take the FP64 pipe (1/64 of FP32) for
// m (m-1) N operations.
constexpr int RB = 4;     // rows per CTA
constexpr int DT = 128;   // objectives per CTA

// (row r of the n is row rows[r] of X, here and in k_objective)
__global__ void __launch_bounds__(DT) k_obj_dot(RunView v, const int32_t* rows_of, int n)
{
    extern __shared__ float xs[];  // RB x k
    const int m = v.m, d = v.d, k = m - 1;
    const int base = blockIdx.x * RB;
    const int rows = min(RB, n - base);
    // (the rows' numbers first: four pairs of dependent loads in flight)
    const float* x[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) x[r] = v.X + (size_t)rows_of[min(base + r, n - 1)] * d;
    for (int c = threadIdx.x; c < k; c += DT) {
        float t[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) t[r] = x[r][c];
#pragma unroll
        for (int r = 0; r < RB; ++r) xs[r * k + c] = r < rows ? t[r] : 0.0f;
    }
    __syncthreads();
    const int j = blockIdx.y * DT + threadIdx.x;
    if (j >= m) return;
    float hi[RB], lo[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        hi[r] = 0.0f;
        lo[r] = 0.0f;
    }
    auto add = [&](int e, float w) {
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const float x = xs[r * k + e];
            const float p = __fmul_rn(w, x);
            const float pe = __fmaf_rn(w, x, -p);  // w x = p + pe exactly
            float s1, t1;
            two_sum(hi[r], p, s1, t1);
            hi[r] = s1;
            lo[r] = __fadd_rn(lo[r], __fadd_rn(t1, pe));
        }
    };
    // eight weights are added while the next eight load (left to an unrolled
    // loop the compiler loaded them one after another: m = 512, N = 300 62.8
    // us, 46 so; m = 200, N = 500 28.7 and 22)
    const float* wt = v.Wt + j;
    auto load = [&](int e, float(&w)[8]) {
#pragma unroll
        for (int t = 0; t < 8; ++t) w[t] = __ldg(wt + (size_t)min(e + t, k - 1) * m);
    };
    float w[8];
    load(0, w);
    int e = 0;
    for (; e + 8 <= k; e += 8) {
        float next[8];
        load(e + 8, next);
#pragma unroll
        for (int t = 0; t < 8; ++t) add(e + t, w[t]);
#pragma unroll
        for (int t = 0; t < 8; ++t) w[t] = next[t];
    }
#pragma unroll
    for (int t = 0; t < 8; ++t)
        if (e + t < k) add(e + t, w[t]);
#pragma unroll
    for (int r = 0; r < RB; ++r)
        if (r < rows) {
            const double a = __dadd_rn((double)hi[r], (double)lo[r]);
            v.fprime[(size_t)(base + r) * m + j] = exp(a);
        }
}

__global__ void __launch_bounds__(OT) k_objective(RunView v, const int32_t* rows_of, float* Fout, int n, int R)
{
    extern __shared__ double sobj[];
    double* sg = sobj;        // R
    double* sden = sg + R;    // R
    double* se = sden + R;    // R x m
    const int m = v.m, d = v.d, k = m - 1;
    const int base = blockIdx.x * R;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    for (int rr = warp; rr < R; rr += OT / 32) {
        float sh = 0.0f, sl = 0.0f;
        if (base + rr < n) {
            const float* x = v.X + (size_t)rows_of[base + rr] * d;
            for (int e = k + lane; e < d; e += 32) {
                const float xv = x[e];
                const float th = __fsub_rn(xv, 0.5f);
                // Fast2Sum error of x + (-0.5); zero when x >= 0.25 (Sterbenz)
                const float tl = xv < 0.25f ? __fsub_rn(xv, __fadd_rn(th, 0.5f)) : 0.0f;
                const float p = __fmul_rn(th, th);
                const float pl = __fmaf_rn(th, th, -p) + 2.0f * th * tl;
                float s1, e1;
                two_sum(sh, p, s1, e1);
                sh = s1;
                sl = sl + (e1 + pl);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, sh, o);
            const float ol = __shfl_xor_sync(0xffffffffu, sl, o);
            float s1, e1;
            two_sum(sh, oh, s1, e1);
            sh = s1;
            sl = sl + (ol + e1);
        }
        if (lane == 0) sg[rr] = __dadd_rn((double)sh, (double)sl);
    }
    for (int idx = threadIdx.x; idx < R * m; idx += OT) {
        const int rr = idx / m, j = idx - rr * m;
        if (base + rr >= n) continue;
        if (m > NSGA3_FAST_M) {  // exponentials from k_obj_dot
            se[idx] = v.fprime[(size_t)(base + rr) * m + j];
            continue;
        }
        const float* x = v.X + (size_t)rows_of[base + rr] * d;
        double a = 0.0;
        for (int e = 0; e < k; ++e) a = __dadd_rn(a, __dmul_rn((double)v.Wobj[j * k + e], (double)x[e]));
        se[idx] = exp(a);
    }
    __syncthreads();
    if (threadIdx.x < R && base + threadIdx.x < n) {
        double den = 0.0;
        for (int t = 0; t < m; ++t) den = __dadd_rn(den, se[threadIdx.x * m + t]);
        sden[threadIdx.x] = den;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < R * m; idx += OT) {
        const int rr = idx / m, j = idx - rr * m;
        if (base + rr >= n) continue;
        const double f = __dmul_rn(__dadd_rn(1.0, sg[rr]), __ddiv_rn(se[idx], sden[rr]));
        Fout[(size_t)(base + rr) * m + j] = __double2float_rn(f);
    }
}


__global__ void k_init(RunView v)
{
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= v.N) return;
    const int lane = lane_id();
    const int slot = v.pold[i];  // as a population set by the caller (k_rows_in)
    float* xrow = v.X + (size_t)slot * v.d;
    for (int e = lane; e < v.d; e += 32) {
        U4 r = philox((uint32_t)i * (uint32_t)v.d + (uint32_t)e, 0u, RNG_INIT, 0u, v.seed);
        xrow[e] = u01(r.x);
    }
    if (lane == 0) {
        v.rank[i] = 0;
        v.pcan[i] = slot;
        v.fslot[i] = v.cslot[i];
    }
}

// Variation only (m > 10: the objective follows in k_obj_dot + k_objective).
// A warp per pair while pairs fill the GPU; with fewer, gridDim.y warps share
// a pair's variables (each repeats its tournament).  400 pairs of 1,000
// variables: 26 us in one warp each, 9.4 in six.
__global__ void k_vary(RunView v)
{
    const int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (q >= v.N / 2) return;
    if (read_status(v.ctrl)) return;
    const uint32_t gen = v.ctrl->gen;
    float* x0 = v.X + (size_t)v.fslot[2 * q] * v.d;
    float* x1 = v.X + (size_t)v.fslot[2 * q + 1] * v.d;
    if (blockIdx.y == 0) merge_pair(v, q);
    vary_pair<false>(
        v, q, gen,
        [&](int var, float c1, float c2) {
            x0[var] = c1;
            x1[var] = c2;
        },
        32 * blockIdx.y, 32 * gridDim.y);
}

// Variation fused with the softmax-simplex objective (m <= 10; see
// vary_eval_pair): one warp per pair
template <int M>
__global__ void __launch_bounds__(256) k_vary_eval(RunView v)
{
    const int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (q >= v.N / 2) return;
    if (read_status(v.ctrl)) return;
    vary_eval_pair<M, false>(v, q, v.ctrl->gen);
}

cudaError_t launch_obj_dot(const RunView& v, const int32_t* rows_of, int n, cudaStream_t s)
{
    if (!v.Wt) return cudaErrorInvalidValue;
    const size_t sm = (size_t)RB * (v.m - 1) * sizeof(float);
    k_obj_dot<<<dim3((n + RB - 1) / RB, (v.m + DT - 1) / DT), DT, sm, s>>>(v, rows_of, n);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_refdirs(const RunView& v, int p1, int p2, double tau, double* Zd, double* nz,
                           float* Zh, cudaStream_t s)
{
    long long w1 = 1;
    {
        // C(p1 + m - 1, m - 1)
        long long r = 1;
        for (int i = 1; i <= v.m - 1; ++i) r = r * (p1 + i) / i;
        w1 = r;
    }
    k_refdirs<<<(v.w + 127) / 128, 128, 0, s>>>(v.m, p1, p2, tau, (int)w1, v.w, Zd, nz, Zh, v.M4);
    return cudaGetLastError();
}

cudaError_t launch_init(const RunView& v, cudaStream_t s)
{
    if (v.problem == 1) return launch_kp_init(v, s);
    long long threads = (long long)v.N * 32;
    k_init<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(v);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (v.m > NSGA3_FAST_M) {
        e = launch_obj_dot(v, v.pold, v.N, s);
        if (e != cudaSuccess) return e;
    }
    const int R = obj_rows(v.m);
    k_objective<<<(v.N + R - 1) / R, OT, obj_smem(v.m), s>>>(v, v.pold, v.PF, v.N, R);
    return cudaGetLastError();
}

cudaError_t launch_vary_eval(const RunView& v, cudaStream_t s)
{
    if (v.problem == 1) return launch_kp_vary_eval(v, s);
    long long threads = (long long)(v.N / 2) * 32;
    const unsigned blocks = (unsigned)((threads + 255) / 256);
    if (v.m <= NSGA3_FAST_M) {
        switch (v.m) {
        case 2: k_vary_eval<2><<<blocks, 256, 0, s>>>(v); break;
        case 3: k_vary_eval<3><<<blocks, 256, 0, s>>>(v); break;
        case 4: k_vary_eval<4><<<blocks, 256, 0, s>>>(v); break;
        case 5: k_vary_eval<5><<<blocks, 256, 0, s>>>(v); break;
        case 6: k_vary_eval<6><<<blocks, 256, 0, s>>>(v); break;
        case 7: k_vary_eval<7><<<blocks, 256, 0, s>>>(v); break;
        case 8: k_vary_eval<8><<<blocks, 256, 0, s>>>(v); break;
        case 9: k_vary_eval<9><<<blocks, 256, 0, s>>>(v); break;
        default: k_vary_eval<10><<<blocks, 256, 0, s>>>(v); break;
        }
        return cudaGetLastError();
    }
    // about 16 warps per SM (a quarter of what is resident: issue-bound)
    const int want = 16 * v.num_sms / (v.N / 2), most = (v.d + 31) / 32;
    const int parts = want < 1 ? 1 : want < most ? want : most;
    k_vary<<<dim3(blocks, parts), 256, 0, s>>>(v);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_obj_dot(v, v.cslot, v.N, s);
    if (e != cudaSuccess) return e;
    const int R = obj_rows(v.m);
    k_objective<<<(v.N + R - 1) / R, OT, obj_smem(v.m), s>>>(v, v.cslot, v.F + (size_t)v.N * v.m, v.N, R);
    return cudaGetLastError();
}
