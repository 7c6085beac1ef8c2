// k_sort.cu -- sort keys of the merged population, used by the dominance
// build and the front peel (Alg. 1, the non-dominated sort).
//
// For m <= 10 every objective q is cut into L = 2^lbits levels by L - 1
// thresholds near its quantiles (from a histogram of the selection's own
// values), and a point's key interleaves the bits of its m levels from the
// top bit down (Morton order), truncated to kbits.  A point i can dominate
// j only if f_iq <= f_jq for every q, so only if every level of i is at most
// the level of j, and then every prefix of the interleaved bits of i is at
// most that of j: dominators never have a larger key, equal vectors have
// equal keys, and points with nearby keys are close in every objective, so
// 32-point blocks of the key order have small bounding boxes that let the
// dominance build rule out most block pairs.  Any thresholds would be
// correct; quantiles balance the levels.  For m > 10 the key is one of 4,096
// buckets of f_0.  A counting sort into the 2^kbits keys orders the points;
// ties and order inside a key do not matter: every pair that can dominate is
// still tested exactly.
// The thresholds (and, for m > 10, the f_0 range of the buckets) come from a
// fixed sample of evenly spaced points (512; 8,192 for the range): they only
// steer how well the blocks prune, and a value outside the sample's range
// still gets a monotone key (levels count thresholds, buckets are clamped).
//   k_front         (m <= 10) the selection's reset and finite check, and per
//                   objective one CTA that sorts its sampled values and takes
//                   the quantiles: 4.4 us in place of the reset, the check,
//                   the range and the histogram kernels (23 of 227 us at
//                   m = 5, N = 10,628; 34 us at m = 10, N = 100,000)
//   k_sort_range    (m > 10) min / max of f_0 over the sample
//   k_sort_hist     every point's key (kept in pkey), key counts and counts of
//                   groups of 32 keys
//   k_sort_scatter  each CTA scans the group counts (nkeys / 32 of them) and a
//                   point adds the counts before its key in its group, instead
//                   of one last CTA scanning every key (both kernels 58 us for
//                   65,536 keys and 200,000 points; now 28);
//                   perm[pos] = i, skey[pos] = key, Fp = F in key order with
//                   -0.0 written as +0.0; row limits of the peel's chunks
#include "kernels.cuh"

namespace {

constexpr int SB = 1024;
constexpr int SAMPLE = 8192;  // points that set the f_0 range
constexpr int FS = 512;       // points that set the level thresholds
constexpr int KGROUP = 32;    // keys per group of the counting sort

// stride of that sample
__device__ __forceinline__ int sample_stride(int n2) { return n2 > SAMPLE ? (n2 + SAMPLE - 1) / SAMPLE : 1; }

__device__ __forceinline__ int bucket_of(float f, float lo, float scale, int nb)
{
    float t = (f - lo) * scale;
    int b = (int)t;
    if (!(t >= 0.0f)) b = 0;
    return b > nb - 1 ? nb - 1 : b;
}

__device__ __forceinline__ void range_of(const Ctrl* c, int nb, float& lo, float& scale)
{
    lo = ord2f(c->f0lo);
    const float hi = ord2f(c->f0hi);
    const float span = hi - lo;
    scale = (span > 0.0f && span < 3.0e38f) ? (float)nb / span : 0.0f;
}

// sort key of point i (see the file comment); thr: the level thresholds
// (m <= 10), staged by the caller
__device__ __forceinline__ uint32_t key_of(const RunView& v, const Ctrl* c, const float (*thr)[SORT_LMAX], int i)
{
    const int m = v.m;
    const float* f = v.F + (size_t)i * m;
    if (m > NSGA3_FAST_M) {
        float lo, scale;
        range_of(c, SORT_NB, lo, scale);
        return (uint32_t)bucket_of(f[0] + 0.0f, lo, scale, SORT_NB);
    }
    const int lb = v.lbits, nthr = (1 << lb) - 1;
    uint32_t lev[NSGA3_FAST_M];
#pragma unroll
    for (int q = 0; q < NSGA3_FAST_M; ++q) {
        uint32_t l = 0u;
        if (q < m) {
            const float x = f[q];
            for (int k = 0; k < nthr; ++k) l += x > thr[q][k] ? 1u : 0u;
        }
        lev[q] = l;
    }
    uint32_t key = 0u;
    for (int b = lb - 1; b >= 0; --b)
#pragma unroll
        for (int q = 0; q < NSGA3_FAST_M; ++q)
            if (q < m) key = (key << 1) | ((lev[q] >> b) & 1u);
    return key >> (lb * m - v.kbits);
}

// m > 10: min / max of the sampled f_0
__global__ void __launch_bounds__(SB) k_sort_range(RunView v)
{
    Ctrl* c = v.ctrl;
    if (read_status(c)) return;
    uint32_t lo = 0xffffffffu, hi = 0u;
    const int st = sample_stride(v.n2);
    for (int i = (blockIdx.x * SB + threadIdx.x) * st; i < v.n2; i += gridDim.x * SB * st) {
        const uint32_t o = f2ord(v.F[(size_t)i * v.m] + 0.0f);
        lo = min(lo, o);
        hi = max(hi, o);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane_id() == 0) {
        atomicMin(&c->f0lo, lo);
        atomicMax(&c->f0hi, hi);
    }
}

// The per-selection reset by the threads [t0, t0 + stride, ...) of a launch
__device__ __forceinline__ void sel_reset(const RunView& v, int tid, int stride)
{
    for (int j = tid; j < v.ld; j += stride) {
        v.cnt[j] = 0;
        v.rank2[j] = -1;
        v.srank[j] = -1;
    }
    const int nk = 1 << v.kbits;
    for (int b = tid; b < nk; b += stride) {
        v.bcnt[b] = 0;
        v.bcur[b] = 0;
    }
    for (int b = tid; b < nk / KGROUP; b += stride) v.bgrp[b] = 0;
    if (v.dnz) {
        // the block bitmap starts empty: only tiles with block pairs to test write bytes
        const long long nb = (long long)v.NW * v.NB8;  // 8 T^2 bytes, T = ld / 256
        uint2* z = reinterpret_cast<uint2*>(v.dnz);
        for (long long e = tid; e < nb / 8; e += stride) z[e] = make_uint2(0u, 0u);
    }
    for (int wd = tid; wd < v.NW; wd += stride) {
        v.selmask[wd] = 0u;
        if (v.domw) {
            v.domw[wd] = 0u;
            v.jpos[wd] = 0;
        }
    }
    for (int j = tid; j < v.w; j += stride) {
        v.rho[j] = 0;
        v.rhop[j] = 0;
        v.cursor[j] = 0;
        v.rprio[j] = philox((uint32_t)j, v.ctrl->gen, RNG_REFPRIO, 0u, v.seed).x;
    }
    Ctrl* c = v.ctrl;
    if (tid < v.m) c->zmin[tid] = 0xffffffffu;
    if (tid < 8) c->domstat[tid] = 0ull;
    if (tid == 0) {
        c->cum = 0;
        c->l = -1;
        c->nS = 0;
        c->K = 0;
        c->nFl = 0;
        c->need_niche = 0;
        c->fallback = 0;
        c->passes = 0;
        c->nT = 0;
        c->Lstar = -1;
        c->rlev = 0;
        c->nsel = 0;
        c->nlarge = 0;
        c->npath = 0u;
        c->ntile = 0;
        c->ntask = 0;
        c->parr = 0u;
        c->nF0 = 0;
        c->nrem = 0;
        c->odd = 0;
        c->peel_rows = 0u;
        c->ncand = 0;
        c->nslow = 0;
        c->ext_done = 0u;
        c->f0lo = 0xffffffffu;
        c->f0hi = 0u;
        c->overflow = 0;
        c->recheck_miss = 0;
    }
}

__global__ void __launch_bounds__(256) k_sel_reset(RunView v)
{
    sel_reset(v, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// m <= 10.  CTA q < m: level thresholds of objective q.  A thread holds one
// sampled value (order-preserving code); a bitonic sort, exchanges within a
// warp by shuffles, wider ones through shared memory (10 of the 45 steps);
// the threshold of level k + 1 is the smallest sampled value with at least
// (k + 1) / L of the sample at or below it.  (Ranking each value by counting
// the smaller ones took 11 us; a sample of 1,024 values 7.2.)  The other CTAs
// reset the selection's buffers and (check != 0) look for non-finite
// objectives.
__global__ void __launch_bounds__(FS) k_front(RunView v, int check)
{
    Ctrl* c = v.ctrl;
    const int tid = threadIdx.x;
    if ((int)blockIdx.x >= v.m) {
        const int t = ((int)blockIdx.x - v.m) * FS + tid, stride = ((int)gridDim.x - v.m) * FS;
        sel_reset(v, t, stride);
        if (check) {
            const long long n = (long long)v.n2 * v.m;
            bool bad = false;
            for (long long e = t; e < n; e += stride) bad |= !isfinite(v.F[e]);
            if (__any_sync(0xffffffffu, bad) && lane_id() == 0) set_status(c, DEV_ENONFINITE);
        }
        return;
    }
    __shared__ uint32_t x[2][FS];  // two buffers: one barrier per exchange
    int buf = 0;
    const int q = blockIdx.x, ns = min(v.n2, FS);
    uint32_t a = 0xffffffffu;
    if (tid < ns) a = f2ord(v.F[(size_t)((long long)tid * v.n2 / ns) * v.m + q] + 0.0f);
#pragma unroll 1
    for (int k = 2; k <= FS; k <<= 1) {
        const bool up = (tid & k) == 0;  // this run's direction
#pragma unroll 1
        for (int o = k >> 1; o >= 32; o >>= 1) {
            x[buf][tid] = a;
            __syncthreads();
            const uint32_t b = x[buf][tid ^ o];
            buf ^= 1;
            a = (((tid & o) == 0) == up) ? min(a, b) : max(a, b);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint32_t b = __shfl_xor_sync(0xffffffffu, a, o);
            const uint32_t y = (((tid & o) == 0) == up) ? min(a, b) : max(a, b);
            a = o < k ? y : a;
        }
    }
    const int L = 1 << v.lbits;
    // thread t holds the t-th smallest: rank t + 1 = ceil((k + 1) ns / L) sets threshold k
    for (int k = 0; k + 1 < L; ++k)
        if (tid + 1 == ((k + 1) * ns + L - 1) / L) c->thr[q][k] = ord2f(a);
}

// (the group counts of a CTA's points meet in shared memory first: most
// points of a converged population share a few groups)
__global__ void __launch_bounds__(SB) k_sort_hist(RunView v)
{
    extern __shared__ int gcnt[];  // nkeys / KGROUP
    __shared__ float thr[NSGA3_FAST_M][SORT_LMAX];
    Ctrl* c = v.ctrl;
    if (read_status(c)) return;
    if (v.m <= NSGA3_FAST_M) {
        if (threadIdx.x < NSGA3_FAST_M * SORT_LMAX)
            thr[threadIdx.x / SORT_LMAX][threadIdx.x % SORT_LMAX] = c->thr[threadIdx.x / SORT_LMAX][threadIdx.x % SORT_LMAX];
    }
    const int ng = (1 << v.kbits) / KGROUP;
    for (int g = threadIdx.x; g < ng; g += SB) gcnt[g] = 0;
    __syncthreads();
    const int i = blockIdx.x * SB + threadIdx.x;
    if (i < v.n2) {
        if (v.domw) {  // k_dominance_front's pair test is for finite objectives
            const float* f = v.F + (size_t)i * v.m;
            bool odd = false;
            for (int q = 0; q < v.m; ++q) odd |= !isfinite(f[q]);
            if (odd) c->odd = 1;
        }
        const uint32_t key = key_of(v, c, thr, i);
        v.pkey[i] = key;
        atomicAdd(&v.bcnt[key], 1);
        atomicAdd(&gcnt[key / KGROUP], 1);
    }
    __syncthreads();
    for (int g = threadIdx.x; g < ng; g += SB)
        if (gcnt[g]) atomicAdd(&v.bgrp[g], gcnt[g]);
}

constexpr int TB = 512;  // threads of the scatter's CTAs

// positions before key group g, for every group: an exclusive scan of the
// group counts in shared memory (each CTA for itself)
__device__ __forceinline__ void scan_groups(const RunView& v, int* off, int* scratch)
{
    const int ng = (1 << v.kbits) / KGROUP, per = (ng + TB - 1) / TB;
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    for (int g = tid; g < ng; g += TB) off[g] = v.bgrp[g];
    __syncthreads();
    const int lo = min(ng, tid * per), hi = min(ng, lo + per);
    int s = 0;
    for (int g = lo; g < hi; ++g) s += off[g];
    int inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) scratch[warp] = inc;
    __syncthreads();
    int run = inc - s;
    for (int t = 0; t < warp; ++t) run += scratch[t];
    for (int g = lo; g < hi; ++g) {
        const int x = off[g];
        off[g] = run;
        run += x;
    }
    __syncthreads();
}

// Position of a point of key b, and where the positions of key b end: the
// group's offset, the counts before b in the group (whole 16-byte loads) and
// the order in which the key's points arrive.
__device__ __forceinline__ int place(const RunView& v, const int* off, uint32_t b, int& end)
{
    const int g0 = (int)(b & ~(uint32_t)(KGROUP - 1));
    int at = off[b / KGROUP], own = 0;
#pragma unroll
    for (int e = 0; e < KGROUP; e += 4) {
        if (g0 + e > (int)b) break;
        const int4 x = *reinterpret_cast<const int4*>(v.bcnt + g0 + e);
        const int y[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            at += g0 + e + t < (int)b ? y[t] : 0;
            own = g0 + e + t == (int)b ? y[t] : own;
        }
    }
    end = at + own;
    return at + atomicAdd(&v.bcur[b], 1);
}

// dominators of a column have a key <= its key: the peel's chunk of columns
// reads row blocks up to the end of its last column's key
__device__ __forceinline__ void chunk_limit(const RunView& v, int pos, int end)
{
    if ((pos & (NSGA3_PEEL_COLS - 1)) == NSGA3_PEEL_COLS - 1 || pos == v.n2 - 1)
        v.chunk_lim[pos / NSGA3_PEEL_COLS] = (uint32_t)((end + 31) >> 5);
    if (v.kend && ((pos & 31) == 31 || pos == v.n2 - 1)) v.kend[pos / 32] = end;
}

__global__ void __launch_bounds__(TB) k_sort_scatter(RunView v)
{
    extern __shared__ int goff[];  // nkeys / KGROUP
    __shared__ int scratch[TB / 32];
    __shared__ int spos[TB];
    Ctrl* c = v.ctrl;
    if (read_status(c)) return;
    scan_groups(v, goff, scratch);
    const int m = v.m, i0 = blockIdx.x * TB, i = i0 + threadIdx.x;
    if (i < v.n2) {
        const uint32_t b = v.pkey[i];
        int end;
        const int pos = place(v, goff, b, end);
        v.perm[pos] = i;
        v.skey[pos] = b;
        chunk_limit(v, pos, end);
        spos[threadIdx.x] = pos;
    }
    __syncthreads();
    // rows: a thread per 16 bytes
    const int n4 = v.fs / 4, ne = min(TB, v.n2 - i0) * n4;
    for (int e = threadIdx.x; e < ne; e += TB) {
        const int r = e / n4, q = 4 * (e - r * n4);
        const float* f = v.F + (size_t)(i0 + r) * m + q;
        float4 x;
        x.x = f[0] + 0.0f;
        x.y = q + 1 < m ? f[1] + 0.0f : 0.0f;
        x.z = q + 2 < m ? f[2] + 0.0f : 0.0f;
        x.w = q + 3 < m ? f[3] + 0.0f : 0.0f;
        *reinterpret_cast<float4*>(v.Fp + (size_t)spos[r] * v.fs + q) = x;
    }
}

// m > NSGA3_FAST_M: a warp per point copies its row
__global__ void __launch_bounds__(TB) k_sort_scatter_rows(RunView v)
{
    extern __shared__ int goff[];
    __shared__ int scratch[TB / 32];
    Ctrl* c = v.ctrl;
    if (read_status(c)) return;
    scan_groups(v, goff, scratch);
    const int i = (blockIdx.x * TB + threadIdx.x) >> 5;
    if (i >= v.n2) return;
    const int lane = lane_id(), m = v.m;
    int pos = 0;
    if (lane == 0) {
        const uint32_t b = v.pkey[i];
        int end;
        pos = place(v, goff, b, end);
        v.perm[pos] = i;
        v.skey[pos] = b;
        chunk_limit(v, pos, end);
    }
    pos = __shfl_sync(0xffffffffu, pos, 0);
    for (int q = lane; q < m; q += 32) v.Fp[(size_t)pos * m + q] = v.F[(size_t)i * m + q] + 0.0f;
}

}  // namespace

cudaError_t launch_front(const RunView& v, int num_sms, bool check, cudaStream_t s)
{
    if (v.m > NSGA3_FAST_M) {
        const int n = v.ld > v.w ? v.ld : v.w;
        int blocks = (n + 255) / 256;
        if (blocks > 2048) blocks = 2048;
        k_sel_reset<<<blocks, 256, 0, s>>>(v);
        const cudaError_t e = cudaGetLastError();
        return e != cudaSuccess || !check ? e : launch_check_finite(v, s);
    }
    long long n = (long long)v.n2 * v.m;  // at least a few elements per thread
    int blocks = (int)((n + 4 * FS - 1) / (4 * FS));
    if (blocks > 4 * num_sms) blocks = 4 * num_sms;
    k_front<<<v.m + blocks, FS, 0, s>>>(v, check ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_sort(const RunView& v, int num_sms, cudaStream_t s)
{
    if (v.m > NSGA3_FAST_M) {
        int blocks = (v.n2 + SB - 1) / SB;
        if (blocks > num_sms) blocks = num_sms;
        k_sort_range<<<blocks, SB, 0, s>>>(v);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const size_t sm = (size_t)((1 << v.kbits) / KGROUP) * sizeof(int);
    k_sort_hist<<<(v.n2 + SB - 1) / SB, SB, sm, s>>>(v);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (v.m > NSGA3_FAST_M)
        k_sort_scatter_rows<<<(unsigned)(((long long)v.n2 * 32 + TB - 1) / TB), TB, sm, s>>>(v);
    else
        k_sort_scatter<<<(v.n2 + TB - 1) / TB, TB, sm, s>>>(v);
    return cudaGetLastError();
}
