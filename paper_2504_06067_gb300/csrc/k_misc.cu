// k_misc.cu -- boundary check of the objectives (m > 10), the
// selected indices and the next population (Alg. 2 last line: P_{t+1} = rows
// with rank < l after selection), and copies of populations in and out.
#include "kernels.cuh"

namespace {

__global__ void k_check_finite(RunView v)
{
    const long long n = (long long)v.n2 * v.m;
    bool bad = false;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x)
        bad |= !isfinite(v.F[e]);
    if (__any_sync(0xffffffffu, bad) && lane_id() == 0) set_status(v.ctrl, DEV_ENONFINITE);
}

// Selected = S u (picked members of F_l), or S u F_l when no niching is
// needed, in ascending index order, in two kernels: every warp builds one
// 32-member mask word (ballot) and every CTA the count of its 32 words; then
// each CTA of k_gather adds up the counts before it (at most 2,048 of them,
// a few loads per thread) instead of one last CTA scanning every word (30 us
// of a 5,600 us selection at N = 100,000, 7 of 227 us at N = 10,628).
__global__ void __launch_bounds__(1024) k_mark(RunView v)
{
    uint32_t* words = v.selword;
    __shared__ int cnt[32];
    Ctrl* c = v.ctrl;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int wd = blockIdx.x * 32 + warp;
    const int j = wd * 32 + lane;
    const int r = wd < v.NW && j < v.n2 ? v.rank2[j] : -1;
    const uint32_t picked = wd < v.NW ? v.selmask[wd] : 0u;
    if (read_status(c)) return;
    const int l = c->l, need = c->need_niche;
    const bool take = r >= 0 && (r < l || (r == l && (!need || ((picked >> lane) & 1u))));
    const uint32_t word = __ballot_sync(0xffffffffu, take);
    if (lane == 0) {
        if (wd < v.NW) words[wd] = word;
        cnt[warp] = __popc(word);
    }
    __syncthreads();
    if (warp == 0) {
        const int t = warp_sum(cnt[lane]);
        if (lane == 0) v.bsum[blockIdx.x] = t;
    }
}

// What k_gather writes for a selected individual i at position p of the next
// population (ascending i): the selection's index list, or the parents' row
// (pcan), objectives (PF) and rank; a dropped individual's row becomes free
// (fslot).  Rows of X do not move.
enum : int {
    GATHER_SEL = 0,   // the index list only (nsga3_select)
    GATHER_POP = 1,   // the next population
    GATHER_INDEX = 2  // ... without its objectives (m > NSGA3_FAST_M: k_gather_rows)
};
constexpr int GB = 256;  // individuals per CTA

__global__ void __launch_bounds__(GB) k_gather(RunView v, int mode)
{
    __shared__ int s_pre[GB / 32], s_tot[GB / 32];
    Ctrl* c = v.ctrl;
    const int lane = lane_id(), warp = threadIdx.x >> 5, tid = threadIdx.x;
    const uint32_t* words = v.selword;
    const int nb = (v.NW + 31) / 32, b0 = blockIdx.x >> 2, w0 = blockIdx.x * (GB / 32);
    int pre = 0, tot = 0;
    for (int t = tid; t < nb; t += GB) {
        const int x = v.bsum[t];
        tot += x;
        if (t < b0) pre += x;
    }
    // the words before this CTA's in its group of 32 (1,024 individuals), and
    // in its own 8
    if (tid < w0 - b0 * 32) pre += __popc(words[b0 * 32 + tid]);
    const uint32_t word = words[w0 + warp];  // NW is a multiple of 8
    int own = 0;
    for (int t = 0; t < warp; ++t) own += __popc(words[w0 + t]);
    const int i = blockIdx.x * GB + tid;
    const int slot = mode == GATHER_SEL || i >= v.n2 ? 0 : i < v.N ? v.pold[i] : v.cslot[i - v.N];
    const int r = mode == GATHER_SEL || i >= v.n2 ? 0 : v.rank2[i];
    if (read_status(c)) return;
    pre = warp_sum(pre);
    tot = warp_sum(tot);
    if (lane == 0) {
        s_pre[warp] = pre;
        s_tot[warp] = tot;
    }
    __syncthreads();
    pre = 0;
    tot = 0;
#pragma unroll
    for (int t = 0; t < GB / 32; ++t) {
        pre += s_pre[t];
        tot += s_tot[t];
    }
    if (tot != v.N) {  // an invariant failed upstream: nothing is written
        if (tid == 0) {
            c->nsel = tot;
            set_status(c, DEV_EINTERNAL);
        }
        return;
    }
    const int p = pre + own + __popc(word & ((1u << lane) - 1u));
    if (i < v.n2) {
        if ((word >> lane) & 1u) {
            v.sel[p] = i;
            if (mode != GATHER_SEL) {
                v.pcan[p] = slot;
                v.rank[p] = r;
                if (mode == GATHER_POP)
                    for (int q = 0; q < v.m; ++q) v.PF[(size_t)p * v.m + q] = v.F[(size_t)i * v.m + q];
            }
        } else if (mode != GATHER_SEL) {
            v.fslot[i - p] = slot;
        }
    }
    if (blockIdx.x == 0 && tid == 0) {
        c->nsel = tot;
        if (mode != GATHER_SEL) c->gen += 1u;
    }
}

// m > NSGA3_FAST_M: the next parents' objectives (warp per row)
__global__ void __launch_bounds__(256) k_gather_rows(RunView v)
{
    const int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (p >= v.N) return;
    const int i = v.sel[p];
    if (read_status(v.ctrl)) return;
    for (int q = lane_id(); q < v.m; q += 32) v.PF[(size_t)p * v.m + q] = v.F[(size_t)i * v.m + q];
}

// Rows between X and a caller's N x d array, in words of 16, 8 or 4 bytes as
// both sides' rows allow.  A CTA moves R * 256 consecutive words of the array,
// a thread R of them 256 apart with all loads in flight; one 64-bit division
// per thread finds the CTA's first row.  (A warp per row left most lanes idle
// at small d and one load in flight at large ones: 11.3 us for 12,800 rows of
// 500, 8.2 now.)  Bound: requests in flight: 50,000 rows of 200 / 202 / 201
// floats 10 / 15 / 20 us (a plain copy 12.6).
constexpr int RW = 4;

// words per thread (eight of 4 bytes leave too few threads at small sizes)
template <class T>
__host__ __device__ constexpr int row_words()
{
    return sizeof(T) == 8 ? 8 : 4;
}
__host__ __device__ inline int plain_ctas(const PlainCopy& p) { return (p.n + 256 * RW - 1) / (256 * RW); }

template <class T, int R, class F>
__device__ __forceinline__ void for_row_words(int N, int words, F&& f)
{
    const long long e0 = (long long)blockIdx.x * (256 * R);
    const long long p0 = e0 / words;
    const int r0 = (int)(e0 - p0 * words);
    T x[R];
    int p[R], q[R];
    // r / words for r < words + 256 R: exact by the reciprocal for rows below
    // 2,048 words (r words < 2^24), one wrap at most for longer ones
    static_assert(R <= 8, "one wrap");
    const unsigned inv = words < 2048 ? (1u << 24) / (unsigned)words + 1u : 0u;
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const unsigned r = (unsigned)r0 + t * 256 + threadIdx.x;
        const unsigned n = words < 2048 ? (unsigned)(((unsigned long long)r * inv) >> 24) : (r >= (unsigned)words ? 1u : 0u);
        p[t] = p0 + n < N ? (int)(p0 + n) : -1;
        q[t] = (int)(r - n * (unsigned)words);
    }
    f(x, p, q);
}

__device__ __forceinline__ void plain_copy(int c, PlainCopy a, const PlainCopy& b)
{
    const int na = plain_ctas(a);
    if (c >= na) {
        c -= na;
        a = b;
    }
    uint32_t x[RW];
#pragma unroll
    for (int t = 0; t < RW; ++t) {
        const int e = (c * RW + t) * 256 + (int)threadIdx.x;
        x[t] = e < a.n ? a.src[e] : 0u;
    }
#pragma unroll
    for (int t = 0; t < RW; ++t) {
        const int e = (c * RW + t) * 256 + (int)threadIdx.x;
        if (e < a.n) a.dst[e] = x[t];
    }
}

__global__ void __launch_bounds__(256) k_copies(PlainCopy a, PlainCopy b) { plain_copy((int)blockIdx.x, a, b); }

// (the objectives and ranks that go out with the rows are copied by further
// CTAs of the same launch: a copy node of their own each took 1.5 us)
template <class T>
__global__ void __launch_bounds__(256) k_rows_out(RunView v, const int32_t* idx, T* dst, int words, int ctas, PlainCopy a,
                                                  PlainCopy b)
{
    if ((int)blockIdx.x >= ctas) {
        plain_copy((int)blockIdx.x - ctas, a, b);
        return;
    }
    constexpr int R = row_words<T>();
    for_row_words<T, R>(v.N, words, [&](T(&x)[R], int(&p)[R], int(&q)[R]) {
#pragma unroll
        for (int t = 0; t < R; ++t)
            if (p[t] >= 0) x[t] = reinterpret_cast<const T*>(v.X)[(size_t)idx[p[t]] * words + q[t]];
#pragma unroll
        for (int t = 0; t < R; ++t)
            if (p[t] >= 0) dst[(size_t)p[t] * words + q[t]] = x[t];
    });
}

// new parents take the rows of the last variation's parents, so that its
// children stay readable; the next children take the last ones' rows
template <class T>
__global__ void __launch_bounds__(256) k_rows_in(RunView v, const T* src, int words, int ctas, PlainCopy a, PlainCopy b)
{
    if ((int)blockIdx.x >= ctas) {
        plain_copy((int)blockIdx.x - ctas, a, b);
        return;
    }
    constexpr int R = row_words<T>();
    for_row_words<T, R>(v.N, words, [&](T(&x)[R], int(&p)[R], int(&q)[R]) {
#pragma unroll
        for (int t = 0; t < R; ++t)
            if (p[t] >= 0) x[t] = src[(size_t)p[t] * words + q[t]];
#pragma unroll
        for (int t = 0; t < R; ++t)
            if (p[t] >= 0) {
                const int slot = v.pold[p[t]];
                reinterpret_cast<T*>(v.X)[(size_t)slot * words + q[t]] = x[t];
                if (q[t] == 0) {
                    v.pcan[p[t]] = slot;
                    v.fslot[p[t]] = v.cslot[p[t]];
                }
            }
    });
}

__global__ void k_slots_init(RunView v)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= v.N) return;
    v.pcan[p] = v.pold[p] = p;
    v.fslot[p] = v.cslot[p] = v.N + p;
}

__global__ void k_nan_pad(RunView v)
{
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)v.n2 * v.m + t0; e < (long long)v.ld * v.m; e += stride) v.F[e] = __int_as_float(0x7fc00000);
    for (long long e = (long long)v.n2 * v.fs + t0; e < (long long)v.ld * v.fs; e += stride)
        v.Fp[e] = __int_as_float(0x7fc00000);
    for (int p = v.n2 + blockIdx.x * blockDim.x + threadIdx.x; p < v.ld; p += gridDim.x * blockDim.x)
        v.skey[p] = 0xffffffffu;
}

// the wait self-test: one thread waits, with the barriers' bounded wait, for
// a word nothing sets
__global__ void k_wait_probe(RunView v)
{
    if (threadIdx.x != 0) return;
    Ctrl* c = v.ctrl;
    bounded_wait(c, v.wait_ns, [&] { return ld_acquire(&c->never) != 0u; });
}

}  // namespace

cudaError_t launch_wait_probe(const RunView& v, cudaStream_t s)
{
    k_wait_probe<<<1, 32, 0, s>>>(v);
    return cudaGetLastError();
}

cudaError_t launch_check_finite(const RunView& v, cudaStream_t s)
{
    long long n = (long long)v.n2 * v.m;
    long long blocks = (n + 255) / 256;
    if (blocks > 1024) blocks = 1024;
    k_check_finite<<<(unsigned)blocks, 256, 0, s>>>(v);
    return cudaGetLastError();
}

cudaError_t launch_mark(const RunView& v, cudaStream_t s)
{
    k_mark<<<(v.NW + 31) / 32, 1024, 0, s>>>(v);
    return cudaGetLastError();
}

cudaError_t launch_select_out(const RunView& v, cudaStream_t s)
{
    k_gather<<<v.ld / GB, GB, 0, s>>>(v, GATHER_SEL);
    return cudaGetLastError();
}

cudaError_t launch_gather(const RunView& v, cudaStream_t s)
{
    const bool wide = v.m > NSGA3_FAST_M;
    k_gather<<<v.ld / GB, GB, 0, s>>>(v, wide ? GATHER_INDEX : GATHER_POP);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !wide) return e;
    k_gather_rows<<<(unsigned)(((long long)v.N * 32 + 255) / 256), 256, 0, s>>>(v);
    return cudaGetLastError();
}

// 16-, 8- or 4-byte words: what the row width and the caller's address allow
static int word_bytes(int d, const void* p)
{
    const uintptr_t a = reinterpret_cast<uintptr_t>(p) | (uintptr_t)d * 4;
    return (a & 15) == 0 ? 16 : (a & 7) == 0 ? 8 : 4;
}

template <class T>
static unsigned row_ctas(int N, int words)
{
    const int per = 256 * row_words<T>();
    return (unsigned)(((long long)N * words + per - 1) / per);
}

template <class T>
static cudaError_t rows_out(const RunView& v, const int32_t* idx, float* dst, PlainCopy a, PlainCopy b, cudaStream_t s)
{
    const int words = v.d * 4 / (int)sizeof(T);
    const unsigned ctas = row_ctas<T>(v.N, words);
    k_rows_out<T><<<ctas + plain_ctas(a) + plain_ctas(b), 256, 0, s>>>(v, idx, reinterpret_cast<T*>(dst), words, (int)ctas,
                                                                       a, b);
    return cudaGetLastError();
}

template <class T>
static cudaError_t rows_in(const RunView& v, const float* src, PlainCopy a, PlainCopy b, cudaStream_t s)
{
    const int words = v.d * 4 / (int)sizeof(T);
    const unsigned ctas = row_ctas<T>(v.N, words);
    k_rows_in<T><<<ctas + plain_ctas(a) + plain_ctas(b), 256, 0, s>>>(v, reinterpret_cast<const T*>(src), words, (int)ctas, a,
                                                                      b);
    return cudaGetLastError();
}

cudaError_t launch_rows_out(const RunView& v, const int32_t* idx, float* dst, PlainCopy a, PlainCopy b, cudaStream_t s)
{
    const int bytes = word_bytes(v.d, dst);
    if (bytes == 16) return rows_out<float4>(v, idx, dst, a, b, s);
    return bytes == 8 ? rows_out<float2>(v, idx, dst, a, b, s) : rows_out<float>(v, idx, dst, a, b, s);
}

cudaError_t launch_copies(PlainCopy a, PlainCopy b, cudaStream_t s)
{
    const int g = plain_ctas(a) + plain_ctas(b);
    if (g == 0) return cudaSuccess;
    k_copies<<<g, 256, 0, s>>>(a, b);
    return cudaGetLastError();
}

cudaError_t launch_rows_in(const RunView& v, const float* src, PlainCopy a, PlainCopy b, cudaStream_t s)
{
    const int bytes = word_bytes(v.d, src);
    if (bytes == 16) return rows_in<float4>(v, src, a, b, s);
    return bytes == 8 ? rows_in<float2>(v, src, a, b, s) : rows_in<float>(v, src, a, b, s);
}

cudaError_t launch_slots_init(const RunView& v, cudaStream_t s)
{
    k_slots_init<<<(v.N + 255) / 256, 256, 0, s>>>(v);
    return cudaGetLastError();
}

cudaError_t launch_nan_pad(const RunView& v, cudaStream_t s)
{
    k_nan_pad<<<64, 256, 0, s>>>(v);
    return cudaGetLastError();
}

