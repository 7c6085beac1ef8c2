// k_small.cu -- one generation (or one selection) of a small population in
// one launch of one thread-block cluster (Alg. 1 and Alg. 2 whole).
//
// At N = 92 the general path runs 21 dependent kernels of 2-30 us each: every
// one waits for its predecessor's writes, walks a chain of global loads and
// leaves most of the chip idle (110 us a generation).  Here the merged
// objectives live in every CTA's shared memory, a CTA owns the columns of a
// few 32-member words, and the phases meet at cluster barriers:
//   variation (a warp per pair) | dominance words of the owned columns,
//   fronts peeled with the front words stored to every CTA | ideal point
//   (each CTA for itself), extreme points of the owned members | intercepts
//   (each CTA for itself), association of the owned members | niche
//   selection in CTA 0 | next population.
// Every decision is the general path's: the same FP64 operation sequences
// (normalize.cuh, associate.cuh), the same priorities, ties to the lowest
// index.  What bounds it: the latency of the chain (FP64 divisions and square
// roots, barriers) and, from N of a few hundred, the pair tests on 8 or 16 SMs.
// Measured per generation, general path -> here: m = 3, N = 92 91 -> 31 us;
// m = 5, N = 500 103 -> 44; m = 8, N = 1,000 113 -> 73; m = 10, N = 1,000
// 122 -> 82 (20 generations and reading the population); selections of
// N = 1,024 with 2 to 35 directions 108-185 -> 47-89.  The limits (SMALL_N2,
// SMALL_W) lie where the objectives, the dominance words and the niche arrays
// still fit one CTA's shared memory.
#include "associate.cuh"
#include "kernels.cuh"
#include "niche.cuh"
#include "normalize.cuh"
#include "variation.cuh"

namespace {

constexpr int ST = 512;        // threads per CTA
constexpr int SWARPS = ST / 32;
constexpr int SCMAX = 16;      // CTAs per cluster at most
constexpr int SWORDS = SMALL_N2 / 32;
constexpr int SCOLS = 128;     // columns per CTA at most
constexpr int SCAND = 8;       // candidate slots per owned column (pooled over the CTA)
constexpr int SBINS = 512;     // bins of the reference-key histogram (top 9 bits)
constexpr int SKEYS = 64;      // keys of one bin ranked in shared memory
constexpr int SLEV = (SMALL_N2 + 1 + ST - 1) / ST;  // niche levels per thread

__device__ __forceinline__ void cluster_arrive()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync()
{
    cluster_arrive();
    cluster_wait();
}
// address of the same shared variable in CTA r of the cluster, and stores to it
__device__ __forceinline__ uint32_t peer(const void* p, int r)
{
    uint32_t d;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(r));
    return d;
}
__device__ __forceinline__ void st_peer(uint32_t a, uint32_t x)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t a, unsigned long long x)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(x) : "memory");
}

// FP32 pairs: two differences in one instruction, each rounded once
__device__ __forceinline__ void sub2(unsigned long long a, unsigned long long b, uint32_t& lo, uint32_t& hi)
{
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(d));
}

// Dynamic shared memory: byte offsets of the arrays for a population.
struct SmallLayout {
    int wpc, colsP;  // words and columns per CTA
    uint32_t dist, own, pi, dom, big, bytes;
};

template <int M>
__host__ __device__ inline SmallLayout small_layout(int n2, int w, int C)
{
    constexpr int MP = (M + 1) & ~1;
    SmallLayout L;
    const int NWs = (n2 + 31) / 32;
    L.wpc = (NWs + C - 1) / C;
    L.colsP = L.wpc * 32;
    uint32_t at = 0;
    auto take = [&](uint32_t b) {
        const uint32_t o = at;
        at += (b + 15u) & ~15u;
        return o;
    };
    L.dist = take(8u * n2);  // CTA 0: distance of every member of T
    // owned members: ASF and nadir keys (2 M), then f' (M), |f'|, best
    // distance, its reference, u (M floats) and the candidates
    const uint32_t asf = 16u * M * L.colsP;
    const uint32_t ass = L.colsP * (8u * M + 16u + 4u * M + 4u) + (uint32_t)L.colsP * SCAND * 16u;
    L.own = take(asf > ass ? asf : ass);
    L.pi = take(4u * n2);    // CTA 0: nearest direction of every member of T, -1 outside
    L.dom = take(4u * NWs * L.colsP);
    const uint32_t F = 4u * n2 * MP;
    const uint32_t nich = 8u * w + 4u * (5u * w + 1u + (n2 + 2u) + 2u * n2 + SBINS) + 16u;
    L.big = take(F > nich ? F : nich);  // merged objectives; CTA 0 then the niche arrays
    L.bytes = at;
    return L;
}

struct SmallShared {
    uint32_t front[2][SWORDS];  // written by every CTA of the cluster
    unsigned long long ek[SCMAX][NSGA3_FAST_M], en[SCMAX][NSGA3_FAST_M];  // ... extreme keys, nadir keys
    int ei[SCMAX][NSGA3_FAST_M];                                          // ... extreme indices
    uint32_t sel[SWORDS];       // ... by CTA 0: selected members
    uint32_t rem[SWORDS], S[SWORDS], Fl[SWORDS];
    int rank[SCOLS], pos[SCOLS], flag[SCOLS], mem[SCOLS];
    double z[NSGA3_FAST_M], a[NSGA3_FAST_M], nad[NSGA3_FAST_M];
    float evec[NSGA3_FAST_M][NSGA3_FAST_M];
    sf64::Divisor da[NSGA3_FAST_M];  // the intercepts as divisors
    double A[NSGA3_FAST_M * (NSGA3_FAST_M + 1)];
    float z32[NSGA3_FAST_M], ia32[NSGA3_FAST_M];
    int ext[NSGA3_FAST_M];
    int scratch[40];
    unsigned long long key[SKEYS];
    int fs, nc, novf, Lstar, bin, before, nkey, fallback, longest;
};

// Dominance words of the owned columns, NC columns (colsP / NC apart) per
// thread and row word: a row's objectives come by broadcast loads, whose rate
// bounds the loop, so one load serves two columns where they come in pairs.
// The OR of the differences f_j - f_i has its sign bit set iff some f_i > f_j
// and is zero only for equal vectors (differences are never -0.0): i
// dominates j iff it is positive.  Finite objectives only.
template <int M, int NC>
__device__ __forceinline__ void dominance_words(const float* Fs, uint32_t* dom, int n2, int c0, int colsP)
{
    constexpr int MP = (M + 1) & ~1;
    const int NWs = (n2 + 31) / 32, half = colsP / NC;
    for (int t = threadIdx.x; t < NWs * half; t += ST) {
        const int I = t / half, cl = t - I * half;
        const int nr = min(32, n2 - I * 32);
        unsigned long long pj[NC][MP / 2];
        uint32_t word[NC];
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            const float* fj = Fs + min(c0 + cl + u * half, n2 - 1) * MP;
#pragma unroll
            for (int h = 0; h < MP / 2; ++h) pj[u][h] = reinterpret_cast<const unsigned long long*>(fj)[h];
            word[u] = 0u;
        }
        const unsigned long long* fr = reinterpret_cast<const unsigned long long*>(Fs + I * 32 * MP);
#pragma unroll 4
        for (int k = nr - 1; k >= 0; --k) {
            unsigned long long fi[MP / 2];
#pragma unroll
            for (int h = 0; h < MP / 2; ++h) fi[h] = fr[k * (MP / 2) + h];
#pragma unroll
            for (int u = 0; u < NC; ++u) {
                uint32_t acc = 0u;
#pragma unroll
                for (int h = 0; h < MP / 2; ++h) {
                    uint32_t lo, hi;
                    sub2(pj[u][h], fi[h], lo, hi);
                    acc |= lo | hi;
                }
                word[u] = __funnelshift_l(0u - acc, word[u], 1);
            }
        }
#pragma unroll
        for (int u = 0; u < NC; ++u) dom[I * colsP + cl + u * half] = word[u];
    }
}

// The same words where some objective is not finite (a caller's parents; equal
// infinities differ by NaN): i dominates j iff no f_i > f_j and some f_i < f_j.
__device__ __noinline__ void dominance_words_any(const float* Fs, uint32_t* dom, int m, int n2, int c0, int colsP)
{
    const int NWs = (n2 + 31) / 32, MP = (m + 1) & ~1;
    for (int t = threadIdx.x; t < NWs * colsP; t += ST) {
        const int I = t / colsP, cl = t - I * colsP;
        const float* fj = Fs + min(c0 + cl, n2 - 1) * MP;
        uint32_t word = 0u;
        for (int k = 0; k < min(32, n2 - I * 32); ++k) {
            const float* fi = Fs + (I * 32 + k) * MP;
            bool greater = false, less = false;
            for (int q = 0; q < m; ++q) {
                greater |= fi[q] > fj[q];
                less |= fi[q] < fj[q];
            }
            if (less && !greater) word |= 1u << k;
        }
        dom[I * colsP + cl] = word;
    }
}

// The members taken where some reference gives a part of a long list: all of
// F_l sorted by (reference, nearest first where rho = 0, priority, index),
// so that a member's place in its reference's order is its position.  Arrays
// as in the kernel; near_d and near_i (w each) are free, keys has a place per
// merged individual and may be the distances' own.
// Bound: the barriers of the sort's 66 steps at 2,048 members (about 10 us).
// Counting the members before each member, a thread per member, walks the
// list once per member: quicker while the list's length times a thread's
// members is below about 400 (SWALK), and 330 us for 2,048 members of one
// direction.  Selections of N = 1,024, m = 3 whose members share 3 directions
// (spread, all at one) took 147 and 401 us with it alone, 64 and 64 now; N = 300,
// m = 3, 3 directions 66 us where all are at one, 33 now.
constexpr int SWALK = 384;

__device__ __noinline__ void pick_sorted(int n, int w, const int* bkt, const uint32_t* prio, const int* pi, const int* rho,
                                         const int* off, const int* take, const unsigned long long* dist,
                                         unsigned long long* near_d, int* near_i, unsigned long long* keys, uint32_t* sel)
{
    const int tid = threadIdx.x;
    for (int j = tid; j < w; j += ST) {
        near_d[j] = ~0ull;
        near_i[j] = 0x7fffffff;
    }
    __syncthreads();
    for (int e = tid; e < n; e += ST) {
        const int i = bkt[e], j = pi[i];
        // (few of the members of a long list find a smaller distance than they read)
        if (rho[j] == 0 && dist[i] < *(volatile unsigned long long*)&near_d[j]) atomicMin(&near_d[j], dist[i]);
    }
    __syncthreads();
    for (int e = tid; e < n; e += ST) {
        const int i = bkt[e], j = pi[i];
        if (rho[j] == 0 && dist[i] == near_d[j]) atomicMin(&near_i[j], i);
    }
    __syncthreads();
    static_assert(SMALL_N2 <= 2048, "an index takes 11 bits of a key");
    for (int e = tid; e < n; e += ST) {
        const int i = bkt[e], j = pi[i];
        keys[e] = (unsigned long long)j << 44 | (near_i[j] == i ? 0ull : 1ull << 43) | (unsigned long long)prio[e] << 11 | (unsigned)i;
    }
    __syncthreads();
    // bitonic merges whose first step compares mirrored places: every exchange
    // leaves the smaller key at the lower place, so places past n (the largest
    // keys) need not exist
    for (int k = 2; (k >> 1) < n; k <<= 1)
        for (int o = k >> 1; o > 0; o >>= 1) {
            for (int t = tid; 2 * (t - (t & (o - 1))) < n; t += ST) {
                const int a = 2 * t - (t & (o - 1));
                const int b = o == (k >> 1) ? (a ^ (k - 1)) : a + o;
                if (b < n) {
                    const unsigned long long x = keys[a], y = keys[b];
                    if (y < x) {
                        keys[a] = y;
                        keys[b] = x;
                    }
                }
            }
            __syncthreads();
        }
    for (int e = tid; e < n; e += ST) {
        const unsigned long long key = keys[e];
        const int j = (int)(key >> 44), i = (int)(key & 2047ull);
        if (e - off[j] < take[j]) atomicOr(&sel[i >> 5], 1u << (i & 31));
    }
}

// Selects (mode 0: objectives Fin, ranks and indices out) or steps (mode 1:
// variation too; mode 2: the merged individuals are in v.F already).
template <int M>
__global__ void __launch_bounds__(ST, 1) k_small(RunView v, int mode, int C, const float* Fin, int32_t* ranks, int32_t* selected)
{
    constexpr int MP = (M + 1) & ~1;
    constexpr int M4 = (M + 3) & ~3;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ SmallShared sh;
    Ctrl* c = v.ctrl;
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const int rank = blockIdx.x;  // one cluster
    const int n2 = v.n2, N = v.N, w = v.w, NWs = (n2 + 31) / 32;
    const SmallLayout L = small_layout<M>(n2, w, C);
    const int wpc = L.wpc, colsP = L.colsP;
    const int c0 = rank * colsP;                          // first owned column
    const int cols = max(0, min(n2 - c0, colsP));         // owned columns
    unsigned long long* dist0 = reinterpret_cast<unsigned long long*>(dyn + L.dist);
    int* pi0 = reinterpret_cast<int*>(dyn + L.pi);
    uint32_t* dom = reinterpret_cast<uint32_t*>(dyn + L.dom);
    float* Fs = reinterpret_cast<float*>(dyn + L.big);
    // A peer's shared memory may be written once that CTA is known to have
    // started: without the variation's cluster barrier the CTAs arrive here and
    // wait before the first front's words, the pair tests in between.
    if (mode != 1) cluster_arrive();
    const uint32_t gen = c->gen;
    const int status = read_status(c);
    if (rank == 0 && tid == 0) {  // as k_sel_reset leaves it
        c->cum = c->nS = c->K = c->nFl = c->need_niche = c->fallback = c->passes = 0;
        c->l = c->Lstar = -1;
        c->nT = c->rlev = c->nsel = c->overflow = c->recheck_miss = c->nlarge = c->ntile = 0;
        c->npath = c->peel_rows = 0u;
        for (int t = 0; t < 8; ++t) c->domstat[t] = 0ull;
    }
    if (status == 0 && mode == 1) {
        for (int q = rank * SWARPS + warp; q < N / 2; q += C * SWARPS) vary_eval_pair<M, true>(v, q, gen);
        cluster_sync();  // merged objectives and rows
    }
    const float* Fg = mode == 0 ? Fin : v.F;
    bool odd = false;  // some objective is not finite, or status (whose load these do not wait for)
    for (int e = tid; e < n2 * M; e += ST) {
        const int p = e / M, q = e - p * M;
        const float x = __ldcg(Fg + e);
        odd |= !isfinite(x);
        Fs[p * MP + q] = x + 0.0f;  // -0.0 as +0.0
    }
    odd |= status != 0;
    if (M & 1)  // the pad of an odd row
        for (int p = tid; p < n2; p += ST) Fs[p * MP + M] = 0.0f;
    if (tid < NWs) {
        const int lo = tid * 32;
        sh.rem[tid] = lo + 32 <= n2 ? 0xffffffffu : (1u << (n2 - lo)) - 1u;
        sh.S[tid] = sh.Fl[tid] = 0u;
    }
    if (tid < colsP) {
        sh.rank[tid] = -1;
        sh.flag[tid] = 0;
    }
    for (int i = tid; i < n2; i += ST) pi0[i] = -1;
    odd = __syncthreads_or(odd);  // the same in every CTA: each reads every objective
    if (odd && (mode == 0 || status != 0)) {
        __syncwarp();
        if (mode != 1) cluster_wait();
        if (tid < cols) ranks[c0 + tid] = -1;
        if (status == 0 && rank == 0 && tid == 0) set_status(c, DEV_ENONFINITE);
        return;
    }

    // ---- dominance: word I of column j = rows 32 I .. 32 I + 31 that dominate j
    if (__builtin_expect(odd, 0))
        dominance_words_any(Fs, dom, M, n2, c0, colsP);
    else if (wpc & 1)
        dominance_words<M, 1>(Fs, dom, n2, c0, colsP);
    else
        dominance_words<M, 2>(Fs, dom, n2, c0, colsP);
    __syncthreads();
    if (mode != 1) cluster_wait();

    // ---- fronts: an unranked column without an unranked dominator is ranked
    int cum = 0, l = -1, passes = 0, nS = 0, nFl = 0;
    {
        const int G = ST / colsP, g = tid / colsP, cl = tid - g * colsP;
        for (int k = 0;; ++k) {
            if (g < G && cl < cols && sh.rank[cl] < 0) {
                uint32_t any = 0u;
                for (int I = g; I < NWs; I += G) any |= dom[I * colsP + cl] & sh.rem[I];
                if (any) sh.flag[cl] = k + 1;
            }
            __syncthreads();
            if (warp < wpc) {
                const int cw = warp * 32 + lane;
                const bool nf = cw < cols && sh.rank[cw] < 0 && sh.flag[cw] != k + 1;
                const uint32_t word = __ballot_sync(0xffffffffu, nf);
                if (nf) sh.rank[cw] = k;
                const int wd = rank * wpc + warp;
                if (lane < C && wd < NWs) st_peer(peer(&sh.front[k & 1][wd], lane), word);
            }
            cluster_sync();
            // every warp counts the front and takes it out of rem for itself
            // (all write the same words, so none waits for another)
            int fs = 0;
            for (int I = lane; I < NWs; I += 32) {
                const uint32_t f = sh.front[k & 1][I];
                sh.rem[I] &= ~f;
                fs += __popc(f);
            }
            fs = __reduce_add_sync(0xffffffffu, fs);
            __syncwarp();  // rem is read by other lanes
            const int ncum = cum + fs;
            const bool first = l < 0 && ncum >= N;
            if (l < 0) {  // S: fronts before the selecting one, F_l: that one
                for (int I = tid; I < NWs; I += ST) {
                    if (first)
                        sh.Fl[I] = sh.front[k & 1][I];
                    else
                        sh.S[I] |= sh.front[k & 1][I];
                }
            }
            if (first) {
                l = k;
                nS = cum;
                nFl = fs;
            }
            cum = ncum;
            passes = k + 1;
            if (fs == 0 && ncum < n2) {  // an invariant failed (not expected): the same in every CTA
                if (rank == 0 && tid == 0) set_status(c, DEV_EINTERNAL);
                cluster_sync();
                return;
            }
            if (!(ncum < n2 && (v.full_sort || l < 0))) break;
        }
    }
    __syncthreads();
    if (tid < cols) ranks[c0 + tid] = sh.rank[tid];
    const int K = N - nS;
    const bool niche = K < nFl;
    if (rank == 0 && tid == 0) {
        c->cum = cum;
        c->passes = passes;
        c->passes_total += (unsigned long long)passes;
        c->peel_rows = (unsigned)((passes - 1) * NWs);
        c->l = l;
        c->nS = nS;
        c->nFl = nFl;
        c->K = K;
        c->need_niche = niche ? 1 : 0;
        c->nT = niche ? nS + nFl : 0;
        c->domstat[4] = (unsigned long long)NWs * (NWs + 1) / 2;
        c->domstat[6] = (unsigned long long)n2 * n2;
        c->domstat[7] = c->domstat[6];
    }
    if (niche) {
        if (__builtin_expect(odd, 0)) {
            // a member of T that is not finite (a NaN anywhere would enter the
            // running ideal point) ends the selection, as not_finite_key does
            // on the general path; no store into a peer is under way
            bool bad = false;
            for (int e = tid; e < n2 * M; e += ST) {
                const int p = e / M;
                const float x = Fs[p * MP + e - p * M];
                bad |= (((sh.S[p >> 5] | sh.Fl[p >> 5]) >> (p & 31)) & 1u) ? !isfinite(x) : v.norm_history && isnan(x);
            }
            if (__syncthreads_or(bad)) {  // the same in every CTA
                if (rank == 0 && tid == 0) set_status(c, DEV_ENONFINITE);
                return;
            }
        }
        // ---- ideal point: a warp per objective, every CTA for itself
        const bool hist = v.norm_history && c->hvalid;
        if (warp < M) {
            uint32_t o = 0xffffffffu;
            for (int I = 0; I < NWs; ++I) {
                const int i = I * 32 + lane;
                const uint32_t T = sh.S[I] | sh.Fl[I];
                if (i < n2 && (v.norm_history || ((T >> lane) & 1u))) o = min(o, f2ord(Fs[i * MP + warp]));
            }
            o = __reduce_min_sync(0xffffffffu, o);
            if (hist) o = min(o, f2ord((float)c->hz[warp]));
            if (lane == 0) sh.z[warp] = __dadd_rn((double)ord2f(o), 0.0);
        }
        __syncthreads();
        // ---- extreme points of the owned members (see k_norm_extreme)
        unsigned long long* ak = reinterpret_cast<unsigned long long*>(dyn + L.own);  // M x colsP
        unsigned long long* nk = ak + M * colsP;
        const uint32_t Tw = tid < colsP && c0 + tid < n2 ? (sh.S[(c0 + tid) >> 5] | sh.Fl[(c0 + tid) >> 5]) : 0u;
        const bool inT = (Tw >> lane) & 1u;
        if (tid < colsP) {
            double ft[M];
            unsigned long long m1 = 0ull, m2 = 0ull;
            int r1 = 0;
            const int i = min(c0 + tid, n2 - 1);
#pragma unroll
            for (int r = 0; r < M; ++r) {
                ft[r] = __dsub_rn((double)Fs[i * MP + r], sh.z[r]);
                const unsigned long long kr = okey(ft[r]);
                if (kr > m1) {
                    m2 = m1;
                    m1 = kr;
                    r1 = r;
                } else if (kr > m2) {
                    m2 = kr;
                }
            }
            const sf64::Divisor micro = sf64::divisor(1e-6);
            unsigned long long k1, k2 = m1;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {  // (one copy of the division's code)
                k1 = k2;
                k2 = okey(sf64::div(__longlong_as_double((long long)(h ? m2 : m1)), micro));
            }
#pragma unroll
            for (int q = 0; q < M; ++q) {
                const unsigned long long other = q == r1 ? k2 : k1, kq = okey(ft[q]);
                ak[q * colsP + tid] = inT ? (kq > other ? kq : other) : ~0ull;
                nk[q * colsP + tid] = inT ? kq : 0ull;
            }
        }
        __syncthreads();
        if (warp < M) {
            unsigned long long b = ~0ull, n = 0ull;
            int bi = 0x7fffffff;
            for (int e = lane; e < colsP; e += 32) {
                const unsigned long long x = ak[warp * colsP + e];
                if (x != ~0ull && key_less(x, c0 + e, b, bi)) {
                    b = x;
                    bi = c0 + e;
                }
                n = max(n, nk[warp * colsP + e]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long ob = __shfl_xor_sync(0xffffffffu, b, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                const unsigned long long on = __shfl_xor_sync(0xffffffffu, n, o);
                if (key_less(ob, oi, b, bi)) {
                    b = ob;
                    bi = oi;
                }
                n = max(n, on);
            }
            if (lane < C) {
                st_peer(peer(&sh.ek[rank][warp], lane), b);
                st_peer(peer(&sh.en[rank][warp], lane), n);
                st_peer(peer(&sh.ei[rank][warp], lane), (uint32_t)bi);
            }
        }
        cluster_sync();
        // ---- intercepts: one warp, every CTA for itself
        if (warp == 0) {
            if (lane < M) {
                unsigned long long b = sh.ek[0][lane], n = sh.en[0][lane];
                int bi = sh.ei[0][lane];
                for (int r = 1; r < C; ++r) {
                    if (key_less(sh.ek[r][lane], sh.ei[r][lane], b, bi)) {
                        b = sh.ek[r][lane];
                        bi = sh.ei[r][lane];
                    }
                    n = max(n, sh.en[r][lane]);
                }
                if (hist)  // the remembered extreme vectors are candidates 2N + r
                    for (int r = 0; r < M; ++r) {
                        double mx = 0.0, tq = 0.0;
#pragma unroll
                        for (int t = 0; t < M; ++t) {
                            const double ft = __dsub_rn((double)v.he[r * M + t], sh.z[t]);
                            if (t == lane)
                                tq = ft;
                            else if (ft > mx)
                                mx = ft;
                        }
                        const unsigned long long kq = okey(tq), ko = okey(__ddiv_rn(mx, 1e-6));
                        const unsigned long long asf = kq > ko ? kq : ko;
                        if (key_less(asf, n2 + r, b, bi)) {
                            b = asf;
                            bi = n2 + r;
                        }
                    }
                sh.ext[lane] = bi;
                sh.nad[lane] = __longlong_as_double((long long)n);
            }
            __syncwarp();
            const int er = sh.ext[lane < M ? lane : 0];
            bool ok = __all_sync(0xffffffffu, er >= 0 && er < n2 + (hist ? M : 0));
#pragma unroll 1
            for (int e = lane; e < M * M; e += 32) {
                const int r = e / M, q = e - r * M, x = sh.ext[r];
                const float f = !ok ? 0.0f : x < n2 ? Fs[x * MP + q] : v.he[(x - n2) * M + q];
                sh.evec[r][q] = f;
                sh.A[r * (M + 1) + q] = ok ? __dsub_rn((double)f, sh.z[q]) : 0.0;
            }
            if (lane < M) sh.A[lane * (M + 1) + M] = 1.0;
            double a = 0.0;
            ok = solve_rows(M, sh.A, ok, a);
            if (lane < M) {
                const double al = ok ? a : sf64::is_zero(sh.nad[lane]) ? 1.0 : sh.nad[lane];
                sh.a[lane] = al;
                sh.da[lane] = sf64::divisor(al);
                sh.z32[lane] = (float)sh.z[lane];
                sh.ia32[lane] = __frcp_rn((float)al);
            }
            if (lane == 0) sh.fallback = ok ? 0 : 1;
        }
        // ---- association of the owned members
        if (tid == 0) sh.nc = sh.novf = 0;
        int nm = 0;  // owned members of T, compacted
        for (int t = 0; t < wpc; ++t) {
            const int wd = rank * wpc + t;
            const uint32_t T = wd < NWs ? (sh.S[wd] | sh.Fl[wd]) : 0u;
            if (tid >= t * 32 && tid < t * 32 + 32 && inT) sh.mem[nm + __popc(T & ((1u << lane) - 1u))] = tid;
            nm += __popc(T);
        }
        __syncthreads();
        double* fp = reinterpret_cast<double*>(dyn + L.own);  // colsP x M
        double* nf = fp + colsP * M;
        unsigned long long* bd = reinterpret_cast<unsigned long long*>(nf + colsP);
        unsigned long long* cd = bd + colsP;                                 // candidates: distance
        int2* cand = reinterpret_cast<int2*>(cd + colsP * SCAND);            // ... (member, direction)
        int* bj = reinterpret_cast<int*>(cand + colsP * SCAND);
        float* us = reinterpret_cast<float*>(bj + colsP);                    // colsP x M
        for (int e = tid; e < nm * M; e += ST) {
            const int p = e / M, q = e - p * M;
            fp[e] = sf64::div(__dsub_rn((double)Fs[(c0 + sh.mem[p]) * MP + q], sh.z[q]), sh.da[q]);
        }
        __syncthreads();
        for (int p = tid; p < nm; p += ST) {
            double ss = 0.0;
#pragma unroll
            for (int q = 0; q < M; ++q) ss = __dadd_rn(ss, __dmul_rn(fp[p * M + q], fp[p * M + q]));
            const double x = sf64::sqrt_rn(ss);
            const bool zero = sf64::is_zero(x);
            nf[p] = x;
            float u[M];
            if (!unit32<M>(Fs + (c0 + sh.mem[p]) * MP, sh.z32, sh.ia32, u)) {
                const double inv = zero ? 0.0 : 1.0 / x;
#pragma unroll
                for (int q = 0; q < M; ++q) u[q] = __double2float_rn(fp[p * M + q] * inv);
            }
#pragma unroll
            for (int q = 0; q < M; ++q) us[p * M + q] = u[q];
            // |f'| = 0: every distance is 0, the first direction
            bd[p] = zero ? 0ull : ~0ull;
            bj[p] = zero ? 0 : 0x7fffffff;
        }
        __syncthreads();
        // FP32 cosines, a lane per direction, four members per warp pass;
        // each lane keeps its best direction and its second-best cosine
        const float band = cos_band<M>();
        const int cap = colsP * SCAND;
        for (int p0 = warp * 4; p0 < nm; p0 += SWARPS * 4) {
            float u[4][M], b1[4], b2[4];
            int j1[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int p = min(p0 + t, nm - 1);
#pragma unroll
                for (int q = 0; q < M; ++q) u[t][q] = us[p * M + q];
                b1[t] = b2[t] = -1.0f;
                j1[t] = -1;
            }
            auto dots = [&](int j, float (&qd)[4]) {
                const float4* z4 = reinterpret_cast<const float4*>(v.Zh + (size_t)j * M4);
                float z[M4];
#pragma unroll
                for (int q4 = 0; q4 < M4 / 4; ++q4) {
                    const float4 x = __ldg(z4 + q4);
                    z[4 * q4 + 0] = x.x;
                    z[4 * q4 + 1] = x.y;
                    z[4 * q4 + 2] = x.z;
                    z[4 * q4 + 3] = x.w;
                }
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    float s = 0.0f;
#pragma unroll
                    for (int q = 0; q < M; ++q) s = fmaf(u[t][q], z[q], s);
                    qd[t] = s;
                }
            };
#pragma unroll 2
            for (int j = lane; j < w; j += 32) {
                float qd[4];
                dots(j, qd);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const bool up = qd[t] > b1[t];
                    b2[t] = fmaxf(b2[t], up ? b1[t] : qd[t]);
                    j1[t] = up ? j : j1[t];
                    b1[t] = fmaxf(b1[t], qd[t]);
                }
            }
            float thr[4];
            unsigned again = 0u;  // members whose other directions of this lane may be in the band
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const float best = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(b1[t], 0.0f))));
                thr[t] = best - band;
                if (p0 + t >= nm || bd[min(p0 + t, nm - 1)] == 0ull) continue;
                if (j1[t] >= 0 && b1[t] >= thr[t]) {
                    const int e = atomicAdd(&sh.nc, 1);
                    if (e < cap)
                        cand[e] = make_int2(p0 + t, j1[t]);
                    else
                        atomicAdd(&sh.novf, 1);
                    if (b2[t] >= thr[t]) again |= 1u << t;
                }
            }
            if (again)
                for (int j = lane; j < w; j += 32) {
                    float qd[4];
                    dots(j, qd);
#pragma unroll
                    for (int t = 0; t < 4; ++t)
                        if (((again >> t) & 1u) && j != j1[t] && qd[t] >= thr[t]) {
                            const int e = atomicAdd(&sh.nc, 1);
                            if (e < cap)
                                cand[e] = make_int2(p0 + t, j);
                            else
                                atomicAdd(&sh.novf, 1);
                        }
                }
        }
        __syncthreads();
        if (sh.novf == 0) {
            const int nc = sh.nc;
            for (int e = tid; e < nc; e += ST) {
                const int2 x = cand[e];
                const double d = perp_dist(fp + x.x * M, nf[x.x], v.Zd + (size_t)x.y * M, v.nz[x.y], M);
                cd[e] = (unsigned long long)__double_as_longlong(d);  // d >= 0: ordered like its bits
                atomicMin(&bd[x.x], cd[e]);
            }
            __syncthreads();
            for (int e = tid; e < nc; e += ST)
                if (cd[e] == bd[cand[e].x]) atomicMin(&bj[cand[e].x], cand[e].y);
        } else {
            // more near-equal directions than the CTA's slots: every direction
            // of every owned member in FP64, a warp per member
            for (int p = warp; p < nm; p += SWARPS) {
                unsigned long long b = ~0ull;
                int j0 = 0x7fffffff;
                for (int j = lane; j < w; j += 32) {
                    const double d = perp_dist(fp + p * M, nf[p], v.Zd + (size_t)j * M, v.nz[j], M);
                    const unsigned long long k = (unsigned long long)__double_as_longlong(d);
                    if (key_less(k, j, b, j0)) {
                        b = k;
                        j0 = j;
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long ob = __shfl_xor_sync(0xffffffffu, b, o);
                    const int oj = __shfl_xor_sync(0xffffffffu, j0, o);
                    if (key_less(ob, oj, b, j0)) {
                        b = ob;
                        j0 = oj;
                    }
                }
                if (lane == 0) {
                    bd[p] = b;
                    bj[p] = j0;
                }
            }
            if (tid == 0) atomicAdd(&c->overflow, nm);
        }
        __syncthreads();
        for (int p = tid; p < nm; p += ST) {
            const int i = c0 + sh.mem[p];
            // (finite members have a candidate; the bound keeps every index in range regardless)
            const int j = (int)min((unsigned)bj[p], (unsigned)(w - 1));
            v.pi[i] = j;
            v.dist[i] = __longlong_as_double((long long)bd[p]);
            st_peer(peer(&pi0[i], 0), (uint32_t)j);
            st_peer(peer(&dist0[i], 0), bd[p]);
        }
        cluster_sync();
        // ---- niche selection: CTA 0 (closed form: see k_niche.cu)
        if (rank == 0) {
            if (tid < M) {
                c->zstar[tid] = sh.z[tid];
                c->a[tid] = sh.a[tid];
                c->ext[tid] = sh.ext[tid];
                if (v.norm_history) {  // every CTA read the history before the last barrier
                    c->hz[tid] = sh.z[tid];
                    for (int q = 0; q < M; ++q) v.he[tid * M + q] = sh.evec[tid][q];
                }
                if (tid == 0) {
                    c->fallback = sh.fallback;
                    if (v.norm_history) c->hvalid = 1;
                }
            }
            unsigned long long* rkey = reinterpret_cast<unsigned long long*>(dyn + L.big);  // w
            int* rho = reinterpret_cast<int*>(rkey + w);
            int* rhop = rho + w;
            int* take = rhop + w;
            int* cur = take + w;
            int* off = cur + w;        // w + 1
            int* lev = off + w + 1;    // n2 + 2
            int* bkt = lev + n2 + 2;   // n2
            uint32_t* prio = reinterpret_cast<uint32_t*>(bkt + n2);  // n2
            int* bins = reinterpret_cast<int*>(prio + n2);           // SBINS
            for (int j = tid; j < w; j += ST) rho[j] = rhop[j] = cur[j] = 0;
            for (int t = tid; t < n2 + 2; t += ST) lev[t] = 0;
            for (int t = tid; t < SBINS; t += ST) bins[t] = 0;
            if (tid == 0) {
                sh.Lstar = 0x7fffffff;
                sh.nkey = sh.longest = 0;
            }
            const int rounds = (nFl + ST - 1) / ST;  // members per thread
            for (int I = tid; I < NWs; I += ST) sh.sel[I] = sh.S[I];
            __syncthreads();
            for (int i = tid; i < n2; i += ST) {
                const int j = pi0[i];
                if (j < 0) continue;
                atomicAdd(((sh.S[i >> 5] >> (i & 31)) & 1u) ? &rho[j] : &rhop[j], 1);
            }
            __syncthreads();
            for (int j = tid; j < w; j += ST)
                if (rhop[j] > 0) {
                    atomicAdd(&lev[rho[j]], 1);
                    atomicAdd(&lev[rho[j] + rhop[j]], -1);
                }
            __syncthreads();
            // count(L) = members of level <= L: prefix sums of the references
            // holding a level-L member
            {
                int loc[SLEV], s = 0, total;
#pragma unroll
                for (int t = 0; t < SLEV; ++t) {
                    const int lv = tid * SLEV + t;
                    s += lv <= n2 ? lev[lv] : 0;
                    loc[t] = s;
                }
                const int o1 = block_excl_scan(s, sh.scratch, &total);
                int s2 = 0;
#pragma unroll
                for (int t = 0; t < SLEV; ++t) {
                    s2 += loc[t] + o1;
                    loc[t] = s2;
                }
                const int o2 = block_excl_scan(s2, sh.scratch, &total);
                int my = 0x7fffffff;
#pragma unroll
                for (int t = SLEV - 1; t >= 0; --t) {
                    const int lv = tid * SLEV + t;
                    if (lv <= n2) {
                        lev[lv] = loc[t] + o2;
                        if (loc[t] + o2 >= K) my = lv;
                    }
                }
                my = __reduce_min_sync(0xffffffffu, my);
                if (lane == 0 && my != 0x7fffffff) atomicMin(&sh.Lstar, my);
                __syncthreads();
            }
            const int Ls = sh.Lstar;  // count(n2) = |F_l| >= K: always found
            const int r = K - (Ls > 0 ? lev[Ls - 1] : 0);
            // references holding a level-L* member: the r smallest keys take it
            for (int j = tid; j < w; j += ST) {
                const int rp = rhop[j], lo = rho[j];
                take[j] = rp > 0 ? min(rp, max(0, Ls - lo)) : 0;
                unsigned long long key = ~0ull;
                if (rp > 0 && lo <= Ls && Ls < lo + rp) {
                    key = ref_key(v.seed, gen, j);
                    atomicAdd(&bins[(int)(key >> 55)], 1);
                }
                rkey[j] = key;
            }
            __syncthreads();
            {
                static_assert(SBINS == ST, "a bin per thread");
                static_assert(SMALL_W < 65536 && SMALL_N2 < 32768, "both sums in one scan");
                // and the offsets of the references' member lists
                const int per = (w + ST - 1) / ST, lo = min(w, tid * per), hi = min(w, lo + per);
                const int x = bins[tid];
                int s = 0, most = 0, total;
                for (int j = lo; j < hi; ++j) {
                    s += rhop[j];
                    most = max(most, rhop[j]);
                }
                if (most * rounds > SWALK) sh.longest = 1;
                const int sums = block_excl_scan(x | (s << 16), sh.scratch, &total), before = sums & 0xffff;
                if (before < r && r <= before + x) {
                    sh.bin = tid;
                    sh.before = before;
                }
                int run = sums >> 16;
                for (int j = lo; j < hi; ++j) {
                    off[j] = run;
                    run += rhop[j];
                }
            }
            __syncthreads();
            {
                const int b = sh.bin, need = r - sh.before;
                for (int j = tid; j < w; j += ST) {
                    const unsigned long long key = rkey[j];
                    if (key == ~0ull || (int)(key >> 55) > b) continue;
                    if ((int)(key >> 55) < b) {
                        take[j] += 1;
                    } else {
                        const int p = atomicAdd(&sh.nkey, 1);
                        if (p < SKEYS) sh.key[p] = key;
                    }
                }
                __syncthreads();
                const int ne = sh.nkey;
                if (ne <= SKEYS) {
                    if (tid < ne) {
                        const unsigned long long key = sh.key[tid];
                        int rk = 0;
                        for (int t = 0; t < ne; ++t) rk += sh.key[t] < key;
                        if (rk < need) take[(int)(key & 0xffffffffull)] += 1;
                    }
                } else {  // (not expected for Philox priorities: about w / SBINS keys a bin)
                    for (int j = tid; j < w; j += ST) {
                        const unsigned long long key = rkey[j];
                        if (key == ~0ull || (int)(key >> 55) != b) continue;
                        int rk = 0;
                        for (int t = 0; t < w; ++t) rk += rkey[t] != ~0ull && (int)(rkey[t] >> 55) == b && rkey[t] < key;
                        if (rk < need) take[j] += 1;
                    }
                }
            }
            for (int i = tid; i < n2; i += ST) {
                const int j = pi0[i];
                if (j < 0 || !((sh.Fl[i >> 5] >> (i & 31)) & 1u)) continue;
                const int e = off[j] + atomicAdd(&cur[j], 1);
                bkt[e] = i;
                prio[e] = mem_prio(v.seed, gen, i);
            }
            __syncthreads();
            bool part = false;  // a part of a long list is taken
            if (__builtin_expect(sh.longest, 0)) {
                for (int j = tid; j < w; j += ST) part |= take[j] > 0 && take[j] < rhop[j] && rhop[j] * rounds > SWALK;
                part = __syncthreads_or(part);
            }
            if (__builtin_expect(part, 0)) {
                if (tid == 0) atomicOr(&c->npath, NPATH_LARGE);
                pick_sorted(nFl, w, bkt, prio, pi0, rho, off, take, dist0, rkey, cur, dist0, sh.sel);
            }
            // (else) a member is taken when fewer than take_j of its reference's
            // members come before it (nearest first when rho_j = 0)
            for (int e = part ? nFl : tid; e < nFl; e += ST) {
                const int i = bkt[e], j = pi0[i];
                const int tk = take[j], cnt = rhop[j];
                bool in = tk >= cnt;
                if (!in && tk > 0) {
                    const int lo = off[j];
                    int before = 0, near = i;
                    unsigned long long nd = dist0[i];
                    uint32_t np = prio[e];
                    const uint32_t mine = prio[e];
                    for (int t = lo; t < lo + cnt; ++t) {
                        const int o = bkt[t];
                        const uint32_t po = prio[t];
                        before += po < mine || (po == mine && o < i);
                        if (key_less(dist0[o], o, nd, near)) {
                            nd = dist0[o];
                            near = o;
                            np = po;
                        }
                    }
                    if (rho[j] == 0) {
                        if (near == i)
                            before = 0;
                        else  // the nearest comes first, wherever its priority stands
                            before += !(np < mine || (np == mine && near < i));
                    }
                    in = before < tk;
                    if (cnt > 32) atomicOr(&c->npath, NPATH_LARGE);
                }
                if (in) atomicOr(&sh.sel[i >> 5], 1u << (i & 31));
            }
            if (tid == 0) {
                c->Lstar = Ls;
                c->rlev = r;
            }
            __syncthreads();
            for (int t = tid; t < (C - 1) * NWs; t += ST) {
                const int rr = 1 + t / NWs, I = t - (rr - 1) * NWs;
                st_peer(peer(&sh.sel[I], rr), sh.sel[I]);
            }
        }
        cluster_sync();
    } else {
        for (int I = tid; I < NWs; I += ST) sh.sel[I] = sh.S[I] | sh.Fl[I];
        __syncthreads();
    }

    // ---- selected indices in ascending order, next population
    if (warp == 0) {
        int run = 0;
        for (int I0 = 0; I0 < NWs; I0 += 32) {
            const int I = I0 + lane;
            const int x = I < NWs ? __popc(sh.sel[I]) : 0;
            int inc = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (I < NWs) sh.rem[I] = (uint32_t)(run + inc - x);  // selected before word I
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) sh.fs = run;
    }
    __syncthreads();
    if (sh.fs != N) {  // an invariant failed (not expected): nothing is written
        if (rank == 0 && tid == 0) {
            c->nsel = sh.fs;
            set_status(c, DEV_EINTERNAL);
        }
        return;
    }
    if (tid < cols) {
        const int i = c0 + tid;
        const uint32_t word = sh.sel[i >> 5];
        const int p = (int)sh.rem[i >> 5] + __popc(word & ((1u << lane) - 1u));
        const bool in = (word >> lane) & 1u;
        sh.pos[tid] = in ? p : -1;
        if (in) selected[p] = i;
        if (mode != 0) {
            const int slot = i < N ? v.pold[i] : v.cslot[i - N];
            if (in) {
                v.pcan[p] = slot;
                v.rank[p] = sh.rank[tid];
            } else {
                v.fslot[i - p] = slot;
            }
        }
    }
    if (rank == 0 && tid == 0) {
        c->nsel = N;
        if (mode != 0) c->gen = gen + 1u;
    }
    if (mode == 0) return;
    __syncthreads();
    for (int e = tid; e < cols * M; e += ST) {
        const int cl = e / M, q = e - cl * M, p = sh.pos[cl];
        if (p >= 0) v.PF[(size_t)p * M + q] = __ldcg(v.F + (size_t)(c0 + cl) * M + q);
    }
}

// CTAs of the cluster: a 32-member word per CTA at least
int small_ctas(int n2)
{
    const int NWs = (n2 + 31) / 32;
    if (NWs > 16) return 16;
    return NWs > 4 ? 8 : NWs > 2 ? 4 : NWs > 1 ? 2 : 1;
}

// the one cluster of a launch
template <int M>
struct SmallConfig {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    const int C;
    SmallConfig(int n2, int w, cudaStream_t s) : C(small_ctas(n2))
    {
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(ST);
        cfg.dynamicSmemBytes = small_layout<M>(n2, w, C).bytes;
        cfg.stream = s;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = C;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
};

template <int M>
cudaError_t launch_m(const RunView& v, int mode, const float* F, int32_t* ranks, int32_t* sel, cudaStream_t s)
{
    const SmallConfig<M> c(v.n2, v.w, s);
    return cudaLaunchKernelEx(&c.cfg, k_small<M>, v, mode, c.C, F, ranks, sel);
}

template <int M>
bool fits_m(int n2, int w)
{
    const SmallConfig<M> c(n2, w, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_small<M>, &c.cfg) == cudaSuccess) return n > 0;
    cudaGetLastError();
    return false;
}

template <int M>
cudaError_t attr_m()
{
    const cudaError_t e = cudaFuncSetAttribute(k_small<M>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)small_layout<M>(SMALL_N2, SMALL_W, 16).bytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_small<M>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

}  // namespace

cudaError_t launch_small(const RunView& v, int mode, const float* F, int32_t* ranks, int32_t* sel, cudaStream_t s)
{
    switch (v.m) {
    case 2: return launch_m<2>(v, mode, F, ranks, sel, s);
    case 3: return launch_m<3>(v, mode, F, ranks, sel, s);
    case 4: return launch_m<4>(v, mode, F, ranks, sel, s);
    case 5: return launch_m<5>(v, mode, F, ranks, sel, s);
    case 6: return launch_m<6>(v, mode, F, ranks, sel, s);
    case 7: return launch_m<7>(v, mode, F, ranks, sel, s);
    case 8: return launch_m<8>(v, mode, F, ranks, sel, s);
    case 9: return launch_m<9>(v, mode, F, ranks, sel, s);
    case 10: return launch_m<10>(v, mode, F, ranks, sel, s);
    default: return cudaErrorInvalidValue;
    }
}

bool small_fits(int m, int n2, int w)
{
    switch (m) {
    case 2: return fits_m<2>(n2, w);
    case 3: return fits_m<3>(n2, w);
    case 4: return fits_m<4>(n2, w);
    case 5: return fits_m<5>(n2, w);
    case 6: return fits_m<6>(n2, w);
    case 7: return fits_m<7>(n2, w);
    case 8: return fits_m<8>(n2, w);
    case 9: return fits_m<9>(n2, w);
    case 10: return fits_m<10>(n2, w);
    default: return false;
    }
}

cudaError_t small_init_attributes()
{
    cudaError_t e = attr_m<2>();
    if (e == cudaSuccess) e = attr_m<3>();
    if (e == cudaSuccess) e = attr_m<4>();
    if (e == cudaSuccess) e = attr_m<5>();
    if (e == cudaSuccess) e = attr_m<6>();
    if (e == cudaSuccess) e = attr_m<7>();
    if (e == cudaSuccess) e = attr_m<8>();
    if (e == cudaSuccess) e = attr_m<9>();
    if (e == cudaSuccess) e = attr_m<10>();
    return e;
}
