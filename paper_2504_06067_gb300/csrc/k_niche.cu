// k_niche.cu -- niche selection of K = N - |S| members of F_l (the niching
// loop of Alg. 1; its cached batched form in Alg. 2).
//
// The paper's loop takes, round after round, one member from every
// reference of minimum niche count (the cache tensor Q and cursor s of
// Alg. 2 serve whole rounds at once) and truncates the last round in
// shuffled-reference order.  Rounds are exhausted level by level, so the
// outcome has a closed form that needs no loop:
//   each reference j orders its F_l members: the nearest first (min d, then
//   lowest index) when rho_j = 0, then by ascending Philox member priority
//   (then index); the member at position t has level rho_j + t;
//   L* = min { L : sum_j min(rho'_j, max(0, L + 1 - rho_j)) >= K };
//   every member of level < L* is taken, and of the references holding a
//   level-L* member, the r = K - count(L* - 1) of smallest (ref priority, j)
//   take that member.
// Random choices use fixed Philox priorities of this generation: reference
// j -> word 0 of Philox(j, gen, 4, 0), member i -> word 0 of
// Philox(i, gen, 5, 0); ties go to the lower index.
#include "kernels.cuh"
#include "niche.cuh"

namespace {

constexpr int LB = 1024;    // threads of the single-CTA kernels
constexpr int LCAP = 4096;  // niche levels resolved by the shared histogram
constexpr int EXACT = 1024; // candidates ranked pairwise in the last select phase
constexpr int CKCAP = 4096; // level-L* reference keys staged in shared memory
constexpr int RRCAP = 12288; // references whose (rho, rho') are staged in shared memory

// key of reference j: its priority (k_sort.cu writes them for the generation:
// one block forming up to 12 Philox values per thread here took 4 us), then j
__device__ __forceinline__ unsigned long long ref_key_of(const RunView& v, int j)
{
    return ((unsigned long long)v.rprio[j] << 32) | (unsigned)j;
}

// ------------------------------------------------ block-wide helpers -------
__device__ int block_sum(int x, int* scratch)
{
    x = warp_sum(x);
    if (lane_id() == 0) scratch[threadIdx.x >> 5] = x;
    __syncthreads();
    int t = 0;
    if (threadIdx.x < 32) {
        t = (threadIdx.x < (blockDim.x >> 5)) ? scratch[threadIdx.x] : 0;
        t = warp_sum(t);
        if (threadIdx.x == 0) scratch[32] = t;
    }
    __syncthreads();
    t = scratch[32];
    __syncthreads();
    return t;
}

// Exclusive scan of a[0..n) into out[0..n] (out[n] = total) by one block:
// each thread scans a contiguous run.
__device__ void block_scan_array(const int32_t* a, int32_t* out, int n, int* scratch)
{
    const int per = (n + (int)blockDim.x - 1) / (int)blockDim.x;
    const int lo = min(n, (int)threadIdx.x * per), hi = min(n, lo + per);
    int s = 0;
#pragma unroll 8
    for (int e = lo; e < hi; ++e) s += a[e];
    int total;
    int run = block_excl_scan(s, scratch, &total);
    for (int e = lo; e < hi; e += 8) {
        int x[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = a[min(e + t, hi - 1)];
#pragma unroll
        for (int t = 0; t < 8; ++t)
            if (e + t < hi) {
                out[e + t] = run;
                run += x[t];
            }
    }
    if (threadIdx.x == 0) out[n] = total;
}

struct SelShared {
    int hist[256];
    int scratch[40];
    unsigned long long keys[EXACT];
    int idxs[EXACT];
    int nex;
    int bsel;
    int before;
};

// Calls mark(idx) for the `need` smallest keys among {idx in [0,n) : pred}.
// Keys are unique 64-bit values.  8-bit radix passes narrow the candidates
// to one digit bucket until at most EXACT remain, which are then ranked
// pairwise.  Every thread of the block must call it.
template <class Key, class Pred, class Mark>
__device__ void block_select_smallest(int n, int need, Key key, Pred pred, Mark mark, SelShared& sh,
                                      unsigned* paths)
{
    unsigned long long prefix = 0ull, pmask = 0ull;
    int shift = 56;
    while (need > 0) {
        int cnt = 0;
        for (int e = threadIdx.x; e < n; e += blockDim.x)
            if (pred(e) && (key(e) & pmask) == prefix) ++cnt;
        cnt = block_sum(cnt, sh.scratch);
        if (cnt <= need) {  // every remaining candidate is taken
            for (int e = threadIdx.x; e < n; e += blockDim.x)
                if (pred(e) && (key(e) & pmask) == prefix) mark(e);
            return;
        }
        if (cnt <= EXACT || shift < 0) {
            if (threadIdx.x == 0) sh.nex = 0;
            __syncthreads();
            for (int e = threadIdx.x; e < n; e += blockDim.x) {
                if (pred(e)) {
                    unsigned long long k = key(e);
                    if ((k & pmask) == prefix) {
                        int p = atomicAdd(&sh.nex, 1);
                        if (p < EXACT) {
                            sh.keys[p] = k;
                            sh.idxs[p] = e;
                        }
                    }
                }
            }
            __syncthreads();
            const int ne = min(sh.nex, EXACT);
            for (int a = threadIdx.x; a < ne; a += blockDim.x) {
                const unsigned long long ka = sh.keys[a];
                int rk = 0;
                for (int b = 0; b < ne; ++b) rk += sh.keys[b] < ka;
                if (rk < need) mark(sh.idxs[a]);
            }
            __syncthreads();
            return;
        }
        if (paths && threadIdx.x == 0) atomicOr(paths, shift == 56 ? NPATH_RADIX : NPATH_RADIX2);
        for (int t = threadIdx.x; t < 256; t += blockDim.x) sh.hist[t] = 0;
        __syncthreads();
        for (int e = threadIdx.x; e < n; e += blockDim.x) {
            if (pred(e)) {
                unsigned long long k = key(e);
                if ((k & pmask) == prefix) atomicAdd(&sh.hist[(int)((k >> shift) & 255ull)], 1);
            }
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            // warp scan of the 256 bins (8 per lane): the bin where the running
            // count reaches `need`, and the count before it
            const int lane = threadIdx.x;
            int h8[8], loc = 0;
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                h8[t] = sh.hist[lane * 8 + t];
                loc += h8[t];
            }
            int inc = loc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            int run = inc - loc;
            const bool here = run < need && need <= inc;
            if (here) {
                int b = lane * 8;
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    if (run + h8[t] >= need) break;
                    run += h8[t];
                    ++b;
                }
                sh.bsel = b;
                sh.before = run;
            }
        }
        __syncthreads();
        const int b = sh.bsel, before = sh.before;
        for (int e = threadIdx.x; e < n; e += blockDim.x) {
            if (pred(e)) {
                unsigned long long k = key(e);
                if ((k & pmask) == prefix && (int)((k >> shift) & 255ull) < b) mark(e);
            }
        }
        __syncthreads();
        need -= before;
        prefix |= (unsigned long long)b << shift;
        pmask |= 255ull << shift;
        shift -= 8;
    }
}

// ------------------------------------------------------------ k_level ------
struct LevelShared {
    int lev[LCAP + 1], lev2[LCAP + 1];  // references whose levels begin, end there
    int scratch[40];
    int Lstar;
    int maxhi;
    int nck;
    SelShared sel;
    unsigned long long ck[CKCAP];
    int2 rr[RRCAP];        // (rho_j, rho'_j)
};

__global__ void __launch_bounds__(LB) k_level(RunView v)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    LevelShared& sh = *reinterpret_cast<LevelShared*>(smraw);
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int w = v.w, K = c->K;
    const bool staged = w <= RRCAP;
    if (staged) {
        // all loads of a thread in flight at once (one SM does this work)
        constexpr int PT = RRCAP / LB;
        int a[PT], b[PT];
#pragma unroll
        for (int t = 0; t < PT; ++t) {
            const int j = threadIdx.x + t * LB;
            a[t] = j < w ? v.rho[j] : 0;
            b[t] = j < w ? v.rhop[j] : 0;
        }
#pragma unroll
        for (int t = 0; t < PT; ++t) {
            const int j = threadIdx.x + t * LB;
            if (j < w) sh.rr[j] = make_int2(a[t], b[t]);
        }
    }
    auto rho_of = [&](int j) { return staged ? sh.rr[j].x : v.rho[j]; };
    auto rhop_of = [&](int j) { return staged ? sh.rr[j].y : v.rhop[j]; };
    // f(j, rho_j, rho'_j) for every reference, four pairs of loads in flight
    auto for_refs = [&](auto f) {
        for (int j0 = threadIdx.x; j0 < w; j0 += 4 * LB) {
            int a[4], b[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int j = min(j0 + t * LB, w - 1);
                a[t] = rho_of(j);
                b[t] = rhop_of(j);
            }
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (j0 + t * LB < w) f(j0 + t * LB, a[t], b[t]);
        }
    };
    for (int t = threadIdx.x; t <= LCAP; t += LB) sh.lev[t] = sh.lev2[t] = 0;
    if (threadIdx.x == 0) {
        sh.Lstar = LCAP;
        sh.maxhi = 0;
    }
    __syncthreads();
    int mymax = 0;
    {
        // most references share a few level values (rho_j = 0 when S is
        // empty): increments by one, which the shared-memory atomics take
        // together for the lanes of a warp (groups of equal lanes by
        // match_any: the kernel 14.1 us for 10,626 references, 12.5 so)
        for_refs([&](int, int lo, int rp) {
            if (rp > 0 && (lo < 0 || rp > v.n2)) {  // counts out of range: an invariant failed upstream
                set_status(c, DEV_EINTERNAL);
                rp = 0;
            }
            const int hi = lo + rp;
            if (rp > 0 && lo < LCAP) atomicAdd(&sh.lev[lo], 1);
            if (rp > 0 && hi < LCAP) atomicAdd(&sh.lev2[hi], 1);
            if (rp > 0) mymax = max(mymax, hi);
        });
    }
    mymax = __reduce_max_sync(0xffffffffu, mymax);
    if ((threadIdx.x & 31) == 0) atomicMax(&sh.maxhi, mymax);
    __syncthreads();
    // n(L) = prefix sum of the difference array; count(L) = prefix sum of n(L)
    {
        constexpr int PER = LCAP / LB;
        int loc[PER];
        int s = 0;
        for (int t = 0; t < PER; ++t) {
            s += sh.lev[threadIdx.x * PER + t] - sh.lev2[threadIdx.x * PER + t];
            loc[t] = s;
        }
        int total;
        int off = block_excl_scan(s, sh.scratch, &total);
        for (int t = 0; t < PER; ++t) loc[t] += off;  // n(L)
        int s2 = 0;
        for (int t = 0; t < PER; ++t) {
            s2 += loc[t];
            loc[t] = s2;
        }
        int off2 = block_excl_scan(s2, sh.scratch, &total);
        for (int t = 0; t < PER; ++t) {
            const int L = threadIdx.x * PER + t;
            sh.lev[L] = loc[t] + off2;  // count(L)
        }
        __syncthreads();
        // count(L) is non-decreasing: the first L of this thread with
        // count >= K, then one atomic per warp
        int myL = LCAP;
        for (int t = PER - 1; t >= 0; --t) {
            const int L = threadIdx.x * PER + t;
            if (sh.lev[L] >= K) myL = L;
        }
        myL = __reduce_min_sync(0xffffffffu, myL);
        if ((threadIdx.x & 31) == 0 && myL < LCAP) atomicMin(&sh.Lstar, myL);
        __syncthreads();
    }
    int Lstar = sh.Lstar;
    int before;
    if (Lstar < LCAP) {
        before = Lstar > 0 ? sh.lev[Lstar - 1] : 0;
    } else {
        // deep levels: binary search with block-reduced counts
        if (threadIdx.x == 0) atomicOr(&c->npath, NPATH_DEEP);
        auto count_le = [&](int L) {
            int s = 0;
            for (int j = threadIdx.x; j < w; j += LB) {
                const int rp = rhop_of(j);
                if (rp > 0) s += min(rp, max(0, L + 1 - rho_of(j)));
            }
            return block_sum(s, sh.scratch);
        };
        int lo = LCAP, hi = max(LCAP, sh.maxhi - 1);
        while (lo < hi) {
            const int mid = lo + (hi - lo) / 2;
            if (count_le(mid) >= K)
                hi = mid;
            else
                lo = mid + 1;
        }
        Lstar = lo;
        before = count_le(Lstar - 1);
    }
    const int r = K - before;
    if (staged) {
        // The r smallest (priority, j) keys among the level-L* references:
        // each thread keeps the keys of its references in registers; one
        // 12-bit radix pass over the priorities' top bits finds the bin
        // holding the r-th key (about nC / 4096 keys per bin), the keys below
        // it are taken and the bin is ranked pairwise.
        constexpr int PT = RRCAP / LB;
        static_assert(LCAP == 4 * LB, "histogram bins per thread");
        unsigned long long kk[PT];
#pragma unroll
        for (int t = 0; t < PT; ++t) {
            const int j = threadIdx.x + t * LB;
            kk[t] = ~0ull;
            if (j < w) {
                const int rp = sh.rr[j].y, lo = sh.rr[j].x;
                v.take[j] = rp > 0 ? min(rp, max(0, Lstar - lo)) : 0;
                if (rp > 0 && lo <= Lstar && Lstar < lo + rp) kk[t] = ref_key_of(v, j);
            }
        }
        __syncthreads();  // every thread has read `before` from the level table
        int* hist = sh.lev;
        for (int t = threadIdx.x; t < LCAP; t += LB) hist[t] = 0;
        __syncthreads();
#pragma unroll
        for (int t = 0; t < PT; ++t)
            if (kk[t] != ~0ull) atomicAdd(&hist[(int)(kk[t] >> 52)], 1);
        __syncthreads();
        {
            int h4[4], loc = 0;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                h4[t] = hist[threadIdx.x * 4 + t];
                loc += h4[t];
            }
            int total;
            int run = block_excl_scan(loc, sh.scratch, &total);
            if (run < r && r <= run + loc) {
                int b = threadIdx.x * 4;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    if (run + h4[t] >= r) break;
                    run += h4[t];
                    ++b;
                }
                sh.sel.bsel = b;
                sh.sel.before = run;
            }
        }
        if (threadIdx.x == 0) sh.sel.nex = 0;
        __syncthreads();
        const int b = sh.sel.bsel, need = r - sh.sel.before;
#pragma unroll
        for (int t = 0; t < PT; ++t) {
            if (kk[t] == ~0ull) continue;
            const int bin = (int)(kk[t] >> 52);
            if (bin < b) {
                v.take[threadIdx.x + t * LB] += 1;
            } else if (bin == b) {
                const int p = atomicAdd(&sh.sel.nex, 1);
                if (p < EXACT) sh.sel.keys[p] = kk[t];
            }
        }
        __syncthreads();
        const int ne = sh.sel.nex;
        if (ne <= EXACT) {
            for (int a = threadIdx.x; a < ne; a += LB) {
                const unsigned long long ka = sh.sel.keys[a];
                int rk = 0;
                for (int q = 0; q < ne; ++q) rk += sh.sel.keys[q] < ka;
                if (rk < need) v.take[(int)(ka & 0xffffffffull)] += 1;
            }
        } else {
            // more than EXACT keys share the bin (not expected for Philox
            // priorities): select among them generically
            if (threadIdx.x == 0) atomicOr(&c->npath, NPATH_BINOVER);
            auto pred = [&](int j) {
                const int rp = sh.rr[j].y, lo = sh.rr[j].x;
                return rp > 0 && lo <= Lstar && Lstar < lo + rp && (int)(ref_key_of(v, j) >> 52) == b;
            };
            auto key = [&](int j) { return ref_key_of(v, j); };
            auto mark = [&](int j) { v.take[j] += 1; };
            block_select_smallest(w, need, key, pred, mark, sh.sel, &c->npath);
        }
    } else {
        if (threadIdx.x == 0) {
            sh.nck = 0;
            atomicOr(&c->npath, NPATH_UNSTAGED);
        }
        __syncthreads();
        for_refs([&](int j, int lo, int rp) {
            v.take[j] = rp > 0 ? min(rp, max(0, Lstar - lo)) : 0;
            if (rp > 0 && lo <= Lstar && Lstar < lo + rp) {
                const int p = atomicAdd(&sh.nck, 1);
                if (p < CKCAP) sh.ck[p] = ref_key_of(v, j);
            }
        });
        __syncthreads();
        const int nC = sh.nck;
        if (nC <= CKCAP) {
            auto key = [&](int e) { return sh.ck[e]; };
            auto pred = [&](int) { return true; };
            auto mark = [&](int e) { v.take[(int)(sh.ck[e] & 0xffffffffull)] += 1; };
            block_select_smallest(nC, r, key, pred, mark, sh.sel, &c->npath);
        } else {
            if (threadIdx.x == 0) atomicOr(&c->npath, NPATH_CKOVER);
            auto pred = [&](int j) {
                const int rp = rhop_of(j);
                const int lo = rho_of(j);
                return rp > 0 && lo <= Lstar && Lstar < lo + rp;
            };
            auto key = [&](int j) { return ref_key_of(v, j); };
            auto mark = [&](int j) { v.take[j] += 1; };
            block_select_smallest(w, r, key, pred, mark, sh.sel, &c->npath);
        }
    }
    __syncthreads();
    if (staged) {
        // exclusive scan of rho' over contiguous runs held in shared memory;
        // offsets replace rho in shared memory, then go out coalesced
        const int per = (w + LB - 1) / LB;
        const int lo = min(w, (int)threadIdx.x * per), hi = min(w, lo + per);
        int sum = 0;
        for (int j = lo; j < hi; ++j) sum += sh.rr[j].y;
        int total;
        int run = block_excl_scan(sum, sh.scratch, &total);
        for (int j = lo; j < hi; ++j) {
            const int cnt = sh.rr[j].y;
            sh.rr[j].x = run;
            run += cnt;
        }
        __syncthreads();
        for (int j = threadIdx.x; j < w; j += LB) v.ref_off[j] = sh.rr[j].x;
        if (threadIdx.x == 0) v.ref_off[w] = total;
    } else {
        block_scan_array(v.rhop, v.ref_off, w, sh.scratch);
    }
    if (threadIdx.x == 0) {
        c->Lstar = Lstar;
        c->rlev = r;
        c->nlarge = 0;
    }
}

// ----------------------------------------------------------- k_bucket ------
// Members of F_l into their references' lists.  With few references (at most
// BK_W) many members share one: a CTA numbers its members of each reference
// in shared memory and takes their places by one global atomic per reference
// (one per member, hundreds on one address, took 30 us at 165,000 members of
// 275 references; 7 now).  Each member's priority and distance go with it:
// the selections read them in list order.
constexpr int BK = 1024;
constexpr int BK_W = 4096;

__global__ void __launch_bounds__(BK) k_bucket(RunView v)
{
    extern __shared__ int cnt[];  // w counts, then first places (w <= BK_W)
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int i = blockIdx.x * BK + threadIdx.x;
    const bool in = i < v.n2 && v.rank2[i] == c->l;
    int j = in ? v.pi[i] : 0;
    if (j < 0 || j >= v.w) {
        set_status(c, DEV_EINTERNAL);
        j = -1;
    }
    const bool mem = in && j >= 0;
    int p = 0;
    const double d = in ? v.dist[i] : 0.0;
    const uint32_t prio = in ? mem_prio(v.seed, c->gen, i) : 0u;
    if (v.w <= BK_W) {
        for (int t = threadIdx.x; t < v.w; t += BK) cnt[t] = 0;
        __syncthreads();
        if (mem) p = atomicAdd(&cnt[j], 1);
        __syncthreads();
        for (int t = threadIdx.x; t < v.w; t += BK)
            if (cnt[t]) cnt[t] = atomicAdd(&v.cursor[t], cnt[t]);
        __syncthreads();
        if (mem) p += cnt[j];
    } else if (mem) {
        p = atomicAdd(&v.cursor[j], 1);
    }
    if (!mem) return;
    if (p < v.rhop[j]) {
        const int at = v.ref_off[j] + p;
        v.bucket[at] = i;
        v.bprio[at] = prio;
        v.bdist[at] = d;
    } else {
        set_status(c, DEV_EINTERNAL);
    }
}

__device__ __forceinline__ void mark_member(const RunView& v, int i)
{
    atomicOr(&v.selmask[i >> 5], 1u << (i & 31));
}

// ------------------------------------------------------------- k_pick ------
// one warp per reference; a partial take from more than 32 members, or all of
// more than 256, goes to a whole CTA (k_pick_large), the nearest member too (a warp walking thousands
// of members for it took 96 us at 165,000 members of 275 references)
__global__ void __launch_bounds__(256) k_pick(RunView v)
{
    Ctrl* c = v.ctrl;
    const int lane = lane_id();
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    if (skip_niche(c)) return;
    for (int j = gw; j < v.w; j += nw) {
        const int take = v.take[j], cnt = v.rhop[j], off = v.ref_off[j], rho = v.rho[j];
        if (take == 0) continue;
        if (take >= cnt && cnt <= 256) {
#pragma unroll 4
            for (int e = lane; e < cnt; e += 32) mark_member(v, v.bucket[off + e]);
            continue;
        }
        if (cnt > 32) {
            if (lane == 0) {
                const int p = atomicAdd(&c->nlarge, 1);
                v.large[p] = make_int4(j, take, rho, 0);
                // more members to take than the nearest: the block-wide selection runs
                if (take < cnt && take > (rho == 0 ? 1 : 0)) atomicOr(&c->npath, NPATH_LARGE);
            }
            continue;
        }
        // one member per lane
        int i = -1;
        double d = CUDART_INF;
        unsigned long long k = ~0ull;
        if (lane < cnt) {
            i = v.bucket[off + lane];
            d = v.bdist[off + lane];
            k = ((unsigned long long)v.bprio[off + lane] << 32) | (unsigned)i;
        }
        int need = take, excl = -1;
        if (rho == 0) {
            // nearest: distances are >= 0 and order like their bits
            unsigned long long b = lane < cnt ? (unsigned long long)__double_as_longlong(d) : ~0ull;
            const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)(b >> 32));
            const unsigned lo = __reduce_min_sync(0xffffffffu, (unsigned)(b >> 32) == hi ? (unsigned)b : 0xffffffffu);
            const bool eq = lane < cnt && b == (((unsigned long long)hi << 32) | lo);
            excl = (int)__reduce_min_sync(0xffffffffu, eq ? (unsigned)i : 0x7fffffffu);
            if (lane == 0) mark_member(v, excl);
            need -= 1;
        }
        if (need == 0) continue;
        if (i == excl) k = ~0ull;
        int rk = 0;
        for (int b = 0; b < cnt; ++b) {
            unsigned long long kb = __shfl_sync(0xffffffffu, k, b);
            rk += kb < k;
        }
        if (lane < cnt && i != excl && rk < need) mark_member(v, i);
    }
}

// Large buckets: one CTA per bucket.  Up to PL_CAP members' keys are staged in
// shared memory while the nearest is found: the passes of the selection then
// cost what their barriers cost, not a trip through L2 each.  Bound: the
// latency of the loads and barriers of the largest buckets' CTAs.  119,000
// members of 462 references: 48 us without the staging, 26 with it.
constexpr int PL_T = 512;
constexpr int PL_CAP = 4096;

__global__ void __launch_bounds__(PL_T) k_pick_large(RunView v)
{
    __shared__ SelShared sh;
    __shared__ unsigned long long sd[PL_T / 32];
    __shared__ int si[PL_T / 32];
    __shared__ unsigned long long keys[PL_CAP];
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int nl = c->nlarge;
    for (int t = blockIdx.x; t < nl; t += gridDim.x) {
        const int4 L = v.large[t];
        const int j = L.x;
        int need = L.y, excl = -1;
        const int cnt = v.rhop[j], off = v.ref_off[j];
        const int32_t* mem = v.bucket + off;
        if (need >= cnt) {
            for (int e = threadIdx.x; e < cnt; e += PL_T) mark_member(v, mem[e]);
            continue;
        }
        const bool staged = cnt <= PL_CAP;
        // rho = 0: the nearest member first; distances are >= 0 and order like
        // their bits (an FP64 compare takes 110 cycles, ten of them in a chain)
        unsigned long long bd = ~0ull;
        int bi = 0x7fffffff;
        if (staged || L.z == 0) {
#pragma unroll 4
            for (int e = threadIdx.x; e < cnt; e += PL_T) {
                const int i = mem[e];
                if (staged) keys[e] = ((unsigned long long)v.bprio[off + e] << 32) | (unsigned)i;
                if (L.z == 0) {
                    const unsigned long long d = (unsigned long long)__double_as_longlong(v.bdist[off + e]);
                    if (d < bd || (d == bd && i < bi)) {
                        bd = d;
                        bi = i;
                    }
                }
            }
        }
        if (L.z == 0) {
            auto warp_nearest = [&]() {
                const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)(bd >> 32));
                const unsigned lo = __reduce_min_sync(0xffffffffu, (unsigned)(bd >> 32) == hi ? (unsigned)bd : 0xffffffffu);
                const unsigned long long b = ((unsigned long long)hi << 32) | lo;
                bi = __reduce_min_sync(0xffffffffu, bd == b ? bi : 0x7fffffff);
                bd = b;
            };
            warp_nearest();
            if (lane_id() == 0) {
                sd[threadIdx.x >> 5] = bd;
                si[threadIdx.x >> 5] = bi;
            }
            __syncthreads();
            bd = sd[lane_id() & (PL_T / 32 - 1)];
            bi = si[lane_id() & (PL_T / 32 - 1)];
            warp_nearest();
            excl = bi;
            if (threadIdx.x == 0) mark_member(v, bi);
            need -= 1;
        }
        auto mark = [&](int e) { mark_member(v, mem[e]); };
        __syncthreads();
        if (staged) {
            auto pred = [&](int e) { return (int)(unsigned)keys[e] != excl; };
            auto key = [&](int e) { return keys[e]; };
            block_select_smallest(cnt, need, key, pred, mark, sh, &c->npath);
        } else {
            auto pred = [&](int e) { return mem[e] != excl; };
            auto key = [&](int e) { return ((unsigned long long)v.bprio[off + e] << 32) | (unsigned)mem[e]; };
            block_select_smallest(cnt, need, key, pred, mark, sh, &c->npath);
        }
        __syncthreads();
    }
}

// Self-test of block_select_smallest on caller keys (one CTA): marks[e] = 1
// for the `need` smallest of keys[0..n), 0 otherwise; *paths gets the radix
// pass bits.
__global__ void __launch_bounds__(512) k_select_probe(const unsigned long long* keys, int n, int need,
                                                      uint32_t* marks, unsigned* paths)
{
    __shared__ SelShared sh;
    for (int e = threadIdx.x; e < n; e += blockDim.x) marks[e] = 0u;
    if (threadIdx.x == 0) *paths = 0u;
    __syncthreads();
    auto pred = [&](int) { return true; };
    auto key = [&](int e) { return keys[e]; };
    auto mark = [&](int e) { marks[e] = 1u; };
    block_select_smallest(n, need, key, pred, mark, sh, paths);
}

}  // namespace

cudaError_t launch_level(const RunView& v, cudaStream_t s)
{
    k_level<<<1, LB, sizeof(LevelShared), s>>>(v);
    return cudaGetLastError();
}

cudaError_t launch_bucket(const RunView& v, cudaStream_t s)
{
    k_bucket<<<(v.n2 + BK - 1) / BK, BK, v.w <= BK_W ? (size_t)v.w * sizeof(int) : 0, s>>>(v);
    return cudaGetLastError();
}

cudaError_t launch_pick(const RunView& v, cudaStream_t s)
{
    int blocks = (v.w + 7) / 8;
    if (blocks > 4096) blocks = 4096;
    k_pick<<<blocks, 256, 0, s>>>(v);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // one CTA per reference listed (how many there are is known on the device
    // only: CTAs without one exit), up to three per SM, or one where there are
    // about as many references as individuals and few hold more than 32 (three:
    // 5.0 us instead of 3.5 at 10,626 references without a large one)
    int lblocks = (v.n2 >= 16 * v.w ? 3 : 1) * v.num_sms;
    if (lblocks > v.w) lblocks = v.w;
    if (lblocks < 16) lblocks = 16;
    k_pick_large<<<lblocks, PL_T, 0, s>>>(v);
    return cudaGetLastError();
}

cudaError_t launch_select_probe(const unsigned long long* keys, int n, int need, uint32_t* marks,
                                unsigned* paths, cudaStream_t s)
{
    k_select_probe<<<1, 512, 0, s>>>(keys, n, need, marks, paths);
    return cudaGetLastError();
}

cudaError_t niche_init_attributes()
{
    return cudaFuncSetAttribute(k_level, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(LevelShared));
}
