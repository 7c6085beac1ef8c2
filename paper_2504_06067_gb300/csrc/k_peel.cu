// k_peel.cu -- non-dominated front peeling over the bit-packed matrix
// (Alg. 1, the non-dominated sort: fronts F_1, F_2, ... until |F_1| + ... + |F_l| >= N,
// splitting R_t into S = F_1..F_{l-1}, F_l and F_drop; Sec. II-C).
//
// One cooperative launch runs every pass: each CTA writes its columns' words
// of the front, waits for the others and counts the words itself, so that all
// take the same decision and the host never synchronises.
// Positions are in key order (k_sort.cu); ranks are written back to the
// original order by k_norm_ideal.
//   cnt[j]    = dominators of j, counted by the dominance build
//   pass k>0: cnt[j] -= popc(Dom[w][j] & front_{k-1}[w]) over the nonzero
//             words w of the previous front's mask
//   front_k   = { j unranked : cnt[j] == 0 }, rank2[j] = k
// A CTA of 16 warps owns 128 columns (uint4 per lane); its warps split the
// dominator rows and meet in shared memory, so the CTA alone updates its
// columns' counts, ranks them and writes their front words.  A chunk of
// columns whose smallest count exceeds the points ranked since it was last
// looked at has no member in this front: it is passed over and later counts
// those fronts off together (half of the points are never ranked, and most
// chunks hold a point of a few fronts only).
//
// Bound: latency.  A pass is a chain of trips through L2 (Dom rows, arrival
// with its release, the poll, the front words), 5 us in all however few the
// points of its front, about 3 of them from the arrival to the words.  So the
// block bitmap is kept in shared memory (it was a dependent load before every
// row), four rows are in flight per warp (eight spill and took 10 % longer)
// and a chunk's counts stay in registers.  Selections of the knapsack (m = 3,
// N = 12,800, 27 to 48 fronts): 296 us before, 202 now; m = 5, N = 10,628,
// three fronts: 38 us before, 20 now; the first generation of m = 10,
// N = 100,000: 342 us before, 128 now.
// Several chunks per CTA keep the masks of the last seven passes in global
// memory, and in shared memory the words of those passes that have a few
// (FEW): a chunk whose pending passes all have few takes its rows from those
// instead of scanning seven masks.  A total order of 200,000 points: 2.97 s
// before any deferral, 3.06 with the scans, 1.07 so (100,000 points, m = 3: 612
// and 337 ms before and so).  A longer ring (16) cost the knapsack 20 us.
// Without the matrix (STREAM) every chunk is tested every pass: putting the
// tests off piles them up on the CTAs whose chunks are due (8.6 -> 17.5 ms at
// m = 3, 2N = 120,000, 32 fronts).
#include <limits.h>
#include <math_constants.h>

#include "kernels.cuh"

namespace {

constexpr int PEEL_THREADS = 512;  // threads per CTA
constexpr int PWMAX = PEEL_THREADS / 32;
constexpr int LISTCAP = 2048;
constexpr int RING = NSGA3_FRONT_RING;
constexpr int PEEL_U = 4;   // Dom rows in flight per warp
constexpr int MAXC = 64;  // chunks of a CTA whose state is kept between passes
constexpr int FEW = 32;   // nonzero words of a pass that are kept beside its mask

// Streaming: the members mk of a front word (rb: SQ x 16 bytes each) against
// this lane's four columns, with the sign-bit test of the dominance build; a
// member whose f_0 is below every f_0 of the chunk (cmin) needs objectives
// 1 .. m - 1 only (f_0 makes the dominance strict).  Q = ceil(m / 4).
// (One loop over ten objectives with a predicate each: 4.7 ms for two fronts
// of m = 3, 2N = 120,000; 1.9 so.)
constexpr int SQ = (NSGA3_FAST_M + 3) / 4;

__device__ __forceinline__ uint32_t sign_or(const float4& a, const float4& b)
{
    return __float_as_uint(a.x - b.x) | __float_as_uint(a.y - b.y) | __float_as_uint(a.z - b.z) |
           __float_as_uint(a.w - b.w);
}

template <int Q>
__device__ __forceinline__ void stream_rows(const float4* rb, uint32_t mk, const float4 (&fc)[4][SQ], float cmin,
                                            uint32_t (&a)[4])
{
    while (mk) {  // warp-uniform: every lane walks the same rows
        const int b = __ffs(mk) - 1;
        mk &= mk - 1u;
        float4 y[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) y[q] = rb[b * SQ + q];
        if (y[0].x < cmin) {
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                uint32_t oa = __float_as_uint(fc[t][0].y - y[0].y) | __float_as_uint(fc[t][0].z - y[0].z) |
                              __float_as_uint(fc[t][0].w - y[0].w);
#pragma unroll
                for (int q = 1; q < Q; ++q) oa |= sign_or(fc[t][q], y[q]);
                a[t] += (~oa) >> 31;  // no f_iq > f_jq
            }
        } else {
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                uint32_t oa = 0u, ob = 0u;
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    oa |= sign_or(fc[t][q], y[q]);
                    ob |= sign_or(y[q], fc[t][q]);
                }
                a[t] += (ob & ~oa) >> 31;  // none greater, some smaller
            }
        }
    }
}

// OWN: a chunk per CTA at most and all front words in shared memory.  KEEP:
// more front words than that, and passes of few keep them.  (All forms in one
// kernel: the knapsack's 20 generations 10.2 ms, 9.7 with OWN apart.)
template <bool STREAM, bool OWN, bool KEEP>
__global__ void __launch_bounds__(PEEL_THREADS, STREAM ? 1 : 2) k_peel(RunView v)
{
    __shared__ int red[PWMAX][NSGA3_PEEL_COLS];
    const int PT = blockDim.x, PW = PT >> 5;
    __shared__ uint2 list[LISTCAP];
    __shared__ int wcnt[2][PWMAX];
    __shared__ uint32_t last[LISTCAP];   // the last pass's front words (the first LISTCAP; own: of all passes not counted off)
    __shared__ unsigned char nibs[LISTCAP];  // of the CTA's only chunk: column blocks with bits, per dominator block
    __shared__ int nlist[2];
    __shared__ unsigned s_fs[3];  // size of a pass's front
    __shared__ int s_fail;
    __shared__ int c_min[MAXC], c_eval[MAXC], c_cum[MAXC];  // per chunk: smallest count left, pass of it, points then
    __shared__ uint2 few[KEEP ? RING : 1][FEW];  // (keep) the last passes' nonzero words ...
    __shared__ int nfew[RING];                      // ... and how many; more than FEW: only the masks hold them
    __shared__ float4 rowbuf[STREAM ? PWMAX : 1][32 * SQ];  // streaming: members of a front word
    Ctrl* c = v.ctrl;
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    if (read_status(c)) return;  // uniform: set only by earlier kernels
    // the view's points, and the fronts and points before them (rest: the
    // first front is taken, or empty where the matrix is of all points; no
    // rest: it held N points)
    const int cum0 = v.rest ? *(volatile const int32_t*)&c->nF0 : 0;
    const int n2 = view_n2(v), before = cum0 > 0 ? 1 : 0;
    if (n2 == 0) return;
    const int nchunks = v.rest ? (n2 + NSGA3_PEEL_COLS - 1) / NSGA3_PEEL_COLS : v.ld / NSGA3_PEEL_COLS;
    if ((int)blockIdx.x >= nchunks) return;  // owns no columns: nobody waits for it
    const int nwords = nchunks * (NSGA3_PEEL_COLS / 32);
    const bool single = OWN || nchunks <= (int)gridDim.x;
    const bool keep = KEEP && nwords > LISTCAP;  // (one round scans fewer words)
    const bool own = OWN || (single && nwords <= LISTCAP);  // pending words stay in shared memory
    int lim1 = 0, my_cnt = 0;
    bool my_open = false;  // not ranked yet
    unsigned nrows = 0u;   // (per warp) Dom rows read
    bool evald = true;  // (own) the chunk was evaluated in the pass before
    if (tid < 2) nlist[tid] = 0;
    if (tid < 3) s_fs[tid] = 0u;
    if (tid == 0) s_fail = 0;
    if (tid < MAXC) c_min[tid] = INT_MAX;
    if (tid < RING) nfew[tid] = 0;
    __syncthreads();
    // every CTA follows the same sequence of front sizes, so each keeps the
    // pass state itself; CTA 0 also publishes it in ctrl
    int cum = cum0, l = -1, par = 0;
    for (int k = 0;; ++k) {
        // cum: the points ranked before pass k
        int slot = 0;
        for (int chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x, ++slot) {
            const int j0 = chunk * NSGA3_PEEL_COLS;
            // the fronts of passes k0 .. k-1 are not counted off yet
            int k0 = k - 1;
            if (k > 0 && slot < MAXC) {
                k0 = c_eval[slot];
                const int least = c_min[slot];
                evald = !(least == INT_MAX || (!STREAM && least > cum - c_cum[slot] && (own || k - k0 < RING - 1)));
                if (!evald) {
                    if (tid < NSGA3_PEEL_COLS / 32)
                        v.front[(size_t)(k % RING) * v.NW + j0 / 32 + tid] = 0u;
                    continue;
                }
            }
            // the points ranked in passes k0 .. k-1, by word
            auto pending = [&](int w) {
                uint32_t x = w < LISTCAP ? last[w] : __ldcg(&v.front[(size_t)((k - 1) % RING) * v.NW + w]);
                if (STREAM || own) return x;
                if (k0 < k - 1) {  // the older ones, their loads in flight together
                    uint32_t y[RING - 2];
#pragma unroll
                    for (int r = 0; r < RING - 2; ++r)
                        y[r] = __ldcg(&v.front[(size_t)(min(k0 + r, k - 1) % RING) * v.NW + w]);
#pragma unroll
                    for (int r = 0; r < RING - 2; ++r) x |= y[r];
                }
                return x;
            };
            // this thread's column: dominators not counted off (0: ranked or
            // no column); used after the reduction
            if (tid < NSGA3_PEEL_COLS && !(single && k > 0)) {
                const bool in = j0 + tid < n2;
                my_cnt = in ? __ldcg(&v.cnt[j0 + tid]) : 0;
                my_open = in && (k == 0 || my_cnt > 0);
            }
            // dominators of a column have a sort key <= its key: the chunk's row
            // blocks end with its last column's key (k_sort.cu)
            const int lim = single && k > 0 ? lim1 : j0 < n2 ? min((int)v.chunk_lim[chunk], v.NW) : 0;
            lim1 = lim;
            const int J0 = j0 / 32;
            const uint8_t* nz = v.dnz ? v.dnz + (J0 >> 3) : nullptr;
            if (!STREAM && k == 0 && single)
                for (int w = tid; w < min(lim, LISTCAP); w += PT)
                    nibs[w] = nz ? (nz[(size_t)w * v.NB8] >> (J0 & 4)) & 15 : 15;

            uint32_t a0 = 0, a1 = 0, a2 = 0, a3 = 0;
            // pass 0 needs no words: the dominance build already counted every
            // column's dominators into cnt[]
            if (STREAM && k > 0) {
                // no matrix: every member of front k-1 (up to the row limit)
                // is tested against this lane's four columns lane*4 .. +3,
                // with the sign-bit test of the dominance build; a member
                // whose f_0 is below every f_0 of the chunk needs objectives
                // 1..m-1 only (f_0 makes the dominance strict)
                const int q4 = v.fs / 4;  // (the pads are 0 in rows and columns)
                const float4* Fp4 = reinterpret_cast<const float4*>(v.Fp);
                float4 fc[4][SQ];
                float cmin = CUDART_INF_F;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
#pragma unroll
                    for (int q = 0; q < SQ; ++q)
                        fc[t][q] = q < q4 ? Fp4[(size_t)(j0 + lane * 4 + t) * q4 + q] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    cmin = fminf(cmin, fc[t][0].x);  // NaN padding columns are ignored by fminf
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) cmin = fminf(cmin, __shfl_xor_sync(0xffffffffu, cmin, o));
                float4* rb = rowbuf[warp];
                uint32_t a[4] = {0u, 0u, 0u, 0u};
                for (int wb = 0; wb < lim; wb += LISTCAP) {
                    const int whe = min(wb + LISTCAP, lim);
                    int* const nl = &nlist[par];
                    for (int w0 = wb + warp * 32; w0 < whe; w0 += PT) {
                        const int w = w0 + lane;
                        const uint32_t msk = w < whe ? pending(w) : 0u;
                        const unsigned bal = __ballot_sync(0xffffffffu, msk != 0u);
                        int at = 0;
                        if (lane == 0 && bal) at = atomicAdd(nl, __popc(bal));
                        at = __shfl_sync(0xffffffffu, at, 0);
                        if (msk) list[at + __popc(bal & ((1u << lane) - 1u))] = make_uint2((unsigned)w, msk);
                    }
                    __syncthreads();
                    const int n = *nl;
                    par ^= 1;
                    if (tid == 0) nlist[par] = 0;
                    if (warp == 0) nrows += (unsigned)n;
                    for (int e = warp; e < n; e += PW) {
                        const uint2 L = list[e];
                        // the word's members, one per lane, into this warp's row buffer
                        if ((L.y >> lane) & 1u) {
                            const float4* f = Fp4 + ((size_t)L.x * 32 + lane) * q4;
#pragma unroll
                            for (int q = 0; q < SQ; ++q)
                                if (q < q4) rb[lane * SQ + q] = __ldg(f + q);
                        }
                        __syncwarp();
                        if (q4 == 1)
                            stream_rows<1>(rb, L.y, fc, cmin, a);
                        else if (q4 == 2)
                            stream_rows<2>(rb, L.y, fc, cmin, a);
                        else
                            stream_rows<3>(rb, L.y, fc, cmin, a);
                        __syncwarp();
                    }
                    __syncthreads();  // list and nlist are reused
                }
                a0 = a[0];
                a1 = a[1];
                a2 = a[2];
                a3 = a[3];
            } else if (!STREAM && k > 0) {
                const uint4* base = reinterpret_cast<const uint4*>(v.Dom + dom_at(v, 0, J0, 0)) + lane;
                // with the block bitmap (m <= 10) only the Dom blocks whose bit
                // is set were written this selection: bit t of an entry's top
                // nibble says that the chunk's t-th column block is read from
                // dominator block w.  Known before the first Dom load, so the
                // loads of PEEL_U entries are in flight at once.
                const unsigned mybit = 1u << (28 + (lane >> 3));
                auto rows = [&](int n) {
                    if (warp == 0) nrows += (unsigned)n;
                    for (int e = warp; e < n; e += PEEL_U * PWMAX) {
                        uint32_t mk[PEEL_U];
                        uint4 x[PEEL_U];
#pragma unroll
                        for (int t = 0; t < PEEL_U; ++t) {
                            const uint2 L = e + PWMAX * t < n ? list[e + PWMAX * t] : make_uint2(0u, 0u);
                            mk[t] = L.y;
                            x[t] = L.x & mybit ? __ldg(base + (size_t)(L.x & 0x0fffffffu) * (NSGA3_PEEL_COLS / 4)) : make_uint4(0u, 0u, 0u, 0u);
                        }
#pragma unroll
                        for (int t = 0; t < PEEL_U; ++t) {
                            a0 += __popc(x[t].x & mk[t]);
                            a1 += __popc(x[t].y & mk[t]);
                            a2 += __popc(x[t].z & mk[t]);
                            a3 += __popc(x[t].w & mk[t]);
                        }
                    }
                };
                bool sparse = keep;  // every pending pass has few words: no scan of the masks
                for (int r = k0; r < k; ++r) sparse = sparse && nfew[r % RING] <= FEW;
                if (sparse) {
                    static_assert((RING - 1) * FEW <= PEEL_THREADS, "a thread per word");
                    const int r = k0 + tid / FEW, e = tid % FEW;
                    uint2 L = make_uint2(0u, 0u);
                    if (r < k && e < nfew[r % RING]) L = few[r % RING][e];
                    bool in = L.y != 0u && (int)L.x < lim;
                    if (in && nz) {
                        const unsigned nib = ((unsigned)nz[(size_t)L.x * v.NB8] >> (J0 & 4)) & 15u;
                        in = nib != 0u;
                        L.x |= nib << 28;
                    } else {
                        L.x |= 15u << 28;
                    }
                    const unsigned bal = __ballot_sync(0xffffffffu, in);
                    if (lane == 0) wcnt[par][warp] = __popc(bal);
                    __syncthreads();
                    const int x0 = lane < PWMAX ? wcnt[par][lane] : 0;
                    const int n = __reduce_add_sync(0xffffffffu, x0);
                    const int at = __reduce_add_sync(0xffffffffu, lane < warp ? x0 : 0);
                    par ^= 1;
                    if (in) list[at + __popc(bal & ((1u << lane) - 1u))] = L;
                    __syncthreads();
                    rows(n);
                }
                for (int wb = 0; !sparse && wb < lim; wb += LISTCAP) {
                    // the words with members that dominate one of the columns,
                    // a warp's after those of the warps before it (adding up
                    // in one counter took 1 us)
                    constexpr int G = LISTCAP / PEEL_THREADS;
                    unsigned nib[G];
                    uint32_t msk[G];
                    int mine = 0;
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        const int w = wb + g * PEEL_THREADS + tid;
                        nib[g] = 0u;
                        msk[g] = 0u;
                        if (w < lim) {
                            nib[g] = single && w < LISTCAP ? nibs[w] : nz ? ((unsigned)nz[(size_t)w * v.NB8] >> (J0 & 4)) & 15u : 15u;
                            msk[g] = pending(w);
                        }
                        mine += __popc(__ballot_sync(0xffffffffu, msk[g] != 0u && nib[g] != 0u));
                    }
                    if (lane == 0) wcnt[par][warp] = mine;
                    __syncthreads();
                    const int x0 = lane < PWMAX ? wcnt[par][lane] : 0;
                    const int n = __reduce_add_sync(0xffffffffu, x0);
                    int at = __reduce_add_sync(0xffffffffu, lane < warp ? x0 : 0);
                    par ^= 1;
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        const bool in = msk[g] != 0u && nib[g] != 0u;
                        const unsigned bal = __ballot_sync(0xffffffffu, in);
                        if (in)
                            list[at + __popc(bal & ((1u << lane) - 1u))] =
                                make_uint2((unsigned)(wb + g * PEEL_THREADS + tid) | nib[g] << 28, msk[g]);
                        at += __popc(bal);
                    }
                    __syncthreads();
                    rows(n);
                    if (wb + LISTCAP < lim) __syncthreads();  // list is reused
                }
            }
            red[warp][lane * 4 + 0] = (int)a0;
            red[warp][lane * 4 + 1] = (int)a1;
            red[warp][lane * 4 + 2] = (int)a2;
            red[warp][lane * 4 + 3] = (int)a3;
            if (tid == 0 && slot < MAXC) c_min[slot] = INT_MAX;
            __syncthreads();
            // this CTA owns its 128 columns: update the counts and rank the new front
            if (tid < NSGA3_PEEL_COLS) {
                int sum = 0;
#pragma unroll
                for (int w = 0; w < PWMAX; ++w) sum += red[w][tid];
                const int j = j0 + tid;
                const int cv = my_cnt - sum;
                const bool open = my_open, nf = open && cv == 0;
                const uint32_t word = __ballot_sync(0xffffffffu, nf);
                if (lane == 0) v.front[(size_t)(k % RING) * v.NW + j0 / 32 + warp] = word;
                const int left = __reduce_min_sync(0xffffffffu, open && !nf ? cv : INT_MAX);
                if (slot < MAXC) {
                    if (lane == 0) atomicMin(&c_min[slot], left);
                    if (tid == 0) {
                        c_eval[slot] = k;
                        c_cum[slot] = cum;
                    }
                }
                if (!single && open && k > 0) v.cnt[j] = cv;
                if (nf) v.srank[v.rest ? v.rmap[j] : j] = k + before;  // (srank is by position among all points)
                my_cnt = cv;
                my_open = open && !nf;
            }
            if (!single) __syncthreads();  // red is reused by the next chunk
        }
        // the pass ends when every CTA has written its front words of it; then
        // each counts them all (the same total everywhere) and keeps them.
        // (Words that carry their pass number and are polled themselves save
        // a trip through L2, but all CTAs polling the same few lines slow
        // every other load: 252 us for the many fronts of the knapsack
        // instead of 225.)
        __syncthreads();
        if (tid == 0) {
            red_release(&c->parr, 1u);
            const unsigned goal = (k + 1u) * (unsigned)min(nchunks, (int)gridDim.x);
            if (!bounded_wait(c, v.wait_ns, [&] { return (int)(ld_acquire(&c->parr) - goal) >= 0; })) s_fail = 1;
        }
        __syncthreads();
        if (s_fail) return;
        {
            unsigned mine = 0u;
            const uint32_t* words = v.front + (size_t)(k % RING) * v.NW;
#pragma unroll 4
            for (int w = tid; w < nwords; w += PT) {
                const uint32_t x = __ldcg(words + w);
                if (w < LISTCAP) last[w] = !STREAM && own && !evald ? last[w] | x : x;
                mine += __popc(x);
                // (once there are more than FEW the count only has to say so)
                if (keep && x && *(volatile int*)&nfew[k % RING] <= FEW) {
                    const int e = atomicAdd(&nfew[k % RING], 1);
                    if (e < FEW) few[k % RING][e] = make_uint2((unsigned)w, x);
                }
            }
            mine = __reduce_add_sync(0xffffffffu, mine);
            if (lane == 0 && mine) atomicAdd(&s_fs[k % 3], mine);
            if (tid == 0) {
                s_fs[(k + 1) % 3] = 0u;  // read two barriers ago
                nfew[(k + 1) % RING] = 0;  // of the pass RING - 1 before this one, which nobody waits for
            }
        }
        __syncthreads();
        // close front k (the same decision in every CTA)
        const int fs = (int)s_fs[k % 3];
        const int ncum = cum + fs;
        bool first = false;
        if (l < 0 && ncum >= v.N) {
            l = k + before;
            first = true;
        }
        const bool broken = fs == 0 && ncum < v.n2;
        const bool more = !broken && fs > 0 && ncum < v.n2 && (v.full_sort || l < 0);
        if (blockIdx.x == 0 && tid == 0) {
            c->cum = ncum;
            c->passes = k + 1 + before;
            c->passes_total += 1ull;
            if (first) {
                c->l = l;
                c->nFl = fs;
                c->nS = cum;
                c->K = v.N - cum;
                c->need_niche = (v.N - cum) < fs ? 1 : 0;
            }
            if (broken) set_status(c, DEV_EINTERNAL);
        }
        cum = ncum;
        if (!more) break;
    }
    if (lane == 0 && nrows) atomicAdd(&c->peel_rows, nrows);
}


int g_peel_occ[2] = {0, 0};  // resident peel CTAs per SM (matrix: of any form; streaming), set at start-up

}  // namespace

// One cooperative launch for all passes: at most as many CTAs as can be
// resident at once (the grid barrier needs them all), at most one per chunk.
cudaError_t launch_peel(const RunView& v, int num_sms, cudaStream_t s)
{
    const int nchunks = v.ld / NSGA3_PEEL_COLS;
    int occ = g_peel_occ[v.streaming ? 1 : 0];
    if (occ <= 0) occ = 1;
    if (v.peel_ctas > 0 && v.peel_ctas < occ) occ = v.peel_ctas;  // launch-shape option
    int grid = num_sms * occ;
    if (v.shared_gpu) {
        // every CTA of a cooperative launch must be resident at once, which a
        // mix of runs rarely allows for a grid the size of the GPU: a CTA for
        // four chunks, or for two with fewer than 16 runs.  Batched runs, 40
        // generations, a CTA for 1, 2, 4, 8 chunks: 6 runs 11.1, 11.0, 11.2,
        // 11.4 ms; 12 runs 13.2, 13.5, 14.8, 17.2; 16 runs 23.2, 21.9, 21.5,
        // 22.9; 64 runs 64.9, 61.3, 60.3, 60.3
        const int g2 = nchunks / v.shared_gpu > 0 ? nchunks / v.shared_gpu : 1;
        if (grid > g2) grid = g2;
    }
    if (grid > nchunks) grid = nchunks;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(PEEL_THREADS);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (v.streaming) return cudaLaunchKernelEx(&cfg, k_peel<true, false, false>, v);
    // (the points a first front leaves have fewer chunks and words)
    if (v.ld / 32 > LISTCAP) return cudaLaunchKernelEx(&cfg, k_peel<false, false, true>, v);
    if (nchunks <= grid) return cudaLaunchKernelEx(&cfg, k_peel<false, true, false>, v);
    return cudaLaunchKernelEx(&cfg, k_peel<false, false, false>, v);
}

cudaError_t peel_init_attributes()
{
    int a = 0, b = 0, c = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_peel<false, false, false>, PEEL_THREADS, 0);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_peel<false, true, false>, PEEL_THREADS, 0);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c, k_peel<false, false, true>, PEEL_THREADS, 0);
    if (e != cudaSuccess) return e;
    g_peel_occ[0] = a < b ? (a < c ? a : c) : (b < c ? b : c);
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&g_peel_occ[1], k_peel<true, false, false>, PEEL_THREADS, 0);
}

