// k_normalize.cu -- the normalization step of Alg. 1 and Alg. 2, read as
// the NSGA-III normalization of Deb & Jain (the paper gives no formula):
//   T = S u F_l;  z*_q = min_T f_q;  f~ = f - z*;
//   e_q = argmin_T max_r f~_r / w_qr  (w_qr = 1 if r == q else 1e-6, ties ->
//         lowest index);  E b = 1 by Gaussian elimination with partial
//         pivoting;  a_q = 1 / b_q;  nadir fallback a_q = max_T f~_q
//         (1 where 0) when a pivot is 0 or an a_q is not finite or <= 1e-6.
// All FP64 operations use the _rn intrinsics, so no FMA contraction occurs
// and every value is the IEEE result of the same operation sequence a
// plain CPU evaluation performs.
// The ASF maximum uses that x -> fl(x / 1e-6) is monotone:
// max_{r != q} fl(f~_r / 1e-6) == fl(max_{r != q} f~_r / 1e-6), so each
// member needs two divisions instead of m * m.
#include "kernels.cuh"
#include "normalize.cuh"

namespace {

constexpr int NB = 256;   // k_norm_ideal
constexpr int EB = 128;   // k_norm_extreme: two blocks per SM

// Ranks back to the original order (every selection), then, when niching
// is needed: members of T are appended to Tlist (in bucket order, which no
// later step depends on) and the ideal point is taken by order-preserving
// atomicMin over Fp (-0.0 is stored as +0.0 there).
__global__ void __launch_bounds__(NB) k_norm_ideal(RunView v)
{
    Ctrl* c = v.ctrl;
    if (read_status(c)) return;
    const int p = blockIdx.x * NB + threadIdx.x;  // position in bucket order
    int i = -1, r = -1;
    if (p < v.n2) {
        i = v.perm[p];
        r = v.srank[p];
        v.rank2[i] = r;
    }
    if (*(volatile const int32_t*)&c->need_niche == 0) return;  // the same for every thread
    const int l = c->l;
    const int lane = lane_id();
    const bool inT = i >= 0 && r >= 0 && r <= l;
    unsigned bal = __ballot_sync(0xffffffffu, inT);
    int base = 0;
    if (lane == 0 && bal) base = atomicAdd(&c->nT, __popc(bal));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (inT) v.Tlist[base + __popc(bal & ((1u << lane) - 1u))] = i;
    // the running ideal (history option) takes every merged point and the
    // previous ideal; a minimum over S u F_l otherwise
    const bool inZ = v.norm_history ? (p < v.n2) : inT;
    if (v.norm_history && blockIdx.x == 0 && threadIdx.x == 0 && c->hvalid)
        for (int q = 0; q < v.m; ++q) atomicMin(&c->zmin[q], f2ord((float)c->hz[q]));
    if (v.m > NSGA3_FAST_M) return;  // k_zmin_gen
    // the block's minimum per objective first (warps, then shared memory),
    // one atomic per block and objective: the ideal point's m words are
    // every block's target
    __shared__ uint32_t smin[NB / 32][NSGA3_FAST_M];
    const int warp = threadIdx.x >> 5;
    for (int q = 0; q < v.m; ++q) {
        uint32_t o = inZ ? f2ord(v.Fp[(size_t)p * v.fs + q]) : 0xffffffffu;
        o = __reduce_min_sync(0xffffffffu, o);
        if (lane == 0) smin[warp][q] = o;
    }
    __syncthreads();
    if (threadIdx.x < v.m) {
        uint32_t o = smin[0][threadIdx.x];
        for (int w = 1; w < NB / 32; ++w) o = min(o, smin[w][threadIdx.x]);
        if (o != 0xffffffffu) atomicMin(&c->zmin[threadIdx.x], o);
    }
}

__device__ __forceinline__ double zstar_of(const Ctrl* c, int q)
{
    // -0.0 and +0.0 are the same minimum: adding +0.0 keeps +0.0
    return __dadd_rn((double)ord2f(c->zmin[q]), 0.0);
}

// Ideal point, E b = 1 (solve_rows), a = 1 / b and the nadir fallback; one
// warp, lane r on row r, m <= 32.  A: m x (m + 1) values of shared memory.
__device__ __noinline__ void solve_intercepts(const RunView& v, Ctrl* c, const int* ext, const double* nad, double* A)
{
    const int m = v.m;
    const int lane = lane_id();
    const bool row = lane < m;
    if (__any_sync(0xffffffffu, row && not_finite_key(sf64::bits(nad[lane])))) {
        if (lane == 0) set_status(c, DEV_ENONFINITE);
        return;
    }
    const double z = row ? zstar_of(c, lane) : 0.0;
    if (row) {
        c->zstar[lane] = z;
        c->ext[lane] = ext[lane];
    }
    const int ncand = v.n2 + ((v.norm_history && c->hvalid) ? m : 0);
    const int er = row ? ext[lane] : 0;
    const bool ok0 = __all_sync(0xffffffffu, er >= 0 && er < ncand);
    // this lane's extreme vector (a merged point or a remembered one)
    const float* ev = er < v.n2 ? v.F + (size_t)er * m : v.he + (size_t)(er - v.n2) * m;
#pragma unroll 4
    for (int q = 0; q < m; ++q) {
        const double zq = __shfl_sync(0xffffffffu, z, q);
        if (row) A[lane * (m + 1) + q] = ok0 ? __dsub_rn((double)ev[q], zq) : 0.0;
    }
    if (row) A[lane * (m + 1) + m] = 1.0;
    double a = 0.0;
    const bool ok = solve_rows(m, A, ok0, a);
    if (row) {
        if (!ok) a = sf64::is_zero(nad[lane]) ? 1.0 : nad[lane];
        c->a[lane] = a;
        if (m <= NSGA3_FAST_M) {
            c->da[lane] = sf64::divisor(a);
            c->z32[lane] = (float)z;
            c->ia32[lane] = __frcp_rn((float)a);
        }
    }
    if (lane == 0) c->fallback = ok ? 0 : 1;
    if (v.norm_history) {
        // the ideal and the extreme vectors become the history; every lane
        // reads its remembered row before any is replaced
        if (row) c->hz[lane] = z;
        __syncwarp();
#pragma unroll 1
        for (int q = 0; q < m; ++q)
            if (row) A[lane * (m + 1) + q] = ok0 ? (double)ev[q] : 0.0;  // A is free again
        __syncwarp();
#pragma unroll 1
        for (int q = 0; q < m; ++q)
            if (row) v.he[lane * m + q] = (float)A[lane * (m + 1) + q];
        if (lane == 0) c->hvalid = 1;
    }
}

// Per-block (min ASF, lowest index) per axis and max of f~; the last block
// to finish reduces the blocks' results and solves for the intercepts.
template <int M>
__global__ void __launch_bounds__(EB) k_norm_extreme(RunView v)
{
    __shared__ unsigned long long s_key[EB / 32][NSGA3_FAST_M];
    __shared__ int s_idx[EB / 32][NSGA3_FAST_M];
    __shared__ unsigned long long s_nad[EB / 32][NSGA3_FAST_M];
    __shared__ unsigned s_ticket;
    __shared__ int f_ext[NSGA3_FAST_M];
    __shared__ double f_nad[NSGA3_FAST_M];
    __shared__ double s_A[M * (M + 1)];
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    constexpr int m = M;
    const int nT = c->nT;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    double zs[M];
    _Pragma("unroll") for (int q = 0; q < m; ++q) zs[q] = zstar_of(c, q);
    unsigned long long best[M], nad[M];
    int bidx[M];
    _Pragma("unroll") for (int q = 0; q < m; ++q) {
        best[q] = ~0ull;
        bidx[q] = 0x7fffffff;
        nad[q] = 0ull;
    }
    for (int s = blockIdx.x * EB + threadIdx.x; s < nT; s += gridDim.x * EB) {
        const int i = v.Tlist[s];
        double ft[M];
        unsigned long long m1 = 0ull, m2 = 0ull;  // largest and second largest key (f~ >= 0)
        int r1 = 0;
        _Pragma("unroll") for (int r = 0; r < m; ++r) {
            ft[r] = __dsub_rn((double)v.F[(size_t)i * m + r], zs[r]);
            const unsigned long long kr = okey(ft[r]);
            if (kr > m1) {
                m2 = m1;
                m1 = kr;
                r1 = r;
            } else if (kr > m2) {
                m2 = kr;
            }
            nad[r] = max(nad[r], kr);
        }
        const double d1 = __ddiv_rn(__longlong_as_double((long long)m1), 1e-6);
        const double d2 = __ddiv_rn(__longlong_as_double((long long)m2), 1e-6);
        const unsigned long long k1 = okey(d1), k2 = okey(d2);
        _Pragma("unroll") for (int q = 0; q < m; ++q) {
            const unsigned long long other = (q == r1) ? k2 : k1;
            const unsigned long long kq = okey(ft[q]);
            const unsigned long long asf = kq > other ? kq : other;
            if (key_less(asf, i, best[q], bidx[q])) {
                best[q] = asf;
                bidx[q] = i;
            }
        }
    }
    _Pragma("unroll") for (int q = 0; q < m; ++q) {
        unsigned long long b = best[q], n = nad[q];
        int bi = bidx[q];
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
        if (lane == 0) {
            s_key[warp][q] = b;
            s_idx[warp][q] = bi;
            s_nad[warp][q] = n;
        }
    }
    __syncthreads();
    unsigned long long* pk = reinterpret_cast<unsigned long long*>(v.ext_part);
    unsigned long long* pn = reinterpret_cast<unsigned long long*>(v.nad_part);
    if (threadIdx.x < m) {
        const int q = threadIdx.x;
        unsigned long long b = s_key[0][q], n = s_nad[0][q];
        int bi = s_idx[0][q];
        for (int w = 1; w < EB / 32; ++w) {
            if (key_less(s_key[w][q], s_idx[w][q], b, bi)) {
                b = s_key[w][q];
                bi = s_idx[w][q];
            }
            n = max(n, s_nad[w][q]);
        }
        pk[blockIdx.x * m + q] = b;
        v.ext_idx[blockIdx.x * m + q] = bi;
        pn[blockIdx.x * m + q] = n;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_ticket = atomicAdd(&c->ext_done, 1u);
    __syncthreads();
    if (s_ticket != gridDim.x - 1) return;
    // last block: reduce over the blocks, one warp per axis; each lane first
    // issues all its loads (independent), then reduces
    __threadfence();
    constexpr int PMAX = 16;  // parts <= 32 * PMAX
    for (int q = warp; q < m; q += EB / 32) {
        unsigned long long lb[PMAX], ln[PMAX];
        int li[PMAX];
#pragma unroll
        for (int t = 0; t < PMAX; ++t) {
            const int p = lane + 32 * t;
            const bool in = p < (int)gridDim.x;
            lb[t] = in ? __ldcg(&pk[p * m + q]) : ~0ull;
            li[t] = in ? __ldcg(&v.ext_idx[p * m + q]) : 0x7fffffff;
            ln[t] = in ? __ldcg(&pn[p * m + q]) : 0ull;
        }
        unsigned long long b = lb[0], n = ln[0];
        int bi = li[0];
#pragma unroll
        for (int t = 1; t < PMAX; ++t) {
            if (key_less(lb[t], li[t], b, bi)) {
                b = lb[t];
                bi = li[t];
            }
            n = max(n, ln[t]);
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
        if (lane == 0) {
            if (v.norm_history && c->hvalid) {
                // the remembered extreme vectors are candidates 2N + r
                for (int r = 0; r < m; ++r) {
                    const float* f = v.he + r * m;
                    double mx = 0.0, tq = 0.0;
                    for (int t = 0; t < m; ++t) {
                        const double ft = __dsub_rn((double)f[t], zs[t]);
                        if (t == q)
                            tq = ft;
                        else if (ft > mx)
                            mx = ft;
                    }
                    const unsigned long long kq = okey(tq), ko = okey(__ddiv_rn(mx, 1e-6));
                    const unsigned long long asf = kq > ko ? kq : ko;
                    if (key_less(asf, v.n2 + r, b, bi)) {
                        b = asf;
                        bi = v.n2 + r;
                    }
                }
            }
            f_ext[q] = bi;
            f_nad[q] = __longlong_as_double((long long)n);
        }
    }
    __syncthreads();
    if (warp == 0) {
        if (lane == 0) c->ext_done = 0u;
        solve_intercepts(v, c, f_ext, f_nad, s_A);
    }
}

// ---------------------------------------------------------------------------
// m > NSGA3_FAST_M.  The candidates of the extreme-point search are "entries":
// the members of T (index = merged index) and, with history, the remembered
// vectors (index 2N + r).  k_ext_keys gives each entry the two ASF keys it
// can have: fl(max_r f~_r / 1e-6) and, for the axis of that maximum (first
// index), fl(second largest / 1e-6).  k_ext_axis takes QG axes per block:
// ASF_q = max(f~_q, that key) per entry, (min, lowest index) per axis, and
// the nadir maxima over the members; k_ext_reduce reduces the blocks (a warp
// per axis) and either solves the intercepts with one warp
// (m <= NSGA3_WARP_M) or leaves E and the nadir to the
// elimination in a cluster below.
constexpr int GB = 128;  // threads per block of the m > NSGA3_FAST_M kernels
constexpr int QG = 8;    // axes per block of k_ext_axis

__device__ __forceinline__ const float* entry_row(const RunView& v, int s, int nT, int& idx)
{
    if (s < nT) {
        idx = v.Tlist[s];
        return v.F + (size_t)idx * v.m;
    }
    idx = v.n2 + (s - nT);
    return v.he + (size_t)(s - nT) * v.m;
}

__device__ __forceinline__ int history_entries(const RunView& v, const Ctrl* c)
{
    return (v.norm_history && c->hvalid) ? v.m : 0;
}

// ideal point for m > NSGA3_FAST_M: thread per objective over a chunk of
// positions (coalesced across objectives), order-preserving atomicMin
constexpr int ZP = 32;  // positions per chunk

__global__ void __launch_bounds__(128) k_zmin_gen(RunView v)
{
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int m = v.m, q = blockIdx.x * 128 + threadIdx.x;
    if (q >= m) return;
    const int l = c->l;
    const int p0 = blockIdx.y * ZP, p1 = min(v.n2, p0 + ZP);
    uint32_t o = 0xffffffffu;
#pragma unroll 8
    for (int p = p0; p < p1; ++p) {
        const int r = v.srank[p];
        const bool in = v.norm_history ? true : (r >= 0 && r <= l);
        if (in) o = min(o, f2ord(v.Fp[(size_t)p * m + q]));
    }
    if (o != 0xffffffffu) atomicMin(&c->zmin[q], o);
}

// a warp per entry: lane-wise (largest key, second largest, first index of
// the largest) over r = lane, lane + 32, ..., merged across the lanes; the
// result is that of one pass over r = 0 .. m-1 (largest, the largest of the
// rest counting a repeated maximum, its first index)
__global__ void __launch_bounds__(GB) k_ext_keys(RunView v)
{
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int m = v.m, nT = c->nT, lane = lane_id();
    const int ne = nT + history_entries(v, c);
    const int nw = gridDim.x * (GB / 32);
    for (int s = (blockIdx.x * GB + threadIdx.x) >> 5; s < ne; s += nw) {
        int idx;
        const float* f = entry_row(v, s, nT, idx);
        unsigned long long m1 = 0ull, m2 = 0ull;  // f~ >= 0: keys order like values
        int r1 = 0x7fffffff;                      // none while m1 == 0
        for (int r = lane; r < m; r += 32) {
            const unsigned long long kr = okey(__dsub_rn((double)f[r], zstar_of(c, r)));
            if (kr > m1) {
                m2 = m1;
                m1 = kr;
                r1 = r;
            } else if (kr > m2) {
                m2 = kr;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long om1 = __shfl_xor_sync(0xffffffffu, m1, o);
            const unsigned long long om2 = __shfl_xor_sync(0xffffffffu, m2, o);
            const int or1 = __shfl_xor_sync(0xffffffffu, r1, o);
            if (om1 > m1) {
                m2 = max(om2, m1);
                m1 = om1;
                r1 = or1;
            } else if (om1 < m1) {
                m2 = max(m2, om1);
            } else if (m1 > 0ull) {  // the maximum occurs on both sides
                m2 = m1;
                r1 = min(r1, or1);
            }
        }
        if (lane == 0) {
            v.ekey[2 * (size_t)s] = okey(__ddiv_rn(__longlong_as_double((long long)m1), 1e-6));
            v.ekey[2 * (size_t)s + 1] = okey(__ddiv_rn(__longlong_as_double((long long)m2), 1e-6));
            v.er1[s] = m1 > 0ull ? r1 : 0;
        }
    }
}

// grid (parts, ceil(m / QG))
__global__ void __launch_bounds__(GB) k_ext_axis(RunView v)
{
    __shared__ unsigned long long s_key[GB / 32][QG];
    __shared__ int s_idx[GB / 32][QG];
    __shared__ unsigned long long s_nad[GB / 32][QG];
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int m = v.m, nT = c->nT;
    const int ne = nT + history_entries(v, c);
    const int parts = gridDim.x;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int q0 = blockIdx.y * QG;
    double zs[QG];
    unsigned long long best[QG], nad[QG];
    int bidx[QG];
#pragma unroll
    for (int t = 0; t < QG; ++t) {
        zs[t] = q0 + t < m ? zstar_of(c, q0 + t) : 0.0;
        best[t] = ~0ull;
        bidx[t] = 0x7fffffff;
        nad[t] = 0ull;
    }
    for (int s = blockIdx.x * GB + threadIdx.x; s < ne; s += parts * GB) {
        int idx;
        const float* f = entry_row(v, s, nT, idx);
        const unsigned long long k1 = v.ekey[2 * (size_t)s], k2 = v.ekey[2 * (size_t)s + 1];
        const int r1 = v.er1[s];
#pragma unroll
        for (int t = 0; t < QG; ++t) {
            const int q = q0 + t;
            if (q >= m) break;
            const unsigned long long kq = okey(__dsub_rn((double)f[q], zs[t]));
            const unsigned long long other = (q == r1) ? k2 : k1;
            const unsigned long long asf = kq > other ? kq : other;
            if (key_less(asf, idx, best[t], bidx[t])) {
                best[t] = asf;
                bidx[t] = idx;
            }
            if (s < nT) nad[t] = max(nad[t], kq);
        }
    }
#pragma unroll
    for (int t = 0; t < QG; ++t) {
        unsigned long long b = best[t], n = nad[t];
        int bi = bidx[t];
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
        if (lane == 0) {
            s_key[warp][t] = b;
            s_idx[warp][t] = bi;
            s_nad[warp][t] = n;
        }
    }
    __syncthreads();
    unsigned long long* pk = reinterpret_cast<unsigned long long*>(v.ext_part);
    unsigned long long* pn = reinterpret_cast<unsigned long long*>(v.nad_part);
    if (threadIdx.x < QG && q0 + (int)threadIdx.x < m) {
        const int t = threadIdx.x, q = q0 + t;
        unsigned long long b = s_key[0][t], n = s_nad[0][t];
        int bi = s_idx[0][t];
        for (int w = 1; w < GB / 32; ++w) {
            if (key_less(s_key[w][t], s_idx[w][t], b, bi)) {
                b = s_key[w][t];
                bi = s_idx[w][t];
            }
            n = max(n, s_nad[w][t]);
        }
        pk[(size_t)blockIdx.x * m + q] = b;
        v.ext_idx[(size_t)blockIdx.x * m + q] = bi;
        pn[(size_t)blockIdx.x * m + q] = n;
    }
}

// per axis (a warp each) the (min, lowest index) over the parts and the
// nadir maximum; with m <= NSGA3_WARP_M the last CTA solves the intercepts
// with one warp, else the elimination in a cluster follows
__global__ void __launch_bounds__(256) k_ext_reduce(RunView v, int parts)
{
    __shared__ unsigned s_ticket;
    __shared__ int f_ext[NSGA3_WARP_M];
    __shared__ double f_nad[NSGA3_WARP_M];
    __shared__ double s_A[NSGA3_WARP_M * (NSGA3_WARP_M + 1)];
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int m = v.m, lane = lane_id();
    const int q = blockIdx.x * 8 + (threadIdx.x >> 5);
    const unsigned long long* pk = reinterpret_cast<const unsigned long long*>(v.ext_part);
    const unsigned long long* pn = reinterpret_cast<const unsigned long long*>(v.nad_part);
    if (q < m) {
        unsigned long long b = ~0ull, n = 0ull;
        int bi = 0x7fffffff;
        for (int p = lane; p < parts; p += 32) {
            const unsigned long long pb = pk[(size_t)p * m + q];
            const int pi = v.ext_idx[(size_t)p * m + q];
            if (key_less(pb, pi, b, bi)) {
                b = pb;
                bi = pi;
            }
            n = max(n, pn[(size_t)p * m + q]);
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
        if (lane == 0) {
            c->ext[q] = bi;
            v.nadv[q] = __longlong_as_double((long long)n);
            if (m > NSGA3_WARP_M && not_finite_key(n)) set_status(c, DEV_ENONFINITE);  // (else solve_intercepts)
        }
    }
    if (m > NSGA3_WARP_M) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_ticket = atomicAdd(&c->ext_done, 1u);
    __syncthreads();
    if (s_ticket != gridDim.x - 1) return;
    __threadfence();
    if (threadIdx.x < m) {
        f_ext[threadIdx.x] = __ldcg(&c->ext[threadIdx.x]);
        f_nad[threadIdx.x] = __ldcg(&v.nadv[threadIdx.x]);
    }
    __syncthreads();
    if (threadIdx.x == 0) c->ext_done = 0u;
    if (threadIdx.x < 32) solve_intercepts(v, c, f_ext, f_nad, s_A);
}

// The intercepts from the solution b of E b = 1 (one CTA of SB threads):
// a = 1 / b where all are usable, else the nadir point's components; the
// history's extreme vectors.
__device__ __noinline__ void finish_solve(const RunView& v, Ctrl* c, bool ok, bool ext_ok, double* sb)
{
    const int m = v.m, tid = threadIdx.x, NT = blockDim.x;
    __syncthreads();
    bool bad = false;
    if (ok)
        for (int q = tid; q < m; q += NT) {
            const double a = __ddiv_rn(1.0, sb[q]);
            bad |= !isfinite(a) || a <= 1e-6;
            sb[q] = a;
        }
    ok = ok && !__syncthreads_or(bad);
    for (int q = tid; q < m; q += NT) {
        const double nq = v.nadv[q];
        c->a[q] = ok ? sb[q] : (nq == 0.0 ? 1.0 : nq);
    }
    if (tid == 0) c->fallback = ok ? 0 : 1;
    if (v.norm_history) {
        for (int q = tid; q < m; q += NT) c->hz[q] = zstar_of(c, q);
        // the staged extreme vectors (zero rows, as in the warp solver, when
        // an extreme index was invalid and nothing was staged)
        for (int e = tid; e < m * m; e += NT) v.he[e] = ext_ok ? v.etmp[e] : 0.0f;
        if (tid == 0) c->hvalid = 1;
    }
}

// m > NSGA3_WARP_M: the elimination in the shared memory of one cluster.  CTA r holds columns r, r + C, ... of [E - z* | 1] (rows in their
// original order; a thread per row in each group of threads, which keeps the
// row's current position).  The owner of the next column brings it up to
// date, finds the pivot, forms the factors and stores them into every CTA
// before it turns to its other columns, so a step waits for one column, one
// quotient and one cluster barrier (0.8 us; a grid barrier and four trips
// through L2 before: 1.7 us), and the other columns' updates, one product and
// one difference on the FP64 pipe each, pass meanwhile.  Same operations, in
// the same order for every element, as the warp solver.
//
// Bound: the chain of a step up to m of about 100, above it the FP64 pipes of
// C SMs (two operations per element, m^3 / 3 elements).  Regular systems, with
// the back substitution: m = 40 188 -> 69 us, m = 64 315 -> 106, m = 128
// 721 -> 240, m = 256 1,680 -> 647, m = 300 2,070 -> 973 (before: a cooperative grid over the rows in
// global memory with a barrier per step).  Eight CTAs up to m = 96: a step's
// factors go to half as many.
constexpr int SC_M = NSGA3_MAX_M;  // rows (a group of threads at least)
constexpr int SC_T = 512;
constexpr int SC_PRE = 4;   // back substitution: columns loaded ahead

__device__ __forceinline__ uint32_t sc_peer(const void* p, int r)
{
    uint32_t d;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(r));
    return d;
}
__device__ __forceinline__ double sc_load(uint32_t a)
{
    double x;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(a) : "memory");
    return x;
}
__device__ __forceinline__ void sc_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void sc_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void sc_group(int threads) { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); }

// CTAs, and bytes of columns in each
inline int sc_ctas(int m) { return m <= 96 ? 8 : 16; }
inline size_t sc_bytes(int m) { return (size_t)(m / sc_ctas(m) + 1) * m * sizeof(double); }

struct ScShared {
    double f[3][SC_M];  // factors by row, three steps of them
    int piv[3][4];      // pivot row, its position before, valid system
    unsigned long long wk[SC_M / 32];
    int wp[SC_M / 32];
    int x0row, x0nan;
    double b[SC_M];
};

__global__ void __launch_bounds__(SC_T) k_solve_cluster(RunView v, int C)
{
    extern __shared__ double cols[];  // m values of each of the CTA's columns
    __shared__ ScShared sh;
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;  // uniform over the cluster
    const int m = v.m, rank = blockIdx.x, tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const int RP = (m + 31) & ~31, G = SC_T / RP, g = tid / RP, row = tid - g * RP;
    const bool mine = row < m && g < G;
    const int ncol = (m - rank) / C + 1;  // columns rank, rank + C, ... <= m
    const int ncand = v.n2 + ((v.norm_history && c->hvalid) ? m : 0);
    bool bad_ext = false;
    if (tid < m) {
        const int e = c->ext[tid];
        bad_ext = e < 0 || e >= ncand;
        if (rank == 0) c->zstar[tid] = zstar_of(c, tid);
    }
    const bool ext_ok = !__syncthreads_or(bad_ext);
    bool ok = ext_ok;
    int pos = row;
    if (ok && mine) {
        const int er = c->ext[row];
        const float* f = er < v.n2 ? v.F + (size_t)er * m : v.he + (size_t)(er - v.n2) * m;
        for (int lc = g; lc < ncol; lc += G) {
            const int k = lc * C + rank;
            double x = 1.0;
            if (k < m) {
                const float ev = f[k];
                if (v.norm_history) v.etmp[(size_t)row * m + k] = ev;
                x = __dsub_rn((double)ev, zstar_of(c, k));
            }
            cols[lc * m + row] = x;
        }
    }
    __syncthreads();
    // column cn of this CTA by its first group: brought up to date with step
    // cn - 1 (pivot row P, factor f), pivot, factors into every CTA
    auto pivot = [&](int cn, int P, double f) {
        double* col = cols + (cn / C) * m;
        double x = row < m ? col[row] : 0.0;
        const bool cand = row < m && pos >= cn;
        if (cn > 0 && cand) {
            x = __dsub_rn(x, __dmul_rn(f, col[P]));
            col[row] = x;
        }
        const unsigned long long k = sf64::bits(x) << 1;  // |x|, twice
        const bool isnan = k > (0x7ff0000000000000ull << 1);
        // the first position of maximal |x|; a NaN replaces nothing, and in
        // the first position is not replaced
        const bool in = cand && !isnan;
        const uint32_t hi = __reduce_max_sync(0xffffffffu, in ? (uint32_t)(k >> 32) : 0u);
        const uint32_t lo = __reduce_max_sync(0xffffffffu, in && (uint32_t)(k >> 32) == hi ? (uint32_t)k : 0u);
        const unsigned long long best = ((unsigned long long)hi << 32) | lo;
        const int at = __reduce_min_sync(0xffffffffu, in && k == best ? pos << 16 | row : 0x7fffffff);
        if (lane == 0) {
            sh.wk[warp] = best;
            sh.wp[warp] = at;
        }
        if (row < m && pos == cn) {
            sh.x0row = row;
            sh.x0nan = isnan ? 1 : 0;
        }
        sc_group(RP);
        unsigned long long bk = 0ull;
        int bp = 0x7fffffff;
        for (int w = 0; w < RP / 32; ++w) {
            const unsigned long long kw = sh.wk[w];
            const int pw = sh.wp[w];
            if (kw > bk || (kw == bk && pw < bp)) {
                bk = kw;
                bp = pw;
            }
        }
        const bool nan0 = sh.x0nan != 0;
        const int np = nan0 ? sh.x0row : bp & 0xffff, pp = nan0 ? cn : bp >> 16;
        const bool good = nan0 || bk != 0ull;
        double fr = 0.0;
        if (good && cand && row != np) fr = div_once(x, col[np]);
        const int buf = cn % 3;
#pragma unroll 1
        for (int r = 0; r < C; ++r) {
            if (row < m)
                asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(sc_peer(&sh.f[buf][row], r)), "d"(fr) : "memory");
            if (tid < 3)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(sc_peer(&sh.piv[buf][tid], r)),
                             "r"(tid == 0 ? np : tid == 1 ? pp : good ? 1 : 0)
                             : "memory");
        }
    };
    // every CTA of the cluster has started (its shared memory is written below)
    sc_arrive();
    sc_wait();
    if (ok) {
        if (rank == 0 && tid < RP) pivot(0, 0, 0.0);
        __syncwarp();
        sc_arrive();
        sc_wait();
        for (int col = 0; col < m; ++col) {
            const int buf = col % 3;
            const int P = sh.piv[buf][0], pp = sh.piv[buf][1];
            if (!sh.piv[buf][2]) {  // the same in every CTA
                ok = false;
                break;
            }
            if (row == P)
                pos = col;
            else if (pos == col)
                pos = pp;
            const bool below = mine && pos > col;
            const double f = below ? sh.f[buf][row] : 0.0;
            if (col + 1 < m && rank == (col + 1) % C && tid < RP) pivot(col + 1, P, f);
            // the factors of the step before last are read no more: a CTA may
            // be one step ahead, so there are three buffers
            __syncwarp();
            sc_arrive();
            if (below) {
                for (int lc = g; lc < ncol; lc += G) {
                    const int k = lc * C + rank;
                    if (k <= col || (k == col + 1 && k < m)) continue;
                    double* a = cols + lc * m;
                    a[row] = __dsub_rn(a[row], __dmul_rn(f, a[P]));
                }
            }
            // the cluster barrier orders the factors; the columns are the
            // CTA's own, and its threads arrived before they updated them
            __syncthreads();
            sc_wait();
        }
    }
    // back substitution column by column from the last unknown (as in the
    // warp solver) by CTA 0, a thread per row; the columns are read from
    // their owners SC_PRE steps ahead
    if (rank == 0 && ok && tid < RP) {
        auto at = [&](int k) { return sc_peer(cols + (k / C) * m + (row < m ? row : 0), k % C); };
        double s = sc_load(at(m));
        const sf64::Divisor dd = sf64::divisor(row < m ? sc_load(at(pos)) : 1.0);
        double u[SC_PRE];
#pragma unroll
        for (int t = 0; t < SC_PRE; ++t) u[t] = m - 1 - t >= 0 ? sc_load(at(m - 1 - t)) : 0.0;
        for (int r0 = m - 1; r0 >= 0; r0 -= SC_PRE) {
#pragma unroll
            for (int t = 0; t < SC_PRE; ++t) {
                const int r = r0 - t;
                if (r < 0) break;
                const double q = sf64::div(s, dd);
                if (row < m && pos == r) sh.b[r] = q;
                sc_group(RP);
                const double br = sh.b[r], ut = u[t];
                if (r - SC_PRE >= 0) u[t] = sc_load(at(r - SC_PRE));
                if (pos < r) s = __dsub_rn(s, __dmul_rn(ut, br));
            }
        }
    }
    __syncwarp();
    sc_arrive();  // the other CTAs' columns are read no more
    sc_wait();
    if (rank == 0) finish_solve(v, c, ok, ext_ok, sh.b);
}

}  // namespace

cudaError_t launch_norm_ideal(const RunView& v, cudaStream_t s)
{
    k_norm_ideal<<<(v.n2 + NB - 1) / NB, NB, 0, s>>>(v);
    return cudaGetLastError();
}

// the one cluster of the elimination
static cudaLaunchConfig_t sc_config(int m, cudaLaunchAttribute* attr, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sc_ctas(m));
    cfg.blockDim = dim3(SC_T);
    cfg.dynamicSmemBytes = sc_bytes(m);
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = sc_ctas(m);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

static cudaError_t launch_norm_extreme_gen(const RunView& v, int num_sms, cudaStream_t s)
{
    if (v.m <= NSGA3_FAST_M || v.m > NSGA3_MAX_M) return cudaErrorInvalidValue;
    const int qgroups = (v.m + QG - 1) / QG;
    int parts = (2 * num_sms + qgroups - 1) / qgroups;
    if (parts > v.ext_parts) parts = v.ext_parts;
    if (parts > (v.n2 + v.m + GB - 1) / GB) parts = (v.n2 + v.m + GB - 1) / GB;
    if (parts < 1) parts = 1;
    k_zmin_gen<<<dim3((v.m + 127) / 128, (v.n2 + ZP - 1) / ZP), 128, 0, s>>>(v);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int kb = (v.n2 + v.m + GB / 32 - 1) / (GB / 32);
    if (kb > 8 * num_sms) kb = 8 * num_sms;
    k_ext_keys<<<kb, GB, 0, s>>>(v);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_ext_axis<<<dim3(parts, qgroups), GB, 0, s>>>(v);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_ext_reduce<<<(v.m + 7) / 8, 256, 0, s>>>(v, parts);
    e = cudaGetLastError();
    if (e != cudaSuccess || v.m <= NSGA3_WARP_M) return e;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = sc_config(v.m, attr, s);
    return cudaLaunchKernelEx(&cfg, k_solve_cluster, v, sc_ctas(v.m));
}

bool solve_fits(int m)
{
    if (m <= NSGA3_WARP_M) return true;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = sc_config(m, attr, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_solve_cluster, &cfg) == cudaSuccess) return n > 0;
    cudaGetLastError();
    return false;
}

cudaError_t norm_init_attributes()
{
    const cudaError_t e = cudaFuncSetAttribute(k_solve_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sc_bytes(SC_M));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_solve_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

cudaError_t launch_norm_extreme(const RunView& v, int num_sms, cudaStream_t s)
{
    if (v.m > NSGA3_FAST_M) return launch_norm_extreme_gen(v, num_sms, s);
    switch (v.m) {
    case 2: k_norm_extreme<2><<<v.ext_parts, EB, 0, s>>>(v); break;
    case 3: k_norm_extreme<3><<<v.ext_parts, EB, 0, s>>>(v); break;
    case 4: k_norm_extreme<4><<<v.ext_parts, EB, 0, s>>>(v); break;
    case 5: k_norm_extreme<5><<<v.ext_parts, EB, 0, s>>>(v); break;
    case 6: k_norm_extreme<6><<<v.ext_parts, EB, 0, s>>>(v); break;
    case 7: k_norm_extreme<7><<<v.ext_parts, EB, 0, s>>>(v); break;
    case 8: k_norm_extreme<8><<<v.ext_parts, EB, 0, s>>>(v); break;
    case 9: k_norm_extreme<9><<<v.ext_parts, EB, 0, s>>>(v); break;
    case 10: k_norm_extreme<10><<<v.ext_parts, EB, 0, s>>>(v); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}
