// k_associate.cu -- association of S u F_l with the reference directions
// (Alg. 2, Eq. 2 read as the perpendicular distance
// D_ij = |f'| sqrt(1 - cos^2), pi_i = argmin_j D_ij, d_i = min_j D_ij) and
// the niche counts rho (over S) and rho' (over F_l) of Alg. 2.
//
// Exactness.  The FP64 distance is evaluated operation for operation like a
// plain CPU evaluation (_rn operations, left-to-right sums), but only for
// candidate references.  Candidates come from FP32 cosines
// qhat_j = u . zhat_j of the unit vectors u = f'/|f'| and zhat_j = z_j/|z_j|
// (all components >= 0).  qhat_j is within Delta = (m+7) 2^-24 of the exact
// cosine up to a factor common to all j (unit32 in associate.cuh; m > 10: u
// rounded from FP64, (m+4) 2^-24).  A reference whose qhat is more than
// band = 2 Delta + 1e-12 below the best qhat has an exact cosine > 1e-12
// below the best reference's; as the vertices e_q are references the best
// cosine is >= 1/sqrt(m), so its exact 1 - c^2 is larger by > 1e-12/sqrt(m),
// far above the FP64 evaluation error (~1e-15): its FP64 distance is
// strictly larger, so it can neither win nor tie.  The FP64 argmin over the
// candidates (ties -> lowest j) equals the argmin over all references.
//
// m <= 10: the references are ordered into spatially compact blocks of 32
// (host, at context creation); a tensor-core product gives every cosine to
// 4.5e-6 and each point's block maxima (k_assoc_mma), and only the blocks that
// can hold its nearest reference are scanned in FP32 (k_assoc_final).
// m > 10: every cosine in FP32 (k_assoc_scan_gen).
//
// FP64 work (GB300 runs FP64 at 1/64 of the FP32 rate) is left to the
// candidates.  A point whose lists overflow is rescanned in FP64 over all
// references by a whole CTA (k_assoc_slow), as is every point in debug mode.
#include <cuda_fp16.h>
#include <cstring>

#include "associate.cuh"
#include "kernels.cuh"

namespace {

constexpr int AB = 256;   // threads per CTA of the FP64 scan

// perp_dist for a run-time m with both rows in memory: sixteen loads of
// each row in flight
__device__ __forceinline__ double perp_dist_mem(const double* fp, double nf, const double* Zj, double nzj,
                                                int m)
{
    if (nf == 0.0) return 0.0;
    double dot = 0.0;
#pragma unroll 16
    for (int q = 0; q < m; ++q) dot = __dadd_rn(dot, __dmul_rn(fp[q], Zj[q]));
    const double den = __dmul_rn(nf, nzj);
    const double cth = __ddiv_rn(dot, den);
    double one_m = __dsub_rn(1.0, __dmul_rn(cth, cth));
    if (one_m < 0.0) one_m = 0.0;
    return __dmul_rn(nf, __dsqrt_rn(one_m));
}

// ---------------------------------------------------------------------------
// m <= 10.

// T slot s: FP32 unit vector (uhat) and its FP16 row for the tensor cores:
// u = h + l with h, l FP16 (to about 2^-23), the row [h, h, l, 0 ...] of
// KP = 16 (m <= 5) or 32 halves, stored as the MMA reads it (see k_assoc_mma).
template <int M>
__host__ __device__ constexpr int kp_of() { return 3 * M <= 16 ? 16 : 32; }

constexpr int PB = 128;

template <int M>
__global__ void __launch_bounds__(PB) k_assoc_prep(RunView v)
{
    constexpr int M4 = (M + 3) & ~3, KP = kp_of<M>();
    __shared__ float sz[M], sa[M];
    Ctrl* c = v.ctrl;
    const int s = blockIdx.x * PB + threadIdx.x;
    if (skip_niche(c)) return;
    if (threadIdx.x < M) {
        sz[threadIdx.x] = c->z32[threadIdx.x];
        sa[threadIdx.x] = c->ia32[threadIdx.x];
    }
    __syncthreads();
    if (s >= c->nT) return;
    const int i = v.Tlist[s];
    float f[M], u[M4];
#pragma unroll
    for (int q = 0; q < M; ++q) f[q] = v.F[(size_t)i * M + q];
#pragma unroll
    for (int q = 0; q < M4; ++q) u[q] = 0.0f;
    if (!unit32<M>(f, sz, sa, u)) {  // out of the FP32 form's range
        double fp[M], ss = 0.0;
#pragma unroll
        for (int q = 0; q < M; ++q) {
            fp[q] = __ddiv_rn(__dsub_rn((double)f[q], c->zstar[q]), c->a[q]);
            ss = __dadd_rn(ss, __dmul_rn(fp[q], fp[q]));
        }
        const double nf = __dsqrt_rn(ss), inv = nf > 0.0 ? 1.0 / nf : 0.0;
#pragma unroll
        for (int q = 0; q < M; ++q) u[q] = __double2float_rn(fp[q] * inv);
    }
#pragma unroll
    for (int q4 = 0; q4 < M4 / 4; ++q4)
        reinterpret_cast<float4*>(v.uhat + (size_t)s * M4)[q4] = make_float4(u[4 * q4], u[4 * q4 + 1], u[4 * q4 + 2], u[4 * q4 + 3]);
    unsigned short r[KP];
#pragma unroll
    for (int e = 0; e < KP; ++e) r[e] = 0;
#pragma unroll
    for (int q = 0; q < M; ++q) {
        const __half h = __float2half_rn(u[q]);
        const __half l = __float2half_rn(u[q] - __half2float(h));
        r[q] = r[M + q] = __half_as_ushort(h);
        r[2 * M + q] = __half_as_ushort(l);
    }
    unsigned char* a = v.aop + (size_t)(s / 128) * (KP * 256) + (s % 128) * 16;
#pragma unroll
    for (int k = 0; k < KP / 8; ++k) {
        uint4 x;
        x.x = r[8 * k + 0] | ((uint32_t)r[8 * k + 1] << 16);
        x.y = r[8 * k + 2] | ((uint32_t)r[8 * k + 3] << 16);
        x.z = r[8 * k + 4] | ((uint32_t)r[8 * k + 5] << 16);
        x.w = r[8 * k + 6] | ((uint32_t)r[8 * k + 7] << 16);
        *reinterpret_cast<uint4*>(a + k * 2048) = x;
    }
}

// Cosines of every point with every direction on the tensor cores, reduced
// to block maxima.  The points' rows [h, h, l] and the directions' rows
// [zh, zl, zh] make one FP16 product with FP32 accumulators equal to
// u . z without the l l term: within MMA_ERR of it (splits: 2^-23 per
// component, so about 2 sqrt(m) 2^-23; l l below m 2^-24; at most 32
// accumulations of partial sums below 1, each truncated at 2^-24; together
// below 3.4e-6).
//
// A CTA takes work items: a group of TP = 256 points (two tiles of 128 rows)
// against a range of chunks of 128 directions.  Per step one chunk meets each
// tile: an MMA (128 x 128 x KP) into one of the tile's two TMEM accumulators
// (all 512 columns).  A warpgroup per tile reads them (a thread one point's
// 128 cosines; tcgen05.ld.red forms the maximum of 32 columns in the load) as
// the maxima of four blocks of 32 directions; a warp per tile issues the MMAs
// and one the bulk copies (the chunks are stored as the MMA reads them:
// K-major core matrices of 8 rows x 16 bytes, so a chunk is one contiguous
// copy; a ring of eight).  Full / empty barriers per accumulator and ring
// slot let the warps drift.  Per point and item the scan keeps the two best
// blocks and the third-best maximum, without a branch.  The block that holds
// the exact nearest direction has a maximum within MBAND of the best:
// k_assoc_final rescans the listed blocks within MBAND of the best in FP32,
// and a point whose third maximum in some item is within it too (about one
// in 20,000) takes the FP32 scan over all directions (k_assoc_slow).
//
// Bound: the chain of product, load and barrier of a step; the tensor pipe is
// busy 32 % of the time at m = 8 and 15 % at m = 5 (K is 32 and 16, so an MMA is
// short against the read of its accumulator).  Measured at m = 8, 38,700 points
// and 11,440 directions, and m = 5, 21,000 points and 10,626 directions:
// 36 and 16-22 us.  FP32 FMAs took 173 us at m = 8 (the FMA pipe's time), a
// scan pruned by cone bounds 42-52 us at m = 5; on the way here: a branch per
// block that lists every block near the best 102 us (m = 8), a block barrier
// per step 56, four tiles of 64 directions 42.
// That bound takes every accumulation as truncated, which no document states:
// measured over 4.3 million block maxima, m = 2 to 10, of points and directions at
// random, 1e-7 .. 1 from an axis and from the centre and with components down
// to 1e-6 of the rest, the largest error is 4.1e-7 (4.4e-7 against the exact
// cosines; the FP32 form's bound is (m + 7) 2^-24, up to 1.0e-6).
constexpr float MMA_ERR = 4.5e-6f;
constexpr float MBAND = 2.0f * MMA_ERR + 3e-6f;  // + the FP32 unit vectors' own error, both sides
constexpr int TILES = 2;            // tiles of 128 points per item, a warpgroup each
constexpr int TP = 128 * TILES;     // points per item
constexpr int MT = TP + 32 * (TILES + 1);  // threads per CTA: one per point, an issuing warp per tile, a loading warp
constexpr int CHUNK = 128;          // directions per step
constexpr int SETS = 512 / (TILES * CHUNK);  // accumulators per tile (512 TMEM columns)
constexpr int RING = 8;             // chunks in shared memory

// items of nT points and nch chunks over `grid` CTAs: groups of points,
// splits per group and chunks per split, the same on the device for both
// kernels and on the host for the maximum.  The split count minimises the
// waves of the grid times the chunks of an item (plus an item's own cost of
// about six chunks), over at most twice the count that fills the grid once
// (so that items <= 2 (grid + groups)).
__host__ __device__ __forceinline__ void tile_split(int nT, int nch, int grid, int& ntile, int& S, int& cps)
{
    ntile = (nT + TP - 1) / TP;
    S = 1;
    cps = nch;
    if (ntile == 0 || nch == 0) return;
    const int fill = (grid + ntile - 1) / ntile;
    const int smax = nch < 2 * fill ? nch : 2 * fill;
    unsigned best = 0xffffffffu;
    for (int t = 1; t <= smax; ++t) {
        const unsigned b = (unsigned)(nch + t - 1) / t;
        const unsigned st = (nch + b - 1) / b;
        const unsigned cost = ((ntile * st + grid - 1) / grid) * (b + 6);  // (all below 2^26)
        if (cost < best) {
            best = cost;
            S = st;
            cps = b;
        }
    }
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* b, uint32_t n)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long* b, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* b)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
// Waits for the barrier's phase of this parity, at most wait_ns of device
// time; false when it did not come or another thread's wait ran out (*fail).
__device__ __forceinline__ bool mbar_wait(unsigned long long* b, uint32_t parity, unsigned long long wait_ns, volatile int* fail)
{
    const uint32_t a = smem_u32(b);
    unsigned long long t0 = 0ull;
    for (unsigned it = 0;; ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(a), "r"(parity)
                     : "memory");
        if (done) return true;
        if ((it & 63u) == 63u) {
            if (*fail) return false;
            const unsigned long long t = global_ns();
            if (t0 == 0ull) t0 = t;
            if (t - t0 > wait_ns || it > (1u << 28)) {
                *fail = 1;
                return false;
            }
        }
    }
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, unsigned long long* b)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(b))
                 : "memory");
}
// K-major operand of `rows` rows without swizzle: core matrices of 8 rows x
// 16 bytes, 16 rows bytes apart along K, 128 bytes apart along the rows
__device__ __forceinline__ unsigned long long mma_desc(uint32_t addr, uint32_t rows)
{
    return (unsigned long long)((addr >> 4) & 0x3fffu) | (unsigned long long)rows << 16 |
           (unsigned long long)(128u >> 4) << 32 | 1ull << 46;
}
__device__ __forceinline__ void mma_f16(uint32_t d, unsigned long long a, unsigned long long b, uint32_t idesc, bool add)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
                 "l"(a), "l"(b), "r"(idesc), "r"(add ? 1 : 0)
                 : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned long long* b)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(b)) : "memory");
}
// Maximum of 32 accumulator columns of each of this warp's 32 lanes, formed
// by the load itself (the loaded values are not used, but their registers are
// not free before the load's wait: tmem_keep after it)
__device__ __forceinline__ void tmem_max32(uint32_t a, float& mx, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.red.sync.aligned.32x32b.x32.max.f32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, %32, [%33];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
                   "=f"(mx)
                 : "r"(a));
}
__device__ __forceinline__ void tmem_keep(const uint32_t (&r)[32])
{
#pragma unroll
    for (int k = 0; k < 32; ++k) asm volatile("" ::"r"(r[k]));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// dynamic shared memory: the point tiles, the ring of chunks
template <int KP>
constexpr size_t mma_smem() { return (size_t)(TP + RING * CHUNK) * KP * 2 + 1024; }

template <int KP>
__global__ void __launch_bounds__(MT, 1) k_assoc_mma(RunView v)
{
    constexpr uint32_t ATILE = 128 * KP * 2, BTILE = CHUNK * KP * 2;  // bytes
    // M = 128, N = CHUNK, FP16 operands, FP32 accumulators
    constexpr uint32_t IDESC = (1u << 4) | ((CHUNK >> 3) << 17) | ((128u >> 4) << 24);
    extern __shared__ unsigned char raw[];
    // loads landed (points, ring slots); slots and tiles free again (an arrival
    // per issuing thread); per set and tile: accumulator written, read
    __shared__ unsigned long long bar_a, bar_afree, bar_b[RING], bar_bfree[RING], bar_full[SETS][TILES], bar_empty[SETS][TILES];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    Ctrl* c = v.ctrl;
    const int tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    if (__syncthreads_or(skip_niche(c))) return;  // the same for every thread of the CTA
    const int nT = c->nT, nch = (v.w + CHUNK - 1) / CHUNK;
    int ntile, S, cps;
    tile_split(nT, nch, gridDim.x, ntile, S, cps);
    const int items = ntile * S;
    if ((int)blockIdx.x >= items) return;
    unsigned char* As = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* Bs = As + TILES * ATILE;
    if (tid == 0) {
        mbar_init(&bar_a, 1);
        mbar_init(&bar_afree, TILES);
        for (int k = 0; k < RING; ++k) {
            mbar_init(&bar_b[k], 1);
            mbar_init(&bar_bfree[k], TILES);
        }
        for (int k = 0; k < SETS * TILES; ++k) {
            mbar_init(&bar_full[k / TILES][k % TILES], 1);
            mbar_init(&bar_empty[k / TILES][k % TILES], 4);  // a lane of each of the tile's reading warps
        }
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == TP / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tmem = s_tmem;
    volatile int* fail = &s_fail;
    auto wait = [&](unsigned long long* bar, uint32_t n) { return mbar_wait(bar, n & 1u, v.wait_ns, fail); };
    // (after a failed wait: the end of what is in flight, or the limit)
    int over = 0;  // (one limit for all of a thread's)
    auto drain = [&](unsigned long long* bar, uint32_t n) { return mbar_wait(bar, n & 1u, v.wait_ns, &over); };
    if (warp == TP / 32 + TILES) {  // loads
        if (lane == 0) {
            uint32_t nload = 0, nitem = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < items && ok; it += gridDim.x, ++nitem) {
                const int g = it / S, sp = it - g * S;
                const int c0 = sp * cps, c1 = min(nch, c0 + cps);
                if (nitem > 0) ok = wait(&bar_afree, nitem - 1);  // the previous item's products are formed
                if (!ok) break;
                mbar_expect(&bar_a, TILES * ATILE);
                bulk_load(As, v.aop + (size_t)g * TILES * ATILE, TILES * ATILE, &bar_a);
                for (int ch = c0; ch < c1; ++ch, ++nload) {
                    const uint32_t k = nload % RING;
                    if (nload >= RING) ok = wait(&bar_bfree[k], nload / RING - 1);
                    if (!ok) break;
                    mbar_expect(&bar_b[k], BTILE);
                    bulk_load(Bs + k * BTILE, v.bop + (size_t)ch * BTILE, BTILE, &bar_b[k]);
                }
            }
            if (!ok) {
                set_status(c, DEV_ETIMEOUT);
                drain(&bar_a, nitem);
                for (uint32_t k = nload > RING ? nload - RING : 0u; k < nload; ++k) drain(&bar_b[k % RING], k / RING);
            }
        }
        __syncwarp();
    } else if (warp >= TP / 32) {  // products of tile t
        if (lane == 0) {
            const int t = warp - TP / 32;
            const uint32_t a = smem_u32(As) + t * ATILE;
            uint32_t nstep = 0, nitem = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < items && ok; it += gridDim.x, ++nitem) {
                const int sp = it % S;
                const int c0 = sp * cps, c1 = min(nch, c0 + cps);
                ok = wait(&bar_a, nitem);
                for (int ch = c0; ch < c1 && ok; ++ch, ++nstep) {
                    const uint32_t k = nstep % RING, set = nstep % SETS;
                    ok = wait(&bar_b[k], nstep / RING);
                    // the accumulator's last maxima are taken
                    if (ok && nstep >= SETS) ok = wait(&bar_empty[set][t], nstep / SETS - 1u);
                    if (!ok) break;
                    tmem_fence_after();
                    const uint32_t b = smem_u32(Bs) + k * BTILE, d = tmem + (set * TILES + t) * CHUNK;
#pragma unroll
                    for (int kk = 0; kk < KP / 16; ++kk)
                        mma_f16(d, mma_desc(a + kk * 4096, 128), mma_desc(b + kk * CHUNK * 32, CHUNK), IDESC, kk > 0);
                    mma_commit(&bar_full[set][t]);
                    mma_commit(&bar_bfree[k]);
                }
                if (ok) mma_commit(&bar_afree);
            }
            // The commits' arrivals on the barriers land before the CTA, and
            // the barriers with it, is gone: the accumulators' are waited for
            // by the maxima, those that free slots and tiles here (each
            // barrier's last phase; the one before it is over, or the load
            // that this thread waited for would not have been made).
            const uint32_t s0 = nstep > RING ? nstep - RING : 0u;
            if (ok) ok = wait(&bar_afree, nitem - 1);
            for (uint32_t k = s0; k < nstep && ok; ++k) ok = wait(&bar_bfree[k % RING], k / RING);
            if (!ok) {
                set_status(c, DEV_ETIMEOUT);
                for (uint32_t k = nstep > SETS ? nstep - SETS : 0u; k < nstep; ++k) drain(&bar_full[k % SETS][t], k / SETS);
                for (uint32_t k = s0; k < nstep; ++k) drain(&bar_bfree[k % RING], k / RING);
            }
        }
        __syncwarp();
    } else {  // maxima of tile t; the warp reads lanes 32 (warp & 3) ...
        const int t = warp >> 2;
        const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
        uint32_t nstep = 0;
        bool ok = true;
        for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
            const int g = it / S, sp = it - g * S;
            const int c0 = sp * cps, c1 = min(nch, c0 + cps);
            // this thread's point: best, second and third block maximum, the
            // blocks of the first two
            float b1 = -4.0f, b2 = -4.0f, b3 = -4.0f;
            int k1 = 0, k2 = 0;
            for (int ch = c0; ch < c1; ++ch, ++nstep) {
                const uint32_t set = nstep % SETS;
                ok = wait(&bar_full[set][t], nstep / SETS);
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0) set_status(c, DEV_ETIMEOUT);
                    ok = false;
                    break;
                }
                tmem_fence_after();
                const uint32_t ta = tmem + lanes + (set * TILES + t) * CHUNK;
                float bm[CHUNK / 32];
#pragma unroll
                for (int h = 0; h < CHUNK / 32; h += 2) {
                    uint32_t r0[32], r1[32];
                    tmem_max32(ta + 32 * h, bm[h], r0);
                    tmem_max32(ta + 32 * h + 32, bm[h + 1], r1);
                    tmem_ld_wait();
                    tmem_keep(r0);
                    tmem_keep(r1);
                }
                tmem_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bar_empty[set][t]);
#pragma unroll
                for (int h = 0; h < CHUNK / 32; ++h) {
                    const int blk = ch * (CHUNK / 32) + h;
                    const bool g1 = bm[h] > b1, g2 = bm[h] > b2;
                    b3 = fmaxf(b3, fminf(b2, bm[h]));
                    k2 = g1 ? k1 : g2 ? blk : k2;
                    b2 = fmaxf(b2, fminf(b1, bm[h]));
                    k1 = g1 ? blk : k1;
                    b1 = fmaxf(b1, bm[h]);
                }
            }
            if (ok && g * TP + tid < nT)  // (blocks number below 2^16)
                v.aent[(size_t)it * TP + tid] = make_int4(__float_as_int(b1), __float_as_int(b2), __float_as_int(b3),
                                                          k1 | (k2 << 16));
        }
    }
    tmem_fence_before();
    __syncthreads();
    if (warp == TP / 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

__device__ __forceinline__ void write_assoc(const RunView& v, Ctrl* c, int i, int rk, int j, double d)
{
    // no candidate: f' and the intercepts are finite here (not_finite_key), so an invariant failed
    if ((unsigned)j >= (unsigned)v.w) {
        set_status(c, DEV_EINTERNAL);
        return;
    }
    v.pi[i] = j;
    v.dist[i] = d;
    if (rk < c->l)
        atomicAdd(&v.rho[j], 1);
    else
        atomicAdd(&v.rhop[j], 1);
}

// Per point the best maximum over the items and the blocks within MBAND of it
// (a thread per T slot); a warp rescans its 32 points' blocks in FP32, a lane
// per direction (coalesced rows; a thread rescanning its own blocks read 32
// scattered lines per load: 26 us at m = 8, 38,700 points); then per thread
// f' and |f'| in FP64 and the FP64 distances of the directions within the
// FP32 band of the best (usually one), and their lexicographic (d, j)
// minimum.  A point with more than FT_BLK blocks or FT_CAND candidates, or a
// third block within MBAND in one item, takes the FP32 scan over all
// directions.
constexpr int FB = 128;
constexpr int FT_BLK = 4;
constexpr int FT_CAND = 8;

// f' and |f'| of objectives f, in FP64
template <int M>
__device__ __forceinline__ double fprime_of(const Ctrl* c, const float* f, double (&fp)[M])
{
    double ss = 0.0;
#pragma unroll
    for (int q = 0; q < M; ++q) {
        fp[q] = sf64::div(__dsub_rn((double)f[q], c->zstar[q]), c->da[q]);
        ss = __dadd_rn(ss, __dmul_rn(fp[q], fp[q]));
    }
    return sf64::sqrt_rn(ss);
}

template <int M>
__global__ void __launch_bounds__(FB) k_assoc_final(RunView v)
{
    constexpr int M4 = (M + 3) & ~3, Q4 = M4 / 4;
    __shared__ int sblk[FT_BLK][FB];
    __shared__ int scand[FT_CAND][FB];
    __shared__ float scos[FT_CAND][FB];
    __shared__ unsigned sjob[FB * FT_BLK];
    __shared__ __align__(16) float suh[FB * M4];
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int nT = c->nT;
    const int tid = threadIdx.x, lane = lane_id(), wb = tid & ~31;
    const int s = blockIdx.x * FB + tid;
    if (blockIdx.x * FB >= nT) return;
    int ntile, S, cps;
    tile_split(nT, (v.w + CHUNK - 1) / CHUNK, v.assoc_grid, ntile, S, cps);
    const int tile = s / TP, l = s - tile * TP;
    const bool in = s < nT;
    // the point's objectives and rank, used after the rescans
    int i = 0, rk = 0;
    float f[M];
    if (in) {
        i = v.Tlist[s];
        rk = v.rank2[i];
    }
#pragma unroll
    for (int q = 0; q < M; ++q) f[q] = in ? v.F[(size_t)i * M + q] : 0.0f;
    bool ovf = false, third = false;
    int nblk = 0;
    if (in) {
        float gbest = -4.0f;
        const int4* ent = v.aent + (size_t)tile * S * TP + l;
        for (int sp = 0; sp < S; ++sp) gbest = fmaxf(gbest, __int_as_float(ent[(size_t)sp * TP].x));
        const float thr = gbest - MBAND;
        for (int sp = 0; sp < S; ++sp) {
            const int4 e = ent[(size_t)sp * TP];
            third = third || __int_as_float(e.z) >= thr;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (__int_as_float(k ? e.y : e.x) < thr) continue;
                if (nblk == FT_BLK)
                    ovf = true;
                else
                    sblk[nblk++][tid] = (e.w >> (16 * k)) & 0xffff;
            }
        }
        if (ovf || third) nblk = 0;
    }
    // the warp's rescans as a list of (point, block), its points' unit vectors
    // in shared memory; JB rescans' loads in flight together
    int at = nblk;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += y;
    }
    const int njob = __shfl_sync(0xffffffffu, at, 31);
    at -= nblk;
    unsigned* job = sjob + (wb >> 5) * (32 * FT_BLK);
    for (int b = 0; b < nblk; ++b) job[at + b] = (unsigned)sblk[b][tid] * 32u + (unsigned)lane;
    float* su = suh + (size_t)wb * M4;
#pragma unroll
    for (int q4 = 0; q4 < Q4; ++q4)
        reinterpret_cast<float4*>(su + lane * M4)[q4] =
            in ? reinterpret_cast<const float4*>(v.uhat + (size_t)s * M4)[q4] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    __syncwarp();
    const float band = cos_band<M>();
    float best = -4.0f;
    int ncand = 0;
    const float4* bz4 = reinterpret_cast<const float4*>(v.blk_z);
    constexpr int JB = M4 <= 8 ? 8 : 4;  // rescans whose loads are in flight together
    for (int j0 = 0; j0 < njob; j0 += JB) {
        float qv[JB];
        int pos[JB], pt[JB];
        float4 z[JB][Q4];
#pragma unroll
        for (int t = 0; t < JB; ++t) {
            const unsigned x = job[min(j0 + t, njob - 1)];
            pt[t] = (int)(x & 31u);
            pos[t] = (int)(x & ~31u) + lane;
#pragma unroll
            for (int q4 = 0; q4 < Q4; ++q4) z[t][q4] = __ldg(bz4 + (size_t)min(pos[t], v.w - 1) * Q4 + q4);
        }
#pragma unroll
        for (int t = 0; t < JB; ++t) {
            const float* u = su + pt[t] * M4;
            float a = 0.0f;
#pragma unroll
            for (int q4 = 0; q4 < Q4; ++q4) {
                const float4 y = reinterpret_cast<const float4*>(u)[q4];
                a = fmaf(y.x, z[t][q4].x, a);
                if (4 * q4 + 1 < M) a = fmaf(y.y, z[t][q4].y, a);
                if (4 * q4 + 2 < M) a = fmaf(y.z, z[t][q4].z, a);
                if (4 * q4 + 3 < M) a = fmaf(y.w, z[t][q4].w, a);
            }
            qv[t] = a;
        }
#pragma unroll
        for (int t = 0; t < JB; ++t) {
            if (j0 + t >= njob) break;
            const int p = pt[t];
            const bool ref = pos[t] < v.w;
            // cosines are >= 0: their bits order like unsigned ints
            const float bm = __uint_as_float(__reduce_max_sync(0xffffffffu, ref ? __float_as_uint(fmaxf(qv[t], 0.0f)) : 0u));
            const float run = fmaxf(__shfl_sync(0xffffffffu, best, p), bm);
            const int n = __shfl_sync(0xffffffffu, ncand, p);
            const bool take = ref && qv[t] >= run - band;
            const unsigned bal = __ballot_sync(0xffffffffu, take);
            if (take) {
                const int e = n + __popc(bal & ((1u << lane) - 1u));
                if (e < FT_CAND) {
                    scand[e][wb + p] = pos[t];
                    scos[e][wb + p] = qv[t];
                }
            }
            if (lane == p) {
                best = run;
                ncand = n + __popc(bal);
            }
        }
    }
    __syncwarp();
    if (!in) return;
    double fp[M];
    const double nf = fprime_of<M>(c, f, fp);
    const bool zero = sf64::is_zero(nf);  // every distance is 0: the first direction
    double bd = 0.0;
    int bj = 0;
    if (!zero) {
        if (ovf || third || ncand > FT_CAND) {
            v.arun[s] = make_int2(third ? -2 : -1, 0);  // (-1: a list overflowed)
            v.slow[atomicAdd(&c->nslow, 1)] = s;
            return;
        }
        bd = CUDART_INF;
        bj = 0x7fffffff;
        for (int e = 0; e < ncand; ++e) {
            if (scos[e][tid] < best - band) continue;
            const int j = v.blk_j[scand[e][tid]];
            const double d = perp_dist(fp, nf, v.Zd + (size_t)j * M, v.nz[j], M);
            if (lex_less(d, j, bd, bj)) {
                bd = d;
                bj = j;
            }
        }
    }
    if (v.debug_recheck_all) {
        v.dist[i] = bd;  // compared by k_assoc_slow
        v.pi[i] = bj;
        v.arun[s] = make_int2(0, 0);
        v.slow[atomicAdd(&c->nslow, 1)] = s;
        return;
    }
    write_assoc(v, c, i, rk, bj, bd);
}

// The points of the slow list where there are many (m <= 10; objectives of a
// few values tie with directions of many blocks), GP of them per CTA.  A warp
// forms the FP32 cosines of GT points with every direction at once, for their
// maxima and then for the directions within the band of them; f' and |f'| take
// a thread per point and the FP64 distances a thread per candidate, which the
// FP64 pipe and the fixed-point quotients serve 32 at a time.  A CTA per point
// (below) repeats f' in every warp.  Niching of objectives of five values at
// m = 10, 2N = 66,000, 220 directions: 552 us with a CTA per point, 162 here;
// at 2N = 10,000, 2,002 directions 461 and 180.
constexpr int GP = 32;
constexpr int GT = GP / (AB / 32);
constexpr int GC = 32;  // candidates of a point; with more, the CTA takes it alone

template <int M>
struct SlowShared {
    int j[GP][GC];
    int n[GP], pt[GP], bj[GP];
    unsigned long long bd[GP];
    float thr[GP], u[GP][M];
    double fp[GP][M], nf[GP];
};

template <int M>
__device__ __forceinline__ void assoc_groups(const RunView& v, Ctrl* c, int ns, SlowShared<M>& sh)
{
    constexpr int M4 = (M + 3) & ~3;
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5, w = v.w;
    for (int g0 = blockIdx.x * GP; g0 < ns; g0 += gridDim.x * GP) {
        const int np = min(GP, ns - g0);
        __syncthreads();  // the last group is written
        if (tid < GP) {
            sh.pt[tid] = v.slow[min(g0 + tid, ns - 1)];
            sh.n[tid] = 0;
            sh.bd[tid] = ~0ull;
            sh.bj[tid] = 0x7fffffff;
        }
        __syncthreads();
        for (int e = tid; e < GP * M; e += AB) {
            const int p = e / M, q = e - p * M;
            sh.u[p][q] = v.uhat[(size_t)sh.pt[p] * M4 + q];
        }
        __syncthreads();
        {
            float u[GT][M], b[GT];
#pragma unroll
            for (int t = 0; t < GT; ++t) {
                b[t] = 0.0f;
#pragma unroll
                for (int q = 0; q < M; ++q) u[t][q] = sh.u[warp * GT + t][q];
            }
            auto dots = [&](int j, float (&x)[GT]) {
                const float4* z4 = reinterpret_cast<const float4*>(v.Zh + (size_t)j * M4);
                float z[M4];
#pragma unroll
                for (int q4 = 0; q4 < M4 / 4; ++q4) {
                    const float4 y = __ldg(z4 + q4);
                    z[4 * q4 + 0] = y.x;
                    z[4 * q4 + 1] = y.y;
                    z[4 * q4 + 2] = y.z;
                    z[4 * q4 + 3] = y.w;
                }
#pragma unroll
                for (int t = 0; t < GT; ++t) {
                    float s = 0.0f;
#pragma unroll
                    for (int q = 0; q < M; ++q) s = fmaf(u[t][q], z[q], s);
                    x[t] = s;
                }
            };
#pragma unroll 4
            for (int j = lane; j < w; j += 32) {
                float x[GT];
                dots(j, x);
#pragma unroll
                for (int t = 0; t < GT; ++t) b[t] = fmaxf(b[t], x[t]);
            }
#pragma unroll
            for (int t = 0; t < GT; ++t) {  // cosines are >= 0: their bits order like unsigned ints
                b[t] = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(b[t]))) - cos_band<M>();
                if (lane == 0) sh.thr[warp * GT + t] = b[t];
            }
#pragma unroll 4
            for (int j = lane; j < w; j += 32) {
                float x[GT];
                dots(j, x);
#pragma unroll
                for (int t = 0; t < GT; ++t)
                    if (x[t] >= b[t]) {
                        const int e = atomicAdd(&sh.n[warp * GT + t], 1);
                        if (e < GC) sh.j[warp * GT + t][e] = j;
                    }
            }
        }
        if (tid < np) {
            double fp[M];
            sh.nf[tid] = fprime_of<M>(c, v.F + (size_t)v.Tlist[sh.pt[tid]] * M, fp);
#pragma unroll
            for (int q = 0; q < M; ++q) sh.fp[tid][q] = fp[q];
        }
        __syncthreads();
        // distances are >= 0 and order like their bits
        unsigned long long d[GP * GC / AB];
#pragma unroll
        for (int k = 0; k < GP * GC / AB; ++k) {
            const int p = (tid + k * AB) / GC, e = tid % GC;
            d[k] = ~0ull;
            if (p < np && sh.n[p] <= GC && e < sh.n[p]) {
                const int j = sh.j[p][e];
                d[k] = sf64::bits(perp_dist(sh.fp[p], sh.nf[p], v.Zd + (size_t)j * M, v.nz[j], M));
                atomicMin(&sh.bd[p], d[k]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < GP * GC / AB; ++k) {
            const int p = (tid + k * AB) / GC;
            if (d[k] != ~0ull && d[k] == sh.bd[p]) atomicMin(&sh.bj[p], sh.j[p][tid % GC]);
        }
        for (int p = 0; p < np; ++p) {
            if (sh.n[p] <= GC) continue;  // the same for every thread
            unsigned long long b = ~0ull;
            int bj = 0x7fffffff;
            for (int j = tid; j < w; j += AB) {
                float x = 0.0f;
#pragma unroll
                for (int q = 0; q < M; ++q) x = fmaf(sh.u[p][q], __ldg(v.Zh + (size_t)j * M4 + q), x);
                if (x < sh.thr[p]) continue;
                const unsigned long long dj = sf64::bits(perp_dist(sh.fp[p], sh.nf[p], v.Zd + (size_t)j * M, v.nz[j], M));
                if (dj < b) {  // (j ascends)
                    b = dj;
                    bj = j;
                }
            }
            atomicMin(&sh.bd[p], b);
            __syncthreads();
            if (b != ~0ull && b == sh.bd[p]) atomicMin(&sh.bj[p], bj);
        }
        __syncthreads();
        if (tid < np) {
            const int i = v.Tlist[sh.pt[tid]];
            if (v.arun[sh.pt[tid]].x == -1) atomicAdd(&c->overflow, 1);
            write_assoc(v, c, i, v.rank2[i], sh.bj[tid], sf64::value(sh.bd[tid]));
        }
    }
}

// One point per CTA over all directions: points whose lists overflowed, and
// in debug mode every point.  m <= 10: the best FP32 cosine, then the FP64
// distances of the directions within the band of it (in debug mode and for
// m > 10, M = 0, of every direction).
template <int M>
__global__ void __launch_bounds__(AB) k_assoc_slow(RunView v)
{
    __shared__ double sd[AB / 32];
    __shared__ int sj[AB / 32];
    __shared__ unsigned s_best;
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int ns = c->nslow;
    if constexpr (M > 0) {
        __shared__ SlowShared<M> sh;
        // waves of either form times a CTA's time in one: 0.24 us per 256
        // directions and 4 us, 0.18 us per 32 and 6 us
        const int grid = gridDim.x, single = (ns + grid - 1) / grid, group = (ns + GP * grid - 1) / (GP * grid);
        if (!v.debug_recheck_all && (long long)group * (6 * v.w + 6400) < (long long)single * (v.w + 4267)) {
            assoc_groups<M>(v, c, ns, sh);
            return;
        }
    }
    const int m = M > 0 ? M : v.m;
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    for (int t = blockIdx.x; t < ns; t += gridDim.x) {
        const int pt = v.slow[t];
        double fr[M > 0 ? M : 1], nf;
        float thr = -4.0f, u[M > 0 ? M : 1];
        if constexpr (M > 0) {
            constexpr int M4 = (M + 3) & ~3;
            nf = fprime_of<M>(c, v.F + (size_t)v.Tlist[pt] * M, fr);
#pragma unroll
            for (int q = 0; q < M; ++q) u[q] = v.uhat[(size_t)pt * M4 + q];
            if (!v.debug_recheck_all) {
                if (threadIdx.x == 0) s_best = 0u;
                __syncthreads();
                float b = 0.0f;
                for (int j = threadIdx.x; j < v.w; j += AB) {
                    float x = 0.0f;
#pragma unroll
                    for (int q = 0; q < M; ++q) x = fmaf(u[q], __ldg(v.Zh + (size_t)j * M4 + q), x);
                    b = fmaxf(b, x);
                }
                const unsigned wm = __reduce_max_sync(0xffffffffu, __float_as_uint(b));  // cosines are >= 0
                if (lane == 0) atomicMax(&s_best, wm);
                __syncthreads();
                thr = __uint_as_float(s_best) - cos_band<M>();
            }
        } else {
            nf = v.fnorm[pt];
        }
        const double* fp = M > 0 ? fr : v.fprime + (size_t)pt * m;
        double d0 = CUDART_INF;
        int j0 = 0x7fffffff;
        for (int j = threadIdx.x; j < v.w; j += AB) {
            if constexpr (M > 0) {
                constexpr int M4 = (M + 3) & ~3;
                float x = 0.0f;
#pragma unroll
                for (int q = 0; q < M; ++q) x = fmaf(u[q], __ldg(v.Zh + (size_t)j * M4 + q), x);
                if (x < thr) continue;
            }
            const double d = perp_dist(fp, nf, v.Zd + (size_t)j * m, v.nz[j], m);
            if (lex_less(d, j, d0, j0)) {
                d0 = d;
                j0 = j;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double od = __shfl_xor_sync(0xffffffffu, d0, o);
            const int oj = __shfl_xor_sync(0xffffffffu, j0, o);
            if (lex_less(od, oj, d0, j0)) {
                d0 = od;
                j0 = oj;
            }
        }
        if (lane == 0) {
            sd[warp] = d0;
            sj[warp] = j0;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < AB / 32; ++q)
                if (lex_less(sd[q], sj[q], d0, j0)) {
                    d0 = sd[q];
                    j0 = sj[q];
                }
            const int i = v.Tlist[pt];
            if (v.arun[pt].x < 0) {
                if (v.arun[pt].x == -1) atomicAdd(&c->overflow, 1);
            } else if (v.debug_recheck_all && (v.pi[i] != j0 || v.dist[i] != d0)) {
                atomicAdd(&c->recheck_miss, 1);
            }
            write_assoc(v, c, i, v.rank2[i], j0, d0);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// m > NSGA3_FAST_M: runtime m, no pruning (the cone bounds lose their grip in
// many dimensions).  A CTA keeps the unit vectors of GPP points in shared
// memory; each warp forms the FP32 cosines of all of them against its
// tiles of 32 references (a lane per reference, read as float4 through the
// read-only cache) and feeds them to the same candidate band; the FP64
// kernels read f' from memory and keep their pipe full (a thread per point
// or per candidate for the sequential sums).

// f' = (f - z*) / a for every element (a thread per element: the divisions
// spread over every SM), then per point (a thread per point: the FP64 pipe
// serves 32 points per warp instruction) the squares added left to right,
// |f'| and the FP32 unit vector
__global__ void __launch_bounds__(256) k_assoc_prep_elem(RunView v)
{
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int m = v.m;
    const long long e = (long long)blockIdx.x * 256 + threadIdx.x;
    if (e >= (long long)c->nT * m) return;
    const int s = (int)(e / m), q = (int)(e - (long long)s * m);
    const int i = v.Tlist[s];
    v.fprime[e] = __ddiv_rn(__dsub_rn((double)v.F[(size_t)i * m + q], c->zstar[q]), c->a[q]);
}

// one warp per CTA, 32 points: the rows come in through a 32 x 32 tile
// (coalesced loads), lane p adds the squares of point p left to right
__global__ void __launch_bounds__(32) k_assoc_prep_norm(RunView v)
{
    __shared__ double tile[32][33];
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int nT = c->nT, s0 = blockIdx.x * 32, lane = threadIdx.x;
    if (s0 >= nT) return;
    const int m = v.m, M4 = v.M4, np = min(32, nT - s0);
    const double* base = v.fprime + (size_t)s0 * m;
    double ss = 0.0;
    for (int q0 = 0; q0 < m; q0 += 32) {
        const int nq = min(32, m - q0);
#pragma unroll 8
        for (int p = 0; p < np; ++p) tile[p][lane] = lane < nq ? base[(size_t)p * m + q0 + lane] : 0.0;
        __syncwarp();
        if (lane < np)
            for (int t = 0; t < nq; ++t) ss = __dadd_rn(ss, __dmul_rn(tile[lane][t], tile[lane][t]));
        __syncwarp();
    }
    const double nf = __dsqrt_rn(ss);
    if (lane < np) v.fnorm[s0 + lane] = nf;
    const double inv = nf > 0.0 ? 1.0 / nf : 0.0;
    for (int p = 0; p < np; ++p) {
        const double ip = __shfl_sync(0xffffffffu, inv, p);
#pragma unroll 8
        for (int q = lane; q < M4; q += 32)
            v.uhat[(size_t)(s0 + p) * M4 + q] = q < m ? __double2float_rn(base[(size_t)p * m + q] * ip) : 0.0f;
    }
}

constexpr int GW = 8;  // warps per CTA of the m > NSGA3_FAST_M scan

// candidate-list update of one point with a block of 32 cosines (qh, j) per
// lane (j = -1: no reference): keeps every reference within band of the best
// so far; a list that cannot hold them marks the point as overflowed
__device__ __forceinline__ void band_take(float qh, int j, float band, float& best, int& nl, bool& ovf,
                                          int* lj, float* lq, int cap)
{
    const int lane = lane_id();
    const float wm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(qh, 0.0f))));
    best = fmaxf(best, wm);
    const bool keep = j >= 0 && qh >= best - band;
    unsigned bal = __ballot_sync(0xffffffffu, keep);
    if (nl + __popc(bal) > cap) {  // drop entries that fell out of the band
        __syncwarp();
        int kept = 0;
        for (int e0 = 0; e0 < nl; e0 += 32) {
            const int e = e0 + lane;
            const bool k2 = e < nl && lq[e] >= best - band;
            const unsigned b2 = __ballot_sync(0xffffffffu, k2);
            int jj = 0;
            float qq = 0.0f;
            if (k2) {
                jj = lj[e];
                qq = lq[e];
            }
            __syncwarp();
            if (k2) {
                const int p = kept + __popc(b2 & ((1u << lane) - 1u));
                lj[p] = jj;
                lq[p] = qq;
            }
            kept += __popc(b2);
            __syncwarp();
        }
        nl = kept;
        if (nl + __popc(bal) > cap) {
            ovf = true;
            bal = 0u;
        }
    }
    if (keep && bal) {
        const int p = nl + __popc(bal & ((1u << lane) - 1u));
        lj[p] = j;
        lq[p] = qh;
    }
    nl += __popc(bal);
    __syncwarp();
}

constexpr int GPP = 8;   // points per CTA (every warp works on all of them)
constexpr int LCW = 64;  // candidate slots per warp and point

// dynamic shared memory: the points' unit vectors (GPP x M4) and the lists
size_t scan_gen_smem(int M4) { return (size_t)GPP * M4 * 4 + (size_t)GW * GPP * LCW * 8; }

// The CTA's warps split the references (warp w takes the tiles of 32
// references w, w + GW, ...) and keep a candidate list per point; the lists
// are then merged against the best cosine over all warps.
__global__ void __launch_bounds__(GW * 32) k_assoc_scan_gen(RunView v)
{
    extern __shared__ __align__(16) float sgen[];
    __shared__ float s_best[GW][GPP];
    __shared__ int s_nl[GW][GPP];
    __shared__ int s_ovf[GW][GPP];
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int nT = c->nT, m = v.m, M4 = v.M4, w = v.w;
    const int lane = lane_id(), warp = threadIdx.x >> 5, tid = threadIdx.x;
    float* Us = sgen;                                                // GPP x M4
    int* lists = reinterpret_cast<int*>(sgen + (size_t)GPP * M4);   // GW x GPP x (LCW ints, LCW floats)
    const float band = 2.0f * (float)(m + 4) * 5.9604644775390625e-08f + 1e-12f;
    for (int g0 = blockIdx.x * GPP; g0 < nT; g0 += gridDim.x * GPP) {  // CTA-uniform
        __syncthreads();  // the previous group is merged
        for (int e = tid; e < GPP * M4; e += GW * 32) {
            const int p = e / M4;
            Us[e] = g0 + p < nT ? v.uhat[(size_t)g0 * M4 + e] : 0.0f;
        }
        __syncthreads();
        float best[GPP];
        int nl[GPP];
        bool ovf[GPP], live[GPP];
#pragma unroll
        for (int p = 0; p < GPP; ++p) {
            best[p] = -4.0f;
            nl[p] = 0;
            ovf[p] = false;
            live[p] = g0 + p < nT && v.fnorm[g0 + p] != 0.0;  // |f'| = 0: every distance is 0
        }
        for (int r0 = warp * 32; r0 < w; r0 += GW * 32) {
            const int j = r0 + lane;
            const float4* z4 = reinterpret_cast<const float4*>(v.Zh + (size_t)(j < w ? j : w - 1) * M4);
            float acc[GPP];
#pragma unroll
            for (int p = 0; p < GPP; ++p) acc[p] = 0.0f;
#pragma unroll 8
            for (int k4 = 0; k4 < M4 / 4; ++k4) {
                const float4 z = __ldg(z4 + k4);
#pragma unroll
                for (int p = 0; p < GPP; ++p) {
                    const float4 u = reinterpret_cast<const float4*>(Us + (size_t)p * M4)[k4];
                    acc[p] = fmaf(u.x, z.x, acc[p]);
                    acc[p] = fmaf(u.y, z.y, acc[p]);
                    acc[p] = fmaf(u.z, z.z, acc[p]);
                    acc[p] = fmaf(u.w, z.w, acc[p]);
                }
            }
#pragma unroll
            for (int p = 0; p < GPP; ++p)
                if (live[p]) {
                    int* lj = lists + (size_t)(warp * GPP + p) * 2 * LCW;
                    band_take(acc[p], j < w ? j : -1, band, best[p], nl[p], ovf[p], lj,
                              reinterpret_cast<float*>(lj + LCW), LCW);
                }
        }
        if (lane == 0)
#pragma unroll
            for (int p = 0; p < GPP; ++p) {
                s_best[warp][p] = best[p];
                s_nl[warp][p] = nl[p];
                s_ovf[warp][p] = ovf[p] ? 1 : 0;
            }
        __syncthreads();
        // merge: warp p takes point p
        const int p = warp;
        const int pt = g0 + p;
        if (p >= GPP || pt >= nT) continue;
        if (!live[p]) {
            if (lane == 0) v.arun[pt] = make_int2(0, 0);
            continue;
        }
        float gb = s_best[0][p];
        bool govf = false;
        for (int q = 0; q < GW; ++q) {
            gb = fmaxf(gb, s_best[q][p]);
            govf = govf || s_ovf[q][p];
        }
        int cnt = 0;
        for (int q = 0; q < GW; ++q) {
            const int* lj = lists + (size_t)(q * GPP + p) * 2 * LCW;
            const float* lq = reinterpret_cast<const float*>(lj + LCW);
            const int n = s_nl[q][p];
            for (int e0 = 0; e0 < n; e0 += 32) {
                const int e = e0 + lane;
                cnt += __popc(__ballot_sync(0xffffffffu, e < n && lq[e] >= gb - band));
            }
        }
        int start = 0;
        if (lane == 0 && !govf) start = atomicAdd(&c->ncand, cnt);
        start = __shfl_sync(0xffffffffu, start, 0);
        if (govf || start + cnt > v.cand_cap) {
            if (lane == 0) {
                v.arun[pt] = make_int2(-1, 0);
                v.slow[atomicAdd(&c->nslow, 1)] = pt;
            }
            continue;
        }
        int off = 0;
        for (int q = 0; q < GW; ++q) {
            const int* lj = lists + (size_t)(q * GPP + p) * 2 * LCW;
            const float* lq = reinterpret_cast<const float*>(lj + LCW);
            const int n = s_nl[q][p];
            for (int e0 = 0; e0 < n; e0 += 32) {
                const int e = e0 + lane;
                const bool k2 = e < n && lq[e] >= gb - band;
                const unsigned b2 = __ballot_sync(0xffffffffu, k2);
                if (k2) v.cand[start + off + __popc(b2 & ((1u << lane) - 1u))] = make_int2(pt, lj[e]);
                off += __popc(b2);
            }
        }
        if (lane == 0) v.arun[pt] = make_int2(start, cnt);
    }
}

// a thread per candidate (the FP64 pipe of a warp instruction serves 32
// candidates): its FP64 distance, the same left-to-right evaluation
__global__ void __launch_bounds__(32) k_assoc_cand_dist(RunView v)
{
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int e = blockIdx.x * 32 + threadIdx.x;
    // ncand counts reservations, also those that did not fit (their points
    // went to the slow path): only the first cand_cap slots exist
    if (e >= min(c->ncand, v.cand_cap)) return;
    const int2 pj = v.cand[e];
    const double nf = v.fnorm[pj.x];
    v.cdist[e] = perp_dist_mem(v.fprime + (size_t)pj.x * v.m, nf, v.Zd + (size_t)pj.y * v.m, v.nz[pj.y], v.m);
}

// a thread per point: lexicographic (d, j) minimum over its candidates
__global__ void __launch_bounds__(256) k_assoc_final_gen(RunView v)
{
    Ctrl* c = v.ctrl;
    if (skip_niche(c)) return;
    const int pt = blockIdx.x * 256 + threadIdx.x;
    if (pt >= c->nT) return;
    const int2 run = v.arun[pt];
    if (run.x < 0) return;  // slow path
    double bd = 0.0;
    int bj = 0;
    if (v.fnorm[pt] != 0.0) {
        bd = CUDART_INF;
        bj = 0x7fffffff;
        for (int e = run.x; e < run.x + run.y; ++e) {
            const double d = v.cdist[e];
            const int j = v.cand[e].y;
            if (lex_less(d, j, bd, bj)) {
                bd = d;
                bj = j;
            }
        }
    }
    if (v.debug_recheck_all) {
        v.dist[v.Tlist[pt]] = bd;
        v.pi[v.Tlist[pt]] = bj;
        v.slow[atomicAdd(&c->nslow, 1)] = pt;
        return;
    }
    write_assoc(v, c, v.Tlist[pt], v.rank2[v.Tlist[pt]], bj, bd);
}

template <int M>
cudaError_t launch_m(const RunView& v, cudaStream_t s, int num_sms)
{
    constexpr int KP = kp_of<M>();
    k_assoc_mma<KP><<<v.assoc_grid, MT, mma_smem<KP>(), s>>>(v);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_assoc_final<M><<<(v.n2 + FB - 1) / FB, FB, 0, s>>>(v);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_assoc_slow<M><<<num_sms, AB, 0, s>>>(v);
    return cudaGetLastError();
}

}  // namespace

int assoc_grid(int num_sms) { return num_sms > 0 ? num_sms : 1; }

size_t assoc_entries(int n2, int num_sms)
{
    // items = ntile x S <= ntile x 2 ceil(grid / ntile) <= 2 (grid + ntile)
    // for every nT <= n2
    const size_t ntile = ((size_t)n2 + TP - 1) / TP;
    return 2 * ((size_t)assoc_grid(num_sms) + ntile) * TP;
}

size_t assoc_rows_bytes(int m, int rows)
{
    const size_t kp = 3 * m <= 16 ? 16 : 32;
    return ((size_t)rows + TP - 1) / TP * TP * kp * 2;
}

namespace {

// The directions' FP16 rows [zh, zl, zh] in chunks of 128 as k_assoc_mma
// reads them, from their w x M4 unit vectors in block order; a thread per
// row.  Rows past w are -1 in every h: their cosines with unit vectors of
// non-negative components are below -0.9.
__global__ void __launch_bounds__(256) k_assoc_pack(int m, int M4, int w, int rows, const float* z, unsigned char* out)
{
    const int j = blockIdx.x * 256 + threadIdx.x;
    if (j >= rows) return;
    const int KP = 3 * m <= 16 ? 16 : 32;
    __half* row = reinterpret_cast<__half*>(out + (size_t)(j / CHUNK) * (CHUNK * KP * 2) + (j % CHUNK) * 16);
    auto put = [&](int e, __half h) { row[(e / 8) * CHUNK * 8 + e % 8] = h; };
    for (int q = 0; q < m; ++q) {
        const float x = j < w ? z[(size_t)j * M4 + q] : -1.0f;
        const __half h = __float2half_rn(x);
        put(q, h);
        put(2 * m + q, h);
        put(m + q, __float2half_rn(x - __half2float(h)));
    }
    for (int e = 3 * m; e < KP; ++e) put(e, __float2half_rn(0.0f));
}

}  // namespace

cudaError_t launch_assoc_pack(int m, int M4, int w, const float* z, unsigned char* out, cudaStream_t s)
{
    const int rows = (w + TP - 1) / TP * TP;  // what assoc_rows_bytes holds
    k_assoc_pack<<<(rows + 255) / 256, 256, 0, s>>>(m, M4, w, rows, z, out);
    return cudaGetLastError();
}

cudaError_t launch_assoc_prep(const RunView& v, cudaStream_t s)
{
    const int g = (v.n2 + PB - 1) / PB;
    switch (v.m) {
    case 2: k_assoc_prep<2><<<g, PB, 0, s>>>(v); break;
    case 3: k_assoc_prep<3><<<g, PB, 0, s>>>(v); break;
    case 4: k_assoc_prep<4><<<g, PB, 0, s>>>(v); break;
    case 5: k_assoc_prep<5><<<g, PB, 0, s>>>(v); break;
    case 6: k_assoc_prep<6><<<g, PB, 0, s>>>(v); break;
    case 7: k_assoc_prep<7><<<g, PB, 0, s>>>(v); break;
    case 8: k_assoc_prep<8><<<g, PB, 0, s>>>(v); break;
    case 9: k_assoc_prep<9><<<g, PB, 0, s>>>(v); break;
    case 10: k_assoc_prep<10><<<g, PB, 0, s>>>(v); break;
    default:
        if (v.m < 2 || v.m > NSGA3_MAX_M) return cudaErrorInvalidValue;
    {
        k_assoc_prep_elem<<<(unsigned)(((long long)v.n2 * v.m + 255) / 256), 256, 0, s>>>(v);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        k_assoc_prep_norm<<<(v.n2 + 31) / 32, 32, 0, s>>>(v);
        break;
    }
    }
    return cudaGetLastError();
}

cudaError_t launch_assoc_scan(const RunView& v, int num_sms, cudaStream_t s)
{
    switch (v.m) {
    case 2: return launch_m<2>(v, s, num_sms);
    case 3: return launch_m<3>(v, s, num_sms);
    case 4: return launch_m<4>(v, s, num_sms);
    case 5: return launch_m<5>(v, s, num_sms);
    case 6: return launch_m<6>(v, s, num_sms);
    case 7: return launch_m<7>(v, s, num_sms);
    case 8: return launch_m<8>(v, s, num_sms);
    case 9: return launch_m<9>(v, s, num_sms);
    case 10: return launch_m<10>(v, s, num_sms);
    default: break;
    }
    if (v.m < 2 || v.m > NSGA3_MAX_M) return cudaErrorInvalidValue;
    int blocks = (v.n2 + GPP - 1) / GPP;
    if (blocks > num_sms * 8) blocks = num_sms * 8;
    k_assoc_scan_gen<<<blocks, GW * 32, scan_gen_smem(v.M4), s>>>(v);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // one warp per CTA: the few candidates of a selection spread over every SM
    k_assoc_cand_dist<<<(v.cand_cap + 31) / 32, 32, 0, s>>>(v);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_assoc_final_gen<<<(v.n2 + 255) / 256, 256, 0, s>>>(v);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_assoc_slow<0><<<num_sms, AB, 0, s>>>(v);
    return cudaGetLastError();
}

cudaError_t assoc_init_attributes()
{
    cudaError_t e = cudaFuncSetAttribute(k_assoc_mma<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mma_smem<16>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_assoc_mma<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mma_smem<32>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_assoc_scan_gen, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)scan_gen_smem(NSGA3_MAX_M));
    return e;
}
