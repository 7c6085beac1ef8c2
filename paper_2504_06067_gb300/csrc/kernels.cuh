// kernels.cuh -- launch wrappers for the NSGA-III kernels (host side).
// Every wrapper enqueues on `s` and returns the launch error; grids are
// derived from the run's fixed sizes, so the same launches can be captured
// into a CUDA graph once and replayed every generation.
#pragma once
#include "common.cuh"

// setup (Sec. II-C reference points; init population)
cudaError_t launch_refdirs(const RunView& v, int p1, int p2, double tau, double* Zd, double* nz,
                           float* Zh, cudaStream_t s);
cudaError_t launch_init(const RunView& v, cudaStream_t s);
cudaError_t launch_nan_pad(const RunView& v, cudaStream_t s);

// variation + objective (Alg. 1, crossover and mutation; Sec. III-A)
cudaError_t launch_vary_eval(const RunView& v, cudaStream_t s);

// one selection or generation in one cluster (k_small.cu); mode 0: objectives
// F in, ranks and indices out; 1: a whole generation; 2: a generation whose
// variation has run
#define SMALL_N2 2048  // merged individuals at most
#define SMALL_W 2048   // reference directions at most
cudaError_t launch_small(const RunView& v, int mode, const float* F, int32_t* ranks, int32_t* sel, cudaStream_t s);
cudaError_t small_init_attributes();
// whether the device has room for that cluster (after small_init_attributes),
// and for the one of the elimination (m > 32; after norm_init_attributes)
bool small_fits(int m, int n2, int w);
bool solve_fits(int m);

// selection (Alg. 1 sort / Alg. 2)
// 0-1 knapsack workload (k_knapsack.cu): bits + repair + objectives
cudaError_t launch_kp_init(const RunView& v, cudaStream_t s);
cudaError_t launch_kp_vary_eval(const RunView& v, cudaStream_t s);
// reset of the selection's buffers, level thresholds (m <= 10), finite check
cudaError_t launch_front(const RunView& v, int num_sms, bool check, cudaStream_t s);
// the device-wait self-test (nsga3_wait_probe)
cudaError_t launch_wait_probe(const RunView& v, cudaStream_t s);
cudaError_t launch_check_finite(const RunView& v, cudaStream_t s);
cudaError_t launch_sort(const RunView& v, int num_sms, cudaStream_t s);
// the first front (v.domw set; nothing otherwise); the view of the points it
// leaves (v itself when there is no first front)
cudaError_t launch_first_front(const RunView& v, cudaStream_t s);
RunView rest_view(const RunView& v);
cudaError_t launch_dominance(const RunView& v, cudaStream_t s);
cudaError_t dom_init_attributes();
// every peel pass in one cooperative launch
cudaError_t launch_peel(const RunView& v, int num_sms, cudaStream_t s);
cudaError_t peel_init_attributes();
cudaError_t launch_norm_ideal(const RunView& v, cudaStream_t s);
// extreme points and intercepts: one launch (m <= 10); above, the ideal
// point, entry keys, per-axis blocks and their reduction (four launches),
// plus the elimination in a cluster for m > 32
cudaError_t launch_norm_extreme(const RunView& v, int num_sms, cudaStream_t s);
cudaError_t norm_init_attributes();
cudaError_t launch_assoc_prep(const RunView& v, cudaStream_t s);
// candidate scan, FP64 distances and per-point argmin, FP64 slow path (three
// launches; four for m > 10, where the distances are a kernel of their own);
// the unit vectors are launch_assoc_prep (one launch, two for m > 10)
cudaError_t launch_assoc_scan(const RunView& v, int num_sms, cudaStream_t s);
// m <= 10: the tensor-core scan's grid for a device of num_sms SMs, the int4
// entries it writes for at most n2 points, the bytes of `rows` FP16 operand
// rows, and the directions' rows
int assoc_grid(int num_sms);
size_t assoc_entries(int n2, int num_sms);
size_t assoc_rows_bytes(int m, int rows);
cudaError_t launch_assoc_pack(int m, int M4, int w, const float* z, unsigned char* out, cudaStream_t s);
cudaError_t assoc_init_attributes();
cudaError_t launch_level(const RunView& v, cudaStream_t s);
cudaError_t launch_bucket(const RunView& v, cudaStream_t s);
cudaError_t launch_pick(const RunView& v, cudaStream_t s);
// self-test of the block-wide selection of the smallest keys (one CTA)
cudaError_t launch_select_probe(const unsigned long long* keys, int n, int need, uint32_t* marks,
                                unsigned* paths, cudaStream_t s);
// masks and counts of the selected individuals, then their indices (a
// selection) or the next population and the generation counter
cudaError_t launch_mark(const RunView& v, cudaStream_t s);
cudaError_t launch_select_out(const RunView& v, cudaStream_t s);
cudaError_t launch_gather(const RunView& v, cudaStream_t s);
// rows of X to dst (row r of dst = row idx[r] of X) and up to two plain copies
// (n = 0: none) in the same launch; plain copies alone; rows back, likewise
struct PlainCopy {
    const uint32_t* src;
    uint32_t* dst;
    int n;  // words
};
cudaError_t launch_rows_out(const RunView& v, const int32_t* idx, float* dst, PlainCopy a, PlainCopy b, cudaStream_t s);
cudaError_t launch_copies(PlainCopy a, PlainCopy b, cudaStream_t s);
cudaError_t launch_rows_in(const RunView& v, const float* src, PlainCopy a, PlainCopy b, cudaStream_t s);
cudaError_t launch_slots_init(const RunView& v, cudaStream_t s);

// issue-rate probe of the dominance test's FADD / LOP3 mix (k_probe.cu)
double issue_probe_instructions(int blocks, int iters);
cudaError_t launch_issue_probe(const float* in, int blocks, int iters, uint32_t* sink, cudaStream_t s);

// one-time attribute setup (dynamic shared memory opt-in)
cudaError_t kernels_init_attributes();
