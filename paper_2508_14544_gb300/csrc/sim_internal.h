// Internal declarations shared by the C ABI (sim_api.cpp) and the CUDA kernels (sim_kernels.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <climits>

namespace simgb {

// Internal per-instance status: the active set outgrew the per-instance capacity of the launch;
// the host re-runs such instances with a larger, global-memory workspace.
constexpr int32_t kStatusCapacity = -100;
constexpr int64_t kMaxM = int64_t(1) << 26;
// Steps are int32: an instance stops with SIM_E_STEPCAP before a step passes kMaxStep, which leaves
// room for a projected length (<= M <= 2^26) on top of any step.
constexpr int32_t kMaxStep = INT32_MAX - (int32_t(1) << 27);
// A_ell queue keys are 2 a (arrival) and 2 t + 1 (promotion at step t): steps stay below 2^30.
constexpr int32_t kAellMaxStep = (int32_t(1) << 30) - 1;

// One waiting request as the queue stores it; queues are ordered by (key, idx).
struct QEnt {
    int32_t key;  // sort key: u (A_max), o (H-SF), current lower bound (A_min), permutation rank
                  // (A_r), queue position 2 a / 2 t + 1 (A_ell)
    int32_t idx;  // request index within its instance
    int32_t s;    // prompt size
    int32_t o;    // true output length
};

// Per-instance constants produced by the staging kernel.
struct InstInfo {
    int64_t base;     // offset of the instance's first request
    int64_t sum_a;    // sum of arrival steps (TEL = sum of completions - sum_a)
    int64_t cap;      // step cap
    int32_t n;        // number of requests
    int32_t status;   // 0 or a sim_status from validation
};

struct DevResult {
    int64_t total_latency, makespan, peak_memory, evictions, steps, request_steps;
    int32_t status, pad;
};

struct StageParams {
    int policy;
    int64_t M;
    int32_t n_inst;
    int32_t n_max;             // largest instance (sizes the staging kernel's shared memory; 0: unknown)
    int64_t max_total;         // capacity of rec / rec_a: an instance reaching past it is rejected (INVAL)
    int32_t max_n;             // requests per instance above this are rejected (INVAL)
    int64_t step_cap;          // 0: default 64 * (n + sum o)
    const int64_t *off;        // n_inst + 1
    const int32_t *a, *s, *l, *u, *o;  // raw copies, n_total each
    const int32_t *rank;       // A_r: permutation rank per request (n_total), else unused
    QEnt *rec;                 // out: per instance, sorted by (a, key, idx)
    int2 *lu;                  // out (A_ell only, else null): (l, u) of request idx at base + idx
    int32_t *rec_a;            // out: arrival step of rec[i]
    InstInfo *info;            // out: n_inst
};

struct RunParams {
    int64_t M;
    int32_t n_work;            // instances to run in this launch
    const int32_t *n_work_dev; // optional: their number on the device (the redo count of an earlier launch)
    const int32_t *work;       // instance ids (n_work)
    int32_t *counter;          // work-queue cursor (zeroed before a launch of more instances than warps)
    int32_t *redo;             // optional: ids of the instances that outgrew the capacity are listed here
    int32_t *redo_count;       // their number (zeroed before launch)
    const QEnt *rec;
    const int32_t *rec_a;
    const InstInfo *info;
    DevResult *res;
    int64_t *completion;       // optional, n_total
    const int2 *lu;            // A_ell: (l, u) per request (staged), else null
    const uint64_t *tie_seed;  // A_min: seed of the random eviction ties per instance, or null (0 for all)
    int64_t *work_count;       // optional, 4 per instance: S2 adds, S3 compare-exchanges, S5 endpoint
                               // evaluations of the per-step method, global bytes moved by the queue
    int64_t *batch_time;       // optional, 6 per instance: the batch-time sums X0..X3, F2, F3
    // workspace
    int32_t ca;                // active-set capacity per instance (a multiple of kCaUnit)
    int32_t dcap;              // delta-queue capacity per warp slot (at most kDcap)
    int32_t use_smem;          // 1: active set + delta queue in shared memory; 0: global workspace
    int32_t wide;              // 1: the copy with more registers a thread and at most 12 warps per SM
    int32_t debug;             // 1: check the simulation state's invariants every iteration (global kernel)
    int32_t evict_index;       // 1: A_min eviction ties by request index instead of the random tie key
    unsigned char *gws;        // global workspace base (use_smem == 0)
    int64_t gws_stride;        // bytes per warp slot
    QEnt *mainbuf;             // ping-pong main-queue buffers, 2 * main_cap per warp slot
    int64_t main_cap;          // 0: two buffers of n entries per instance, at twice its first request
};

constexpr int kCaUnit = 128;       // active-set slots are passed over and allotted in pages of this many
// Slots that no instance of n requests fills (one that fills the slots stops with kStatusCapacity).
__host__ __device__ constexpr int ca_above(int64_t n) { return int(n / kCaUnit + 1) * kCaUnit; }

constexpr int kDenseCa = 384;      // active-set slots per warp of the dense configuration
constexpr int kDenseWarps = 4;     // warps per block of the dense configuration
constexpr int kSmemCaDefault = 512;  // active-set slots per warp in shared memory by default
constexpr int kDcap = 256;         // largest delta-queue capacity (multiple of 32)
constexpr int kMc = 64;            // cached entries of the main queue (two per lane)

// Delta-queue entries used for an instance of n requests.
__host__ __device__ constexpr int delta_cap(int64_t n) { return n <= 1024 ? 64 : (n <= 4096 ? 128 : kDcap); }

// Workspace of one simulating warp, in this order: ca slots of {E, W}, B, F (16 bytes) and {P, I} (8), the
// head cache of the main queue (whose space also holds the positions of a merge), the A_min estimate per
// slot (4) and the delta queue.
constexpr size_t kWsCacheBytes = size_t(kMc) * sizeof(QEnt);
static_assert(size_t(kDcap) * 4 <= kWsCacheBytes, "merge positions");
__host__ __device__ constexpr size_t ws_bytes(int ca, int dcap) {
    return size_t(ca) * 28 + kWsCacheBytes + size_t(dcap) * sizeof(QEnt);
}

cudaError_t launch_stage(const StageParams &p, cudaStream_t st, int *launches);
// Blocks of the kernel that p selects that one SM holds at a time; raises its shared-memory limit.
cudaError_t run_blocks_per_sm(int policy, const RunParams &p, int warps_per_block, size_t smem_bytes, int *blocks);
cudaError_t launch_run(int policy, const RunParams &p, int blocks, int warps_per_block, size_t smem_bytes,
                       cudaStream_t st);
cudaError_t launch_ratio(const DevResult *pol, const DevResult *ref, double *out, int32_t n, cudaStream_t st);
cudaError_t launch_batch_time(const int64_t *sums, const DevResult *res, const double *coef, double *out, int32_t n,
                              cudaStream_t st);
constexpr int kLemmaMaxLen = 8192;  // lengths of a histogram
cudaError_t launch_lemma(int32_t n_hist, int32_t len, int32_t l, double s, const double *x, double *out,
                         cudaStream_t st);
// Launch shape of the spectral-radius kernel for n_u values of which the largest is u_max.
struct RhoPlan {
    int threads;      // per block
    int cluster;      // blocks per value
    size_t smem;      // bytes of shared memory per block, 0 when the arrays live in scratch
    int64_t scratch;  // doubles of global scratch per value (0: none, and scratch must be null)
};
cudaError_t rho_plan(int32_t n_u, int32_t u_max, RhoPlan *plan);
cudaError_t launch_rho(const RhoPlan &plan, int32_t n_u, const int32_t *us, double *out, double *scratch,
                       int32_t max_iter, cudaStream_t st);

}  // namespace simgb
