// Staging and result kernels of the batched scheduler simulator (sm_103a).
//
//   k_stage  - per instance (one CTA): validate the requests against the Section 2 model
//              (1 <= l <= o <= u, s >= 1, a >= 0, s + o <= M; s + u <= M under A_max), compute the
//              constants the simulation needs (sum of arrivals for TEL, the step cap), and sort
//              the requests by (arrival step, policy key, index) so that every arrival batch is
//              already in the order of the waiting set R_t (key u for Algorithm malb, l for
//              Algorithms milb / milbrevise, o for Algorithm off, the given permutation rank for
//              Algorithm random, and the FIFO position 2 a for Algorithm promote_l, which also
//              gets its (l, u) table).
//   k_stage_large - the same for instances of more than kStageSmemN requests, one CTA of 1024 threads
//              each.  When the requests come in arrival order in groups of at most 32 per step, every
//              request finds its place by comparing itself with its group; otherwise an LSD radix sort in
//              global memory on 8-bit digits.
//   k_ratio  - per instance TEL(pi) / TEL(H-SF) in IEEE double (Definition cr).
//   k_batch_time - per instance total latency and makespan in time units under a linear
//              batch-time model (Section 6), from the integer sums the simulation recorded.
#include <climits>
#include <cstdint>

#include "sim_internal.h"

namespace simgb {

namespace {

constexpr unsigned FULL = 0xffffffffu;
enum { P_AMAX = 0, P_AMIN = 1, P_HSF = 2, P_AR = 3, P_AELL = 4 };
enum { ST_OK = 0, ST_INVAL = -1, ST_INFEASIBLE = -2 };

struct BtCoef {
    double k[5];
};

// Policy key of the request at g (validity is checked by stage_check).
__device__ __forceinline__ int stage_key(const StageParams &S, int64_t g) {
    switch (S.policy) {
        case P_AMAX: return S.u[g];
        case P_HSF: return S.o[g];
        case P_AR: return S.rank[g];
        case P_AELL: return 2 * min(S.a[g], kAellMaxStep);
        default: return S.l[g];
    }
}

// Validates the request at g, fills A_ell's (l, u) table and adds to the instance's sums.
struct StageSums {
    int64_t bad_inval, bad_inf, sum_a, sum_o;
    int kmax, amax;
};

__device__ __forceinline__ void stage_check(const StageParams &S, int64_t g, int a, int s, int o, int key, StageSums &z) {
    const int l = S.l[g], u = S.u[g];
    if (s < 1 || a < 0 || l < 1 || l > o || o > u) z.bad_inval = 1;
    if (int64_t(s) + o > S.M) z.bad_inf = 1;
    if ((S.policy == P_AMAX || S.policy == P_AELL) && int64_t(s) + u > S.M) z.bad_inf = 1;
    if (S.policy == P_AR && key < 0) z.bad_inval = 1;
    if (S.policy == P_AELL) {
        if (a > kAellMaxStep) z.bad_inval = 1;
        S.lu[g] = make_int2(l, u);
    }
    z.sum_a += a;
    z.sum_o += o;
    z.kmax = max(z.kmax, key);
    z.amax = max(z.amax, a);
}

template <typename T>
__device__ T block_reduce(T v, T *sh, bool is_max) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const T o = __shfl_xor_sync(FULL, v, d);
        v = is_max ? (o > v ? o : v) : v + o;
    }
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    T acc = sh[0];
    for (int i = 1; i < nw; ++i) acc = is_max ? (sh[i] > acc ? sh[i] : acc) : acc + sh[i];
    return acc;
}

// Block-wide sums of z (kmax and amax are replaced by the block's), the instance's constants and status.
__device__ int stage_finish(const StageParams &S, int inst, int64_t base, int n, StageSums &z, int64_t *sh64) {
    const int64_t bad_inval = block_reduce<int64_t>(z.bad_inval, sh64, true);
    const int64_t bad_inf = block_reduce<int64_t>(z.bad_inf, sh64, true);
    const int64_t sum_a = block_reduce<int64_t>(z.sum_a, sh64, false);
    const int64_t sum_o = block_reduce<int64_t>(z.sum_o, sh64, false);
    z.kmax = int(block_reduce<int64_t>(z.kmax, sh64, true));
    z.amax = int(block_reduce<int64_t>(z.amax, sh64, true));
    const int status = bad_inval ? ST_INVAL : bad_inf ? ST_INFEASIBLE : ST_OK;
    if (threadIdx.x == 0) {
        InstInfo in;
        in.base = base;
        in.n = n;
        in.status = status;
        in.sum_a = sum_a;
        in.cap = S.step_cap > 0 ? S.step_cap : 64 * (int64_t(n) + sum_o);
        S.info[inst] = in;
    }
    __syncthreads();
    return status;
}

// Instances of up to this many requests are sorted in shared memory: per request its key, arrival,
// prompt and true length and two index buffers (24 bytes), plus the radix counters.
constexpr int kStageSmemN = 2048;
constexpr int kStageSmemBytesPerReq = 24;
constexpr int kStageSmemIpt = kStageSmemN / 256;  // elements per thread of a radix pass
constexpr size_t kStageCntBytes = size_t(16) * kStageSmemIpt * 8 * sizeof(uint16_t);

// Instances held in shared memory are sorted by an LSD radix sort of request indices, 4-bit digits
// of the policy key and then of the arrival step, each pass stable, so the order is (a, key, idx)
// (both are >= 0 in a valid instance).  A pass ranks element e = r * 256 + thread (iteration r):
// within a warp and iteration, __match_any_sync groups the lanes with equal digits and a lane's
// rank in its group is the number of group lanes below it; the groups' sizes go to counters in
// (digit, iteration, warp) order, whose exclusive prefix sums are the groups' first output
// positions.  Elements are thereby placed in (digit, e) order: stable.
constexpr int kRadixBits = 4;
constexpr int kRadixBins = 1 << kRadixBits;
constexpr int kStageThreads = 256;
constexpr int kStageWarps = kStageThreads / 32;

template <int IPT>
__device__ __forceinline__ void radix_pass(const int32_t *keyof, const int32_t *in, int32_t *out, uint16_t *cnt,
                                           int *wsum, int n, int shift) {
    constexpr int kCnt = kRadixBins * IPT * kStageWarps;  // a multiple of 4 * kStageThreads / 4
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int f = t; f < kCnt; f += kStageThreads) cnt[f] = 0;
    __syncthreads();
    int dg[IPT], rk[IPT], ix[IPT];
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const int e = r * kStageThreads + t;
        const bool v = e < n;
        ix[r] = v ? in[e] : 0;
        dg[r] = v ? ((keyof[ix[r]] >> shift) & (kRadixBins - 1)) : kRadixBins;  // past the end: a group of its own
        const unsigned peers = __match_any_sync(FULL, dg[r]);
        rk[r] = __popc(peers & lt);
        if (v && rk[r] == 0) cnt[(dg[r] * IPT + r) * kStageWarps + w] = uint16_t(__popc(peers));
    }
    __syncthreads();
    // exclusive prefix sums of the counters, kCnt / kStageThreads consecutive ones per thread
    constexpr int kPer = kCnt / kStageThreads;
    int c[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        c[i] = cnt[kPer * t + i];
        sum += c[i];
    }
    int x = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(FULL, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    int run = x - sum;
    for (int i = 0; i < w; ++i) run += wsum[i];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        cnt[kPer * t + i] = uint16_t(run);
        run += c[i];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const int e = r * kStageThreads + t;
        if (e < n) out[cnt[(dg[r] * IPT + r) * kStageWarps + w] + rk[r]] = ix[r];
    }
    __syncthreads();
}

// Sorts the indices 0..n-1 held in i0 (scratch i1) by (ka, kk, index); returns the buffer that
// holds the result.  kmax, amax: the largest key and arrival step (>= 0).
__device__ int32_t *radix_sort_idx(const int32_t *kk, const int32_t *ka, int32_t *i0, int32_t *i1, uint16_t *cnt,
                                   int *wsum, int n, int kmax, int amax) {
    int32_t *in = i0, *out = i1;
    const int kbits = kmax > 0 ? 32 - __clz(kmax) : 0;
    const int abits = amax > 0 ? 32 - __clz(amax) : 0;
    for (int sh = 0; sh < kbits; sh += kRadixBits) {
        radix_pass<kStageSmemIpt>(kk, in, out, cnt, wsum, n, sh);
        int32_t *tmp = in;
        in = out;
        out = tmp;
    }
    for (int sh = 0; sh < abits; sh += kRadixBits) {
        radix_pass<kStageSmemIpt>(ka, in, out, cnt, wsum, n, sh);
        int32_t *tmp = in;
        in = out;
        out = tmp;
    }
    return in;
}

// An instance that is larger than the n_max the launch was made for: the offsets were read again, by the
// replay of a captured call, after the caller changed them.  Every request counts those before it.
__device__ __noinline__ void stage_by_counting(const StageParams &S, int inst, int64_t base, int n, int64_t *sh64) {
    StageSums z = {0, 0, 0, 0, 0, 0};
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int64_t g = base + j;
        stage_check(S, g, S.a[g], S.s[g], S.o[g], stage_key(S, g), z);
    }
    if (stage_finish(S, inst, base, n, z, sh64) != ST_OK) return;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int64_t g = base + j;
        const int a = S.a[g];
        QEnt e;
        e.key = stage_key(S, g);
        e.idx = j;
        e.s = S.s[g];
        e.o = S.o[g];
        int place = 0;
        for (int k = 0; k < n; ++k) {
            const int ak = S.a[base + k], kk = stage_key(S, base + k);
            place += ak < a || (ak == a && (kk < e.key || (kk == e.key && k < j))) ? 1 : 0;
        }
        S.rec[base + place] = e;
        S.rec_a[base + place] = a;
    }
}

__global__ void __launch_bounds__(kStageThreads) k_stage(StageParams S, int np) {
    __shared__ int64_t sh64[32];
    __shared__ int wsum[kStageWarps];
    extern __shared__ __align__(16) unsigned char stage_smem[];
    const int inst = blockIdx.x;
    const int64_t base = S.off[inst];
    const int64_t n64 = S.off[inst + 1] - base;
    // offsets that reach outside the staged buffers (or above the per-instance limit) reject the
    // instance before anything is written: it is staged as empty with status INVAL
    const bool oob = base < 0 || n64 < 0 || n64 > S.max_n || base + n64 > S.max_total;
    const int n = oob ? 0 : int(n64);
    if (n > np) {
        if (S.n_max <= np) stage_by_counting(S, inst, base, n, sh64);
        return;  // otherwise k_stage_large follows
    }
    int32_t *kk = reinterpret_cast<int32_t *>(stage_smem);
    int32_t *ka = kk + np;
    int32_t *ss = ka + np;
    int32_t *so = ss + np;
    int32_t *i0 = so + np;
    int32_t *i1 = i0 + np;
    uint16_t *cnt = reinterpret_cast<uint16_t *>(i1 + np);
    StageSums z = {oob ? 1 : 0, 0, 0, 0, 0, 0};
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int64_t g = base + j;
        const int a = S.a[g], s = S.s[g], o = S.o[g], key = stage_key(S, g);
        stage_check(S, g, a, s, o, key, z);
        kk[j] = key;
        ka[j] = a;
        ss[j] = s;
        so[j] = o;
        i0[j] = j;
    }
    const int status = stage_finish(S, inst, oob ? 0 : base, n, z, sh64);
    const int32_t *ord = i0;
    if (status == ST_OK && n > 1) ord = radix_sort_idx(kk, ka, i0, i1, cnt, wsum, n, z.kmax, z.amax);
    // write the (sorted, or for a rejected instance unsorted) records out
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int idx = ord[j];
        QEnt e;
        e.key = kk[idx];
        e.idx = idx;
        e.s = ss[idx];
        e.o = so[idx];
        S.rec[base + j] = e;
        S.rec_a[base + j] = ka[idx];
    }
}

// ---- instances of more than kStageSmemN requests ----------------------------------------------

constexpr int kLargeThreads = 1024;
constexpr int kLargeWarps = kLargeThreads / 32;
constexpr int kLargeGroup = 32;  // longest run of equal arrival steps that is ranked directly

// One stable pass of the LSD radix sort over n (value, index) pairs by the 8 bits of the value at
// `shift`, value replaced by a[index] first if a is given.  Per tile of 4096 pairs a warp takes 128
// consecutive ones: ranks within the warp by match_any and per-warp counters, whose sums over the
// warps (one thread per digit) on top of the digit's running position are the output positions.
__device__ void large_radix_pass(const int2 *in, int2 *out, const int32_t *a, int n, int shift, int32_t *cnt,
                                 int32_t *pos) {
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const unsigned lt = (1u << lane) - 1u;
    if (t < 256) pos[t] = 0;
    __syncthreads();
    for (int b = 0; b < n; b += kLargeThreads) {
        const int e = b + t;
        int d = 256;
        if (e < n) {
            const int2 x = in[e];
            d = ((a ? a[x.y] : x.x) >> shift) & 255;
        }
        const unsigned peers = __match_any_sync(FULL, d);
        if (d < 256 && (peers & lt) == 0) atomicAdd(&pos[d], __popc(peers));
    }
    __syncthreads();
    if (t < 32) {  // exclusive prefix sums of the 256 digit counts
        int v[8], sum = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            v[k] = pos[8 * t + k];
            sum += v[k];
        }
        int x = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(FULL, x, d);
            if (lane >= d) x += y;
        }
        int run = x - sum;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            pos[8 * t + k] = run;
            run += v[k];
        }
    }
    __syncthreads();
    for (int b = 0; b < n; b += 4 * kLargeThreads) {
        for (int k = t; k < 256 * kLargeWarps; k += kLargeThreads) cnt[k] = 0;
        __syncthreads();
        int2 x[4];
        int d[4], rk[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int e = b + w * 128 + r * 32 + lane;
            d[r] = 256;
            if (e < n) {
                x[r] = in[e];
                if (a) x[r].x = a[x[r].y];
                d[r] = (x[r].x >> shift) & 255;
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const unsigned peers = __match_any_sync(FULL, d[r]);
            int32_t *c = cnt + w * 256 + (d[r] & 255);
            rk[r] = d[r] < 256 ? *c + __popc(peers & lt) : 0;
            __syncwarp();
            if (d[r] < 256 && (peers & lt) == 0) *c += __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        if (t < 256) {
            int run = pos[t];
            for (int k = 0; k < kLargeWarps; ++k) {
                const int c = cnt[k * 256 + t];
                cnt[k * 256 + t] = run;
                run += c;
            }
            pos[t] = run;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (d[r] < 256) out[cnt[w * 256 + d[r]] + rk[r]] = x[r];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kLargeThreads) k_stage_large(StageParams S, int np) {
    __shared__ int64_t sh64[32];
    __shared__ int32_t pos[256];
    extern __shared__ __align__(16) unsigned char stage_smem[];
    const int inst = blockIdx.x;
    const int64_t base = S.off[inst];
    const int64_t n64 = S.off[inst + 1] - base;
    if (base < 0 || n64 <= np || n64 > S.max_n || base + n64 > S.max_total) return;  // k_stage
    const int n = int(n64);
    StageSums z = {0, 0, 0, 0, 0, 0};
    int far = 0;  // requests not in arrival order, or more than kLargeGroup of them in one step
    for (int j = threadIdx.x; j < n; j += kLargeThreads) {
        const int64_t g = base + j;
        const int a = S.a[g];
        stage_check(S, g, a, S.s[g], S.o[g], stage_key(S, g), z);
        if (j > 0 && S.a[g - 1] > a) far = 1;
        if (j >= kLargeGroup && S.a[g - kLargeGroup] >= a) far = 1;
    }
    const int status = stage_finish(S, inst, base, n, z, sh64);
    if (status != ST_OK) return;
    if (!__syncthreads_or(far)) {
        // place = the group's first place + the group's smaller (key, index)
        for (int j = threadIdx.x; j < n; j += kLargeThreads) {
            const int64_t g = base + j;
            QEnt e;
            e.key = stage_key(S, g);
            e.idx = j;
            e.s = S.s[g];
            e.o = S.o[g];
            const int a = S.a[g];
            int place = j;
            for (int k = j - 1; k >= 0 && S.a[base + k] == a; --k)
                if (stage_key(S, base + k) > e.key) --place;
            for (int k = j + 1; k < n && S.a[base + k] == a; ++k)
                if (stage_key(S, base + k) < e.key) ++place;
            S.rec[base + place] = e;
            S.rec_a[base + place] = a;
        }
        return;
    }
    // the pairs live in the instance's record space (two buffers of n pairs), the final order in rec_a
    int2 *in = reinterpret_cast<int2 *>(S.rec + base), *out = in + n;
    int32_t *cnt = reinterpret_cast<int32_t *>(stage_smem);
    for (int j = threadIdx.x; j < n; j += kLargeThreads) in[j] = make_int2(stage_key(S, base + j), j);
    __syncthreads();
    const int kbits = z.kmax > 0 ? 32 - __clz(z.kmax) : 0, abits = z.amax > 0 ? 32 - __clz(z.amax) : 0;
    for (int p = 0; p < kbits + abits + 14; p += 8) {
        const bool arr = p >= ((kbits + 7) & ~7);
        const int shift = arr ? p - ((kbits + 7) & ~7) : p;
        if (arr && shift >= abits) break;
        large_radix_pass(in, out, arr && shift == 0 ? S.a + base : nullptr, n, shift, cnt, pos);
        int2 *tmp = in;
        in = out;
        out = tmp;
    }
    for (int j = threadIdx.x; j < n; j += kLargeThreads) S.rec_a[base + j] = in[j].y;
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += kLargeThreads) {
        const int idx = S.rec_a[base + j];
        const int64_t g = base + idx;
        QEnt e;
        e.key = stage_key(S, g);
        e.idx = idx;
        e.s = S.s[g];
        e.o = S.o[g];
        S.rec[base + j] = e;
        S.rec_a[base + j] = S.a[g];
    }
}

__global__ void k_ratio(const DevResult *pol, const DevResult *ref, double *out, int32_t n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const DevResult a = pol[i], b = ref[i];
    double v = __longlong_as_double(0x7ff8000000000000ll);  // NaN
    if (a.status == ST_OK && b.status == ST_OK && b.total_latency > 0)
        v = double(a.total_latency) / double(b.total_latency);
    out[i] = v;
}

// Total latency and makespan in time units under the linear batch-time model (Section 6: each
// batch's time from a linear predictor; coef = c0, c1, c2, c3, c_idle):
//   out[2i]     = c0 X0 + c1 X1 + c2 X2 + c3 X3,
//   out[2i + 1] = c0 steps + c1 request_steps + c2 F2 + c3 F3 + c_idle (makespan - steps),
// from sums = X0..X3, F2, F3 of instance i, evaluated left to right with round-to-nearest products
// and sums (no fused multiply-add), so the result is the IEEE value of that expression.  NaN for an
// instance that did not finish.
__global__ void k_batch_time(const int64_t *sums, const DevResult *res, BtCoef c, double *out, int32_t n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const DevResult r = res[i];
    const int64_t *x = sums + 6 * int64_t(i);
    double tel = __longlong_as_double(0x7ff8000000000000ll), span = tel;
    if (r.status == ST_OK) {
        tel = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(c.k[0], __ll2double_rn(x[0])), __dmul_rn(c.k[1], __ll2double_rn(x[1]))),
                                  __dmul_rn(c.k[2], __ll2double_rn(x[2]))),
                        __dmul_rn(c.k[3], __ll2double_rn(x[3])));
        span = __dadd_rn(__dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(c.k[0], __ll2double_rn(r.steps)),
                                                       __dmul_rn(c.k[1], __ll2double_rn(r.request_steps))),
                                             __dmul_rn(c.k[2], __ll2double_rn(x[4]))),
                                   __dmul_rn(c.k[3], __ll2double_rn(x[5]))),
                         __dmul_rn(c.k[4], __ll2double_rn(r.makespan - r.steps)));
    }
    out[2 * int64_t(i)] = tel;
    out[2 * int64_t(i) + 1] = span;
}

}  // namespace

cudaError_t launch_batch_time(const int64_t *sums, const DevResult *res, const double *coef, double *out, int32_t n,
                              cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    BtCoef c;
    for (int k = 0; k < 5; ++k) c.k[k] = coef[k];
    k_batch_time<<<(n + 255) / 256, 256, 0, st>>>(sums, res, c, out, n);
    return cudaGetLastError();
}

cudaError_t launch_stage(const StageParams &p, cudaStream_t st, int *launches) {
    *launches = 0;
    if (p.n_inst <= 0) return cudaSuccess;
    // shared memory for the largest instance up to kStageSmemN, rounded up to a power of two
    int np = 1;
    const int want = (p.n_max > 0 && p.n_max < kStageSmemN) ? p.n_max : kStageSmemN;
    while (np < want) np <<= 1;
    const size_t smem = size_t(np) * kStageSmemBytesPerReq + kStageCntBytes;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k_stage, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
    }
    k_stage<<<p.n_inst, kStageThreads, smem, st>>>(p, np);
    *launches = 1;
    if (p.n_max > np) {
        k_stage_large<<<p.n_inst, kLargeThreads, 256 * kLargeWarps * sizeof(int32_t), st>>>(p, np);
        *launches = 2;
    }
    return cudaGetLastError();
}

cudaError_t launch_ratio(const DevResult *pol, const DevResult *ref, double *out, int32_t n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_ratio<<<(n + 255) / 256, 256, 0, st>>>(pol, ref, out, n);
    return cudaGetLastError();
}

}  // namespace simgb
