// Analytic competitive-ratio evaluators of A_min (double precision, sm_103a).
//
//   k_lemma   - Lemma thm:Amin for a batch of length histograms, walked from the longest length down.
//               With X_k, S1_k, S2_k the sums over i >= k of x_i, i x_i, x_i / (s + i) and
//               G_k = sum over i > k of (i - k) x_i / (s + i) = G_{k+1} + S2_{k+1},
//                 numerator   = sum_k d_k S1_k (2 G_k + d_k S2_k)   (d_k = 1, and s + l at k = l),
//                 denominator = sum_k k (s + k) x_k (x_k + 2 X_{k+1}) = sum_k D_k X_k^2,
//               D_k = k (s + k) - (k - 1)(s + k - 1) = s + 2 k - 1 above l and l (s + l) at l
//               (x_k (x_k + 2 X_{k+1}) = X_k^2 - X_{k+1}^2, summed by parts): eight FP64 operations
//               per length and, for a histogram of counts, sums of positive terms only.
//               GB300's FP64 rate (two lanes per SM and cycle) bounds it, not HBM.  A group of T
//               lanes shares a histogram: T = 1 when there are enough histograms to fill the FP64
//               pipes; otherwise each lane first sums its segment of lengths (four operations per
//               length), the lanes' sums are scanned and each lane walks its segment with the sums of
//               the segments above it.  2^20 histograms of 64 lengths take 0.97 ms (14 operations per
//               length and a cancelling T - k S2 in place of G: 1.72 ms); 333 of 1999 lengths 0.044 ms
//               (one lane each: 1.96 ms).  RMS error against 128-bit sums 1.0e-16 and 1.4e-16 (before:
//               1.3e-16 and 1.1e-15).
//   k_rho     - spectral radius of B_u^{-1} A_u (Corollary A/B; s = 0, l = 1), the bound on the
//               Rayleigh quotient of Section 4.1, by power iteration from v = (1, .., 1).
//               b_ij = min(i, j)^2, so with the suffix sums S_i = sum_{j >= i} v_j,
//                 v' B v = sum_i (2 i - 1) S_i^2,
//               and one step v <- B^{-1} A v reads, in the suffix sums (w_i = 3 i^2 - 3 i + 1),
//                 S_i <- [ (3 - 2 / i) S_i + sum_k S_k + (sum_{k < i} w_k S_k) / (i (i - 1))
//                          + w_i sum_{k > i} S_k / (k (k - 1)) ] / (2 (2 i - 1))
//               (a_ij = i j / 2 + j^2 - j^3 / (2 i) for j <= i; differences of A v in i, summed by
//               parts).  Every term is positive, so nothing cancels, and v' A v = sum_i (2 i - 1) S_i S'_i.
//               A thread-block cluster works on one u, each thread on a run of consecutive i: sums of
//               its run, a scan over the block and the cluster (one cluster barrier per step), then its
//               run again.  The arrays stay in shared memory when they fit.  12 FP64 operations per
//               index and step (constants from arrays); FP64 rate and the serial steps (about 15) bound it.  u = 20,000:
//               0.37 ms, 10^5: 0.71 ms, 2^20: 4.8 ms; 25 values up to 20,000: 0.50 ms, half of it the call's
//               allocation and copies.  (One warp per u,
//               with four scans of totals minus prefixes, seven divisions per index and the tridiagonal
//               B^{-1} applied to A v: 573 ms for the 25 values, relative error 2e-9 at u = 20,000 against
//               4e-16 now.)
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "sim_internal.h"

namespace simgb {

namespace {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(FULL, v, d);
    return v;
}

// Sum over the lanes below this one (up) or above it (down).
__device__ __forceinline__ double excl_up(double v, double &total) {
    const int lane = threadIdx.x & 31;
    double x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const double y = __shfl_up_sync(FULL, x, d);
        if (lane >= d) x += y;
    }
    total = __shfl_sync(FULL, x, 31);
    const double e = __shfl_up_sync(FULL, x, 1);
    return lane == 0 ? 0.0 : e;
}

__device__ __forceinline__ double excl_down(double v, double &total) {
    const int lane = threadIdx.x & 31;
    double x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const double y = __shfl_down_sync(FULL, x, d);
        if (lane + d < 32) x += y;
    }
    total = __shfl_sync(FULL, x, 0);
    const double e = __shfl_down_sync(FULL, x, 1);
    return lane == 31 ? 0.0 : e;
}

// The running sums of a walk that has passed n lengths.
struct LemmaSums {
    double X, S1, S2, G;
    int n;
};

// The sums after the segment b follows the lengths summed in a.
__device__ __forceinline__ LemmaSums then(const LemmaSums &a, const LemmaSums &b) {
    return {a.X + b.X, a.S1 + b.S1, a.S2 + b.S2, fma(double(b.n), a.S2, a.G) + b.G, a.n + b.n};
}

static_assert(3 * kLemmaMaxLen * sizeof(double) <= 227 * 1024, "k_lemma's table");

template <int T>
__global__ void __launch_bounds__(256) k_lemma(int32_t n_hist, int32_t len, int32_t l, double s,
                                                const double *__restrict__ x, double *__restrict__ out) {
    // per-length constants shared by every histogram: 1/(s+k), k, D_k
    extern __shared__ double tab[];
    double *rinv = tab, *kk = tab + len, *dk = tab + 2 * len;
    for (int j = threadIdx.x; j < len; j += blockDim.x) {
        const double k = double(l + j);
        rinv[j] = 1.0 / (s + k);
        kk[j] = k;
        dk[j] = j == 0 ? k * (s + k) : s + 2.0 * k - 1.0;
    }
    __syncthreads();
    const int64_t h = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) / T;
    if (T == 1 && h >= n_hist) return;
    const int g = threadIdx.x % T;
    const double *xh = x + min(h, int64_t(n_hist) - 1) * int64_t(len);
    // lane g of the group takes the lengths [lo, hi), lane 0 the longest ones; an odd number per
    // lane keeps the lanes' table reads on different banks
    const int m = T == 1 ? len : ((len + T - 1) / T) | 1;
    const int hi = max(len - g * m, 0), lo = T == 1 ? 0 : max(hi - m, 0);
    LemmaSums p = {0.0, 0.0, 0.0, 0.0, 0};
    if (T > 1) {
        for (int j = hi - 1; j >= lo; --j) {
            const double xk = __ldg(xh + j);
            p.X += xk;
            p.S1 = fma(kk[j], xk, p.S1);
            p.S2 = fma(rinv[j], xk, p.S2);
            p.G += p.S2;
        }
        p.n = hi - lo;
        // inclusive scan over the group, then shift by one lane
#pragma unroll
        for (int d = 1; d < T; d <<= 1) {
            const LemmaSums q = {__shfl_up_sync(FULL, p.X, d, T), __shfl_up_sync(FULL, p.S1, d, T),
                                 __shfl_up_sync(FULL, p.S2, d, T), __shfl_up_sync(FULL, p.G, d, T),
                                 __shfl_up_sync(FULL, p.n, d, T)};
            if (g >= d) p = then(q, p);
        }
        p = {__shfl_up_sync(FULL, p.X, 1, T), __shfl_up_sync(FULL, p.S1, 1, T), __shfl_up_sync(FULL, p.S2, 1, T),
             __shfl_up_sync(FULL, p.G, 1, T), 0};
        if (g == 0) p = {0.0, 0.0, 0.0, 0.0, 0};
    }
    double num = 0.0, den = 0.0;
#pragma unroll 4
    for (int j = hi - 1; j >= max(lo, 1); --j) {
        const double xk = __ldg(xh + j);
        p.X += xk;                                      // sum_{i>=k} x_i
        p.S1 = fma(kk[j], xk, p.S1);                    // sum_{i>=k} i x_i
        p.S2 = fma(rinv[j], xk, p.S2);                  // sum_{i>=k} x_i/(s+i)
        num = fma(p.S1, fma(2.0, p.G, p.S2), num);      // G: sum_{i>k} (i-k) x_i/(s+i)
        den = fma(dk[j], p.X * p.X, den);
        p.G += p.S2;
    }
    if (lo == 0 && hi > 0) {  // k = l
        const double xk = __ldg(xh);
        const double delta = s + double(l);
        p.X += xk;
        p.S1 = fma(kk[0], xk, p.S1);
        p.S2 = fma(rinv[0], xk, p.S2);
        num = fma(delta * p.S1, fma(2.0, p.G, delta * p.S2), num);
        den = fma(dk[0], p.X * p.X, den);
    }
    if (T > 1) {
#pragma unroll
        for (int d = T / 2; d >= 1; d >>= 1) {
            num += __shfl_xor_sync(FULL, num, d, T);
            den += __shfl_xor_sync(FULL, den, d, T);
        }
    }
    if (g == 0 && h < n_hist) out[h] = num / den;
}

// Blocks of 256 threads, or of one warp for small u: threads without an index take part in the scans all the
// same, and those keep the FP64 pipes busy (10^5 values of u = 7: 42.4 ms with 256 threads, 7.1 with one warp;
// of u = 128: 45.8 and 14.0).  A few values fill no pipe and gain from more threads above one index per lane
// (u = 7: 0.215 and 0.192 ms, u = 128: 0.212 and 0.244).
constexpr int kRhoThreads = 256;
static int rho_threads(int32_t n_u, int32_t u_max) { return u_max <= (n_u > 1024 ? 128 : 32) ? 32 : kRhoThreads; }
constexpr size_t kRhoSmemMax = size_t(200) * 1024;
constexpr int kRhoArrays = 7;  // per i: S, T, 1/(i(i-1)), 1/(8(2i-1)), w_i, 3 - 2/i, 2i - 1

template <int NT>
__global__ void __launch_bounds__(NT) k_rho(const int32_t *__restrict__ us, double *__restrict__ out,
                                                      double *scratch, int64_t stride, int32_t max_iter) {
    namespace cg = cooperative_groups;
    constexpr int kW = NT / 32;
    extern __shared__ double rho_smem[];
    __shared__ double wsum[5][kW];  // per warp: p1, Q, T, numerator, denominator
    __shared__ double part[2][5];   // per block, double-buffered over steps, read by the cluster
    cg::cluster_group cl = cg::this_cluster();
    const int C = int(cl.num_blocks()), rank = int(cl.block_rank());
    const int64_t id = blockIdx.x / C;
    const int u = us[id];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    // this block's indices [lo, hi) (0-based: entry e is i = e + 1), this thread's [a, b)
    const int R = (u + C - 1) / C;
    const int lo = min(rank * R, u), hi = min(lo + R, u);
    const int m = ((hi - lo + NT - 1) / NT) | 1;  // odd: the runs start on different banks
    const int a = min(lo + tid * m, hi), b = min(a + m, hi);
    // arrays over the block's indices, in shared memory or in the scratch of this u
    double *S = scratch ? scratch + id * stride + int64_t(kRhoArrays) * lo : rho_smem;
    double *tv = S + (hi - lo), *rk = tv + (hi - lo), *bb = rk + (hi - lo);
    double *ww = bb + (hi - lo), *cc = ww + (hi - lo), *dd = cc + (hi - lo);
    S -= lo;
    tv -= lo;
    rk -= lo;
    bb -= lo;
    ww -= lo;
    cc -= lo;
    dd -= lo;
    for (int e = a; e < b; ++e) {
        const double i = double(e + 1);
        S[e] = double(u - e);
        rk[e] = e == 0 ? 0.0 : 1.0 / (i * (i - 1.0));
        bb[e] = 0.125 / (2.0 * i - 1.0);  // a quarter of 1 / (2 (2 i - 1)): S neither grows nor vanishes
        ww[e] = fma(3.0 * i, i - 1.0, 1.0);
        cc[e] = 3.0 - 2.0 / i;
        dd[e] = 2.0 * i - 1.0;
    }
    double lam = 0.0, num = 0.0, den = 0.0;
    for (int it = 0; it <= max_iter; ++it) {
        // sums over this thread's run
        double p1 = 0.0, Q = 0.0, T = 0.0;
        for (int e = a; e < b; ++e) {
            const double v = S[e];
            p1 += v;
            Q = fma(ww[e], v, Q);
            T = fma(rk[e], v, T);
        }
        // exclusive prefix of Q, suffix of T, and totals, over the warp, the block and the cluster
        double tq, tt;
        double q = excl_up(Q, tq), tl = excl_down(T, tt);
        p1 = warp_sum(p1);
        num = warp_sum(num);
        den = warp_sum(den);
        if (lane == 0) {
            wsum[0][wid] = p1;
            wsum[1][wid] = tq;
            wsum[2][wid] = tt;
            wsum[3][wid] = num;
            wsum[4][wid] = den;
        }
        __syncthreads();
        double *mine = part[it & 1];
        if (tid < 5) {
            double acc = 0.0;
            for (int k = 0; k < kW; ++k) acc += wsum[tid][k];
            mine[tid] = acc;
        }
        for (int k = 0; k < wid; ++k) q += wsum[1][k];
        for (int k = kW - 1; k > wid; --k) tl += wsum[2][k];
        cl.sync();
        double tot[3] = {0.0, 0.0, 0.0};  // p1, numerator, denominator over the cluster
        for (int k = 0; k < C; ++k) {
            const double *pk = cl.map_shared_rank(mine, k);
            tot[0] += pk[0];
            if (k < rank) q += pk[1];
            if (k > rank) tl += pk[2];
            tot[1] += pk[3];
            tot[2] += pk[4];
        }
        if (it > 0) {  // the Rayleigh quotient of the vector of step it - 1
            const double nl = 0.5 * tot[1] / tot[2];
            const bool done = it > 1 && fabs(nl - lam) <= 1e-15 * nl;
            lam = nl;
            if (done) break;
        }
        // T_i = sum over k > i, from the end of the run
        for (int e = b - 1; e >= a; --e) {
            tv[e] = tl;
            tl = fma(rk[e], S[e], tl);
        }
        // the step, from its start
        num = den = 0.0;
        for (int e = a; e < b; ++e) {
            const double v = S[e], w = ww[e];
            const double br = fma(w, tv[e], fma(rk[e], q, fma(cc[e], v, tot[0])));
            num = fma(v, br, num);
            den = fma(dd[e] * v, v, den);
            q = fma(w, v, q);
            S[e] = bb[e] * br;
        }
    }
    if (rank == 0 && tid == 0) out[id] = lam;
    cl.sync();  // no block leaves while another may still read its sums
}

}  // namespace

cudaError_t launch_lemma(int32_t n_hist, int32_t len, int32_t l, double s, const double *x, double *out,
                         cudaStream_t st) {
    if (n_hist <= 0) return cudaSuccess;
    int dev = 0, n_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    // Lanes per histogram: the least (rounds of one warp per scheduler) x (operations of a lane's
    // walk, 8 per length alone and 12 shared); a scheduler's FP64 pipe is busy with one warp.
    const auto cost = [&](int T) {
        const int64_t warps = (int64_t(n_hist) * T + 31) / 32, rounds = (warps + 4 * n_sm - 1) / (4 * n_sm);
        return rounds * ((len + T - 1) / T) * (T == 1 ? 8 : 12);
    };
    int T = 1;
    for (int c = 2; c <= 32 && c <= len; c <<= 1)
        if (cost(c) < cost(T)) T = c;
    // blocks of four warps (one per scheduler, which also share the table's divisions) unless larger ones
    // still give every SM one: 333 histograms of 1999 lengths take 44 us with 128 threads, 50 with 64 and
    // 66 with 256
    const int64_t lanes = int64_t(n_hist) * T;
    const int threads = (lanes + 255) / 256 < n_sm ? 128 : 256;
    const unsigned blocks = unsigned((lanes + threads - 1) / threads);
    const size_t smem = size_t(3) * len * sizeof(double);
    using Fn = void (*)(int32_t, int32_t, int32_t, double, const double *, double *);
    const Fn fn = T == 1 ? k_lemma<1> : T == 2 ? k_lemma<2> : T == 4 ? k_lemma<4> : T == 8 ? k_lemma<8>
                  : T == 16 ? k_lemma<16> : k_lemma<32>;
    if (smem > 48 * 1024) {
        // to the longest histograms' bytes, not to this launch's: other threads share the kernel
        e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(3 * kLemmaMaxLen * sizeof(double)));
        if (e != cudaSuccess) return e;
    }
    fn<<<blocks, threads, smem, st>>>(n_hist, len, l, s, x, out);
    return cudaGetLastError();
}

static size_t rho_smem_bytes(int cluster, int32_t u_max) {
    const size_t b = size_t((u_max + cluster - 1) / cluster) * kRhoArrays * sizeof(double);
    return b <= kRhoSmemMax ? b : 0;  // 0: the arrays live in global scratch
}

static cudaLaunchConfig_t rho_config(const RhoPlan &plan, int32_t n_u, cudaLaunchAttribute *attr, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(n_u) * unsigned(plan.cluster));
    cfg.blockDim = dim3(unsigned(plan.threads));
    cfg.dynamicSmemBytes = plan.smem;
    cfg.stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = unsigned(plan.cluster);
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Blocks per cluster: about 512 indices of the largest u each, at most 8 blocks, or 16 (which k_rho opts
// in to) for a few values: a GPU partition holds few clusters of 16, and 25 values of up to 20,000 took
// 0.79 ms with 16 blocks each, one of 10^5 0.70 ms (8 blocks: 1.0).
cudaError_t rho_plan(int32_t n_u, int32_t u_max, RhoPlan *plan) {
    cudaError_t e = cudaFuncSetAttribute((const void *)k_rho<kRhoThreads>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kRhoSmemMax));
    if (e == cudaSuccess) e = cudaFuncSetAttribute((const void *)k_rho<kRhoThreads>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    plan->threads = rho_threads(n_u, u_max);
    const int most = n_u <= 8 ? 16 : 8;
    plan->cluster = 1;
    while (plan->cluster < most && 512 * plan->cluster < u_max) plan->cluster <<= 1;
    plan->smem = rho_smem_bytes(plan->cluster, u_max);
    if (plan->cluster == 16) {  // needs 16 SMs of one partition, where not every SM need be available
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = rho_config(*plan, 1, &attr, nullptr);
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, k_rho<kRhoThreads>, &cfg) != cudaSuccess || fit < 1) {
            cudaGetLastError();
            plan->cluster = 8;
            plan->smem = rho_smem_bytes(8, u_max);
        }
    }
    plan->scratch = plan->smem ? 0 : int64_t(kRhoArrays) * u_max;
    return cudaSuccess;
}

cudaError_t launch_rho(const RhoPlan &plan, int32_t n_u, const int32_t *us, double *out, double *scratch,
                       int32_t max_iter, cudaStream_t st) {
    if (n_u <= 0) return cudaSuccess;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = rho_config(plan, n_u, &attr, st);
    return cudaLaunchKernelEx(&cfg, plan.threads == 32 ? k_rho<32> : k_rho<kRhoThreads>, us, out, scratch, plan.scratch,
                              max_iter);
}

}  // namespace simgb
