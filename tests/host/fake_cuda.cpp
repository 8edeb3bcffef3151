// The CUDA runtime and kernel launches that sim_api.cpp calls, on the host: streams are lists of operations
// that run when the stream is waited for, memory is malloc under a limit, and the simulation "kernel" notes
// the tie seeds that it finds.  For tests of the host code without a GPU.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <new>
#include <vector>

#include "sim.h"
#include "sim_internal.h"

namespace {

struct Stream {
    std::deque<std::function<void()>> ops;
    void run() {
        while (!ops.empty()) {
            auto op = ops.front();
            ops.pop_front();
            op();
        }
    }
};

Stream g_legacy;  // the null stream; every other one is non-blocking
size_t g_limit = size_t(1) << 40, g_used = 0, g_throw_above = SIZE_MAX;
std::map<void *, size_t> g_blocks;
cudaError_t g_last = cudaSuccess;
uint64_t g_seed = 0;
int32_t g_status = 0;
int64_t g_slots = 0, g_rho_calls = 0;

Stream &of(cudaStream_t s) { return s ? *reinterpret_cast<Stream *>(s) : g_legacy; }

std::map<const char *, size_t> g_pinned;
bool pinned(const void *p) {
    const char *c = static_cast<const char *>(p);
    auto it = g_pinned.upper_bound(c);
    return it != g_pinned.begin() && (--it, c < it->first + it->second);
}

void later_copy(Stream &st, void *dst, const void *src, size_t n, bool staged) {
    if (staged) {  // pageable: in a staging buffer when the call returns, on the device later
        std::vector<char> data(static_cast<const char *>(src), static_cast<const char *>(src) + n);
        st.ops.push_back([=] { std::memcpy(dst, data.data(), n); });
    } else {
        st.ops.push_back([=] { std::memcpy(dst, src, n); });
    }
}

}  // namespace

// an allocation on the host above the limit fails
void *operator new(size_t n, const std::nothrow_t &) noexcept { return n > g_throw_above ? nullptr : std::malloc(n ? n : 1); }
void *operator new(size_t n) {
    void *p = operator new(n, std::nothrow);
    if (!p) throw std::bad_alloc();
    return p;
}
void *operator new[](size_t n, const std::nothrow_t &t) noexcept { return operator new(n, t); }
void operator delete[](void *p) noexcept { std::free(p); }
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

extern "C" {

void fake_limits(size_t device_bytes, size_t host_bytes) {
    g_limit = device_bytes;
    g_throw_above = host_bytes;
}
size_t fake_used() { return g_used; }
uint64_t fake_seed() { return g_seed; }
void fake_status(int32_t s) { g_status = s; }
int64_t fake_slots() { return g_slots; }
int64_t fake_rho_calls() { return g_rho_calls; }
void *fake_stream() { return new Stream(); }

cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char *cudaGetErrorName(cudaError_t) { return "fake"; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 232448;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) {
    *p = nullptr;
    if (g_used + n > g_limit) return g_last = cudaErrorMemoryAllocation;
    // of very large blocks (queue buffers, never touched here) only the size counts
    *p = std::malloc(n < (size_t(1) << 31) ? n : 64);
    if (n < (size_t(1) << 26)) std::memset(*p, 0xab, n);
    g_blocks[*p] = n;
    g_used += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (p) {
        g_used -= g_blocks[p];
        g_blocks.erase(p);
        std::free(p);
    }
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    *p = std::malloc(n);
    g_pinned[static_cast<char *>(*p)] = n;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    g_pinned.erase(static_cast<char *>(p));
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = reinterpret_cast<cudaStream_t>(new Stream());
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return delete reinterpret_cast<Stream *>(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return of(s).run(), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind k, cudaStream_t s) {
    later_copy(of(s), dst, src, n, k == cudaMemcpyHostToDevice && !pinned(src));
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *dst, const void *src, size_t n, cudaMemcpyKind k) {
    later_copy(g_legacy, dst, src, n, k == cudaMemcpyHostToDevice && !pinned(src));
    if (k != cudaMemcpyHostToDevice) g_legacy.run();
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) {
    of(s).ops.push_back([=] { std::memset(p, v, n); });
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }

}  // extern "C"

namespace simgb {

cudaError_t launch_stage(const StageParams &, cudaStream_t, int *launches) { return *launches = 1, cudaGetLastError(); }
cudaError_t run_blocks_per_sm(int, const RunParams &, int, size_t, int *blocks) { return *blocks = 3, cudaSuccess; }
cudaError_t launch_run(int, const RunParams &p, int blocks, int warps_per_block, size_t, cudaStream_t st) {
    g_slots = int64_t(blocks) * warps_per_block;
    of(st).ops.push_back([p] {
        if (p.tie_seed) g_seed = p.tie_seed[0];
        for (int k = 0; k < p.n_work; ++k) {
            DevResult &r = p.res[p.work ? p.work[k] : k];
            std::memset(&r, 0, sizeof(r));
            r.status = p.use_smem ? g_status : 0;
        }
    });
    return cudaGetLastError();
}
cudaError_t launch_ratio(const DevResult *, const DevResult *, double *, int32_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_batch_time(const int64_t *, const DevResult *, const double *, double *, int32_t, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_lemma(int32_t, int32_t, int32_t, double, const double *, double *, cudaStream_t) { return cudaSuccess; }
cudaError_t rho_plan(int32_t, int32_t u_max, RhoPlan *plan) {
    *plan = {256, 8, 0, 7 * int64_t(u_max)};
    return cudaSuccess;
}
cudaError_t launch_rho(const RhoPlan &, int32_t n_u, const int32_t *us, double *out, double *, int32_t, cudaStream_t) {
    ++g_rho_calls;
    of(nullptr).ops.push_back([=] {
        for (int k = 0; k < n_u; ++k) out[k] = us[k];
    });
    return cudaGetLastError();
}

}  // namespace simgb
