// Simulation kernel of the batched scheduler simulator (sm_103a): k_run<policy, shared, instrumented>.
//
// One warp simulates one instance at a time (persistent warps pull instance ids from a work
// queue).  Each step follows the paper's algorithms:
//   S1  arrivals with a_i <= t join the waiting set R_t (extension: the paper has a_i = 0);
//   S3  A_min only (Algorithm milb): if the next step of the active set would exceed M, cancel
//       jobs in ascending estimate order, ties broken uniformly at random by a key drawn afresh
//       at every step (SplitMix64 of the instance's seed and the counter t * 2^32 + index, then
//       the index), until it fits; each cancelled job's estimate becomes max(estimate, tokens
//       generated) and it re-enters R_t in the same step;
//   S5  admit the largest prefix of R_t (sorted by (key, index)) for which eq. Constraint holds at
//       every future step (Algorithms malb / milb / off);
//   S6  process the batch: one token per member, the step's memory sum(s + tokens) (eq.
//       constraintM), completions, TEL (eq. latency).
// Two more policies share the loop: A_r (Algorithm random: the queue key is a given permutation
// rank, the projected length the true o) and A_ell (Algorithm promote_l: FIFO queue, estimate l;
// at the start of a step a job that used up its estimate unfinished is removed, takes u and
// re-enters the queue at its end; the queue key is 2 a on arrival and 2 t + 1 on re-entry).
//
// Active set (per warp, shared memory; a global-memory workspace of the same layout serves
// instances that outgrow it): an unordered array of slots, a job keeps its slot until it ends.
//   E = p + Lhat - 1   projected last step (Lhat = u, o or the A_min estimate)
//   V                  projected memory of the whole set at step E, kept up to date (valid while
//                      E >= t)
//   B = s - p + 1      the job's memory at step x is B + x
//   F = p + o - 1      true last step (completion at step F, C = F + 1)
//   P = p, I = request index, K = the estimate (A_min cancellation key)
// A free slot has E = F = -1 and K = 2^32 - 1, which no test below selects, so a pass over the set
// reads whole blocks of 64 slots without bounds checks.  With V(x) = sum over E_j >= x of
// (B_j + x) the projected memory of the set at step x (eq. Constraint restricted to S'), a
// candidate (prompt s, estimate L) started at step t ends at y = t + L - 1 and fits iff
//   (1) need + s + 1 <= M, need = sum of (B_j + t), the memory of the coming step,
//   (2) V_i + s + 1 + (E_i - t) <= M for every active endpoint t <= E_i <= y,
//   (3) V(y) + s + L <= M at its own last step.
// Between endpoints V(x) grows, so these points decide every future step.  (2) and (3) are one pass
// over the slots and three warp reductions.  A job (E, B) that joins or leaves adds or subtracts
// B + E_i at every endpoint E_i <= E: that update is left pending and applied by the next pass that
// tests a candidate, so an admission costs one pass, and a job that leaves at or after its E
// (every H-SF, A_r and A_min completion, every A_ell promotion) changes no V at all.  There are no
// sorted arrays, prefix sums or moves; freed slots are reclaimed by a compaction once they outnumber
// half of the live ones.  A candidate that fails also yields the first later step at which (2) and
// (3) could hold with the set unchanged; the steps up to the next event (that step, a completion, an
// arrival, an A_min overflow, an A_ell promotion) are processed in closed form.
//
// What bounds it: every instance is a serial chain of events, each a few dependent warp operations
// (a shared-memory round trip, three reductions, a decision), so the time of an event is latency and
// the rate of a full launch is the number of resident warps over that latency.
#include <climits>
#include <cstdint>

#include "sim_internal.h"

namespace simgb {

namespace {

constexpr unsigned FULL = 0xffffffffu;
enum { P_AMAX = 0, P_AMIN = 1, P_HSF = 2, P_AR = 3, P_AELL = 4 };
enum { ST_OK = 0, ST_INVAL = -1, ST_STEPCAP = -3, ST_STATE = -5 };
// Loops whose trip count is known only at run time carry `#pragma unroll 1`: unrolled copies grow
// the simulation loop, which the warps of a scheduler share through its instruction cache.
constexpr int kPage = 128;  // active-set slots per pass iteration (four per lane)
// s of the entry that stands for the head of an empty queue: never fits, greater than every entry
constexpr int kNoHead = 1 << 28;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

// Random tie key of request i at step t for A_min's cancellation order: the high 32 bits of
// output number t * 2^32 + i + 1 of the SplitMix64 generator seeded with `seed` (Steele, Lea and
// Flood, OOPSLA 2014, with the finalizer of Vigna's splitmix64.c): the state after k steps is
// seed + k * 0x9E3779B97F4A7C15, mixed by two xor-shift-multiply rounds and a final xor-shift.
// `base` = seed + t * 2^32 * 0x9E3779B97F4A7C15 (mod 2^64) is computed once per step.
__device__ __forceinline__ uint64_t tie_base(uint64_t seed, int t) {
    return seed + (uint64_t(uint32_t(t) * 0x7F4A7C15u) << 32);  // t * 2^32 * gamma mod 2^64
}

__device__ __forceinline__ unsigned tie_key(uint64_t base, int i) {
    uint64_t z = base + uint64_t(uint32_t(i) + 1u) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return unsigned(z >> 32);
}


__device__ __forceinline__ bool qless(const QEnt &a, const QEnt &b) {
    return a.key < b.key || (a.key == b.key && a.idx < b.idx);
}

// Projected length of a queue entry.  For A_max, A_min and H-SF the sort key is that length; A_r
// projects the true length o and A_ell the current estimate (l before a promotion, u after:
// promotions have odd keys).
template <int POL>
__device__ __forceinline__ int proj_len(const RunParams &P, int64_t base, const QEnt &e) {
    if (POL == P_AR) return e.o;
    if (POL == P_AELL) {
        const int2 lu = __ldg(P.lu + base + e.idx);
        return (e.key & 1) ? lu.y : lu.x;
    }
    return e.key;
}

// Number of leading positions i in [0, len) with pred(i) true (pred true on a prefix); warp-wide.
template <class Pred>
__device__ __forceinline__ int warp_prefix_count(int len, Pred pred) {
    if (len <= 0) return 0;
    const int lane = lane_id();
    const int c = (len + 31) >> 5;
    const int pos = min((lane + 1) * c - 1, len - 1);
    const int full = __popc(__ballot_sync(FULL, pred(pos)));
    int cnt = full * c;
    if (cnt >= len) return len;
    const int end = min(cnt + c, len);
    #pragma unroll 1
    for (int off = cnt; off < end; off += 32) {
        const int i = off + lane;
        const unsigned b = __ballot_sync(FULL, i < end && pred(i));
        const int k = __popc(b);
        cnt += k;
        if (k < 32) break;
    }
    return cnt;
}

// The same, computed by one lane alone (binary search).
template <class Pred>
__device__ __forceinline__ int lane_prefix_count(int len, Pred pred) {
    int lo = 0, hi = len;
    #pragma unroll 1
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (pred(mid)) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// ---------------------------------------------------------------------------------------------
// Per-warp workspace (layout: ws_bytes in sim_internal.h)
// ---------------------------------------------------------------------------------------------
struct Ws {
    int4 *H;         // active-set slots {E, V, B, F}, capacity ca (a multiple of kPage)
    QEnt *dq;        // delta queue, dcap entries, sorted DESCENDING (head = dq[dn-1])
    QEnt *mc;        // cached head of the main queue, kMc entries
    int32_t *cnt;    // merge histogram, dcap + 1 entries: the cache's space (a merge invalidates it)
    int2 *C;         // {P, I} per slot
    unsigned *K;     // A_min: the estimate per slot, UINT_MAX in a free one
    QEnt *mb0, *mb1;  // global ping-pong main-queue buffers
    int32_t ca, dcap;
};

__device__ __forceinline__ Ws carve_ws(unsigned char *base, int ca, int dcap) {
    Ws w;
    w.H = reinterpret_cast<int4 *>(base);
    w.dq = reinterpret_cast<QEnt *>(w.H + ca);
    w.mc = w.dq + dcap;
    w.cnt = reinterpret_cast<int32_t *>(w.mc);
    w.C = reinterpret_cast<int2 *>(reinterpret_cast<unsigned char *>(w.mc) + ws_cache_bytes(dcap));
    w.K = reinterpret_cast<unsigned *>(w.C + ca);
    w.ca = ca;
    w.dcap = dcap;
    return w;
}

// Position of the job A_min cancels when several jobs share the smallest estimate mk: the smallest
// (tie key, index) among them, the tie key drawn from `base` (tie_base of the step) or, under the
// index rule, the index itself.  Warp-wide; every lane gets the position.  Out of line: ties are a
// small share of the cancellations, and keeping the hashing out of the simulation loop keeps that
// loop's code small.
__device__ __noinline__ int tie_position(const unsigned *K, const int2 *C, int end, unsigned mk, uint64_t base,
                                         int rnd) {
    const int lane = lane_id();
    unsigned br = UINT_MAX, bi = UINT_MAX;
    int bp = -1;
    #pragma unroll 1
    for (int i = lane; i < end; i += 32) {
        if (K[i] == mk) {
            const unsigned id = unsigned(C[i].y);
            const unsigned r = rnd ? tie_key(base, int(id)) : id;
            if (r < br || (r == br && id < bi)) {
                br = r;
                bi = id;
                bp = i;
            }
        }
    }
    const unsigned mr = __reduce_min_sync(FULL, br);
    const unsigned mi = __reduce_min_sync(FULL, br == mr ? bi : UINT_MAX);
    const unsigned b = __ballot_sync(FULL, bp >= 0 && br == mr && bi == mi);
    return b ? __shfl_sync(FULL, bp, __ffs(b) - 1) : -1;
}

// ---------------------------------------------------------------------------------------------
// Waiting set R_t: a sorted main array in global memory [mh, me) (a run of kMc entries from its head
// cached in the workspace) plus a small sorted delta array (descending, so the head is the last
// entry).  Together they hold R_t in (key, idx) order.  Inserts go to the delta; a full delta is
// merged into the main array.
// ---------------------------------------------------------------------------------------------
struct Queue {
    const QEnt *mq;  // main array (global, ascending): the staged records or a merge buffer
    int mh, me;      // head / end
    int lim;         // entries of mq that may be read (the cache reads ahead of me up to here)
    int mbuf;        // -1: mq is the staged records; 0/1: ping-pong buffer in use
    int dn;          // delta size
    int mcb;         // main cache base: w.mc[i] = mq[mcb + i] for i < kMc; -1 invalid
};

// Make w.mc cover mq[mh].  The staged records are constant, so a cached run of them stays valid
// when later arrivals extend the main array.  gb counts the global-memory bytes the queue moves (a
// work counter of the instrumented kernel; a dead variable otherwise).
__device__ __forceinline__ void main_cache_at_head(const Ws &w, Queue &q, int64_t &gb) {
    if (q.mcb >= 0 && unsigned(q.mh - q.mcb) < unsigned(kMc)) return;
    const int lane = lane_id();
    gb += int64_t(min(kMc, q.lim - q.mh)) * int64_t(sizeof(QEnt));
    const int i0 = q.mh + lane, i1 = q.mh + 32 + lane;
    QEnt a, b;
    if (i0 < q.lim) a = q.mq[i0];
    if (i1 < q.lim) b = q.mq[i1];
    __syncwarp();
    if (i0 < q.lim) w.mc[lane] = a;
    if (i1 < q.lim) w.mc[32 + lane] = b;
    __syncwarp();
    q.mcb = q.mh;
}

// Merge the delta into the main array (into the other ping-pong buffer).  Rare (a full delta, or
// a long arrival run), so it is kept out of line: the simulation loop stays small enough for the
// instruction cache when two warps share a scheduler.  Takes the few workspace pointers it needs
// by value and the queue by pointer; gb (null in the plain kernel) counts the global bytes moved.
__device__ __noinline__ void merge_delta(int32_t *cnt, const QEnt *dq, QEnt *mb0, QEnt *mb1, Queue *qp, int64_t *gb) {
    const int lane = lane_id();
    Queue q = *qp;
    const int dn = q.dn;
    const int nx = q.me - q.mh;
    QEnt *out = (q.mbuf == 0) ? mb1 : mb0;
    const QEnt *X = q.mq + q.mh;
    #pragma unroll 1
    for (int j = lane; j <= dn; j += 32) cnt[j] = 0;
    __syncwarp();
    const int c = (nx + 31) >> 5;
    const int s0 = lane * c;
    const int s1 = min(s0 + c, nx);
    if (s0 < s1) {
        const QEnt x0 = X[s0];
        int r = lane_prefix_count(dn, [&](int m) { return qless(dq[dn - 1 - m], x0); });
        int run_r = r, run_len = 0;
        #pragma unroll 1
        for (int i = s0; i < s1; ++i) {
            const QEnt x = X[i];
            #pragma unroll 1
            while (r < dn && qless(dq[dn - 1 - r], x)) ++r;
            out[i + r] = x;
            if (r != run_r) {
                if (run_len) atomicAdd(&cnt[run_r], run_len);
                run_r = r;
                run_len = 0;
            }
            ++run_len;
        }
        if (run_len) atomicAdd(&cnt[run_r], run_len);
    }
    __syncwarp();
    // delta element j (ascending) goes to j + #{main entries smaller} = j + sum_{r <= j} cnt[r]
    int carry = 0;
    #pragma unroll 1
    for (int c0 = 0; c0 < dn; c0 += 32) {
        const int j = c0 + lane;
        int v = (j < dn) ? cnt[j] : 0;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(FULL, v, d);
            if (lane >= d) v += y;
        }
        v += carry;
        if (j < dn) out[j + v] = dq[dn - 1 - j];
        carry = __shfl_sync(FULL, v, 31);
    }
    __syncwarp();
    __threadfence_block();
    if (gb && lane == 0) *gb += int64_t(2 * nx + dn) * int64_t(sizeof(QEnt));  // main read once, merged written
    q.mq = out;
    q.mbuf = (q.mbuf == 0) ? 1 : 0;
    q.mh = 0;
    q.me = nx + dn;
    q.lim = nx + dn;
    q.dn = 0;
    q.mcb = -1;
    *qp = q;
}

__device__ __forceinline__ void merge_delta(const Ws &w, Queue &q, int64_t *gb) {
    Queue qq = q;
    merge_delta(w.cnt, w.dq, w.mb0, w.mb1, &qq, gb);
    q = qq;
}

// Insert one entry into the delta (merging the delta into main first if it is full: returns true).
__device__ __forceinline__ bool delta_insert(const Ws &w, Queue &q, const QEnt &e, int64_t *gb) {
    const int lane = lane_id();
    const bool full = q.dn == w.dcap;
    if (full) merge_delta(w, q, gb);
    const int dn = q.dn;
    // the smaller entries move one place right: usually all of them are among the last 32
    const int base = max(dn - 32, 0), i0 = base + lane;
    const QEnt d = w.dq[i0];
    const bool in = i0 < dn;
    const unsigned gt = __ballot_sync(FULL, in && qless(e, d));
    if (__reduce_max_sync(FULL, gt != 0u || base == 0)) {
        if (in && lane >= __popc(gt)) w.dq[i0 + 1] = d;
        w.dq[base + __popc(gt)] = e;
        __syncwarp();
        q.dn = dn + 1;
        return full;
    }
    const int pos = warp_prefix_count(dn, [&](int i) { return qless(e, w.dq[i]); });  // #entries > e
    #pragma unroll 1
    for (int hi = dn; hi > pos; hi -= 32) {
        const int lo = max(pos, hi - 32);
        const int i = lo + lane;
        QEnt v;
        const bool act = i < hi;
        if (act) v = w.dq[i];
        __syncwarp();
        if (act) w.dq[i + 1] = v;
        __syncwarp();
    }
    w.dq[pos] = e;
    __syncwarp();
    q.dn = dn + 1;
    return full;
}

// Head of R_t (smallest (key, idx)) and which part holds it (src 0: main, 1: delta), or the kNoHead entry
// if R_t is empty.  The main cache must cover q.mh.  No branches: both parts are read at a clamped
// position and an absent one is replaced by the kNoHead entry.
__device__ __forceinline__ QEnt queue_head(const Ws &w, const Queue &q, int &src) {
    const bool have_m = q.mh < q.me, have_d = q.dn > 0;
    QEnt hm = w.mc[have_m ? (q.mh - q.mcb) & (kMc - 1) : 0];
    QEnt hd = w.dq[have_d ? q.dn - 1 : 0];
    if (!have_m) {
        hm.key = hm.idx = INT_MAX;
        hm.s = kNoHead;
    }
    if (!have_d) {
        hd.key = hd.idx = INT_MAX;
        hd.s = kNoHead;
    }
    src = qless(hd, hm) ? 1 : 0;
    return src ? hd : hm;
}

// Arrival batch: the staged records [ap, ae), an ascending run.  It becomes the main array if that
// is empty and extends it under A_ell when it follows it in the staged records (FIFO keys); a few
// entries go into the delta one by one; a long batch is copied into the emptied delta in chunks.
template <int POL>
__device__ __forceinline__ void insert_run(const Ws &w, Queue &q, const QEnt *rec, int n, int ap, int ae, int64_t &gb,
                                           int64_t *gbp) {
    const int lane = lane_id();
    const int len = ae - ap;
    gb += int64_t(len) * int64_t(sizeof(QEnt));
    if (q.mh >= q.me) {
        if (q.mbuf != -1) {
            q.mq = rec;
            q.lim = n;
            q.mbuf = -1;
            q.mcb = -1;
        }
        q.mh = ap;
        q.me = ae;
        return;
    }
    if (POL == P_AELL && q.mbuf == -1 && q.me == ap) {
        q.me = ae;
        return;
    }
    const QEnt *run = rec + ap;
    int done = 0;
    #pragma unroll 1
    while (done < len) {
        const int rem = len - done;
        if (rem <= 8) {
            #pragma unroll 1
            for (int j = 0; j < rem; ++j) delta_insert(w, q, run[done + j], gbp);
            break;
        }
        if (q.dn > 0) merge_delta(w, q, gbp);
        const int k = min(rem, w.dcap);
        #pragma unroll 1
        for (int j = lane; j < k; j += 32) w.dq[j] = run[done + k - 1 - j];  // descending
        __syncwarp();
        q.dn = k;
        done += k;
    }
}

// A job (e, b) leaves the set: V loses b + E at the endpoints E <= e (free slots compare greater).
__device__ __forceinline__ void subtract_job(const Ws &w, int end, int e, int b) {
    #pragma unroll 1
    for (int p = 0; p < end; p += kPage) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = p + 32 * j + lane_id();
            const int2 ev = *reinterpret_cast<const int2 *>(&w.H[i]);
            if (unsigned(ev.x) <= unsigned(e)) w.H[i].y = ev.y - b - ev.x;
        }
    }
}

// Free slots [from, from + kPage).
template <int POL>
__device__ __forceinline__ void free_page(const Ws &w, int from) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int i = from + 32 * j + lane_id();
        w.H[i] = make_int4(-1, 0, 0, -1);
        if (POL == P_AMIN) w.K[i] = UINT_MAX;
    }
}

// Move the live slots to the front, in place, and free the rest of their blocks.
template <int POL>
__device__ __forceinline__ void compact(const Ws &w, int &end) {
    const int lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    int wpos = 0;
    #pragma unroll 1
    for (int b = 0; b < end; b += 32) {
        const int i = b + lane;
        const int4 h = w.H[i];
        const int2 c = w.C[i];
        const unsigned k = POL == P_AMIN ? w.K[i] : 0u;
        const bool live = i < end && h.w >= 0;
        const unsigned m = __ballot_sync(FULL, live);
        __syncwarp();
        if (live) {
            const int d = wpos + __popc(m & lt);
            w.H[d] = h;
            w.C[d] = c;
            if (POL == P_AMIN) w.K[d] = k;
        }
        __syncwarp();
        wpos += __popc(m);
    }
    #pragma unroll 1
    for (int i = wpos + lane; i < end; i += 32) {
        w.H[i] = make_int4(-1, 0, 0, -1);
        if (POL == P_AMIN) w.K[i] = UINT_MAX;
    }
    end = wpos;
    __syncwarp();
}

// Invariants of the simulation state between events (SIM_OPT_DEBUG_CHECKS; global-memory kernel
// only): the live slots number A and sum to need; nextF is their smallest F; V is the projected memory
// at every endpoint not yet passed (with the pending update); under A_max, H-SF and A_r no job runs
// past its projected last step; free slots are free; the delta queue is strictly descending and the
// cached head of the main array ascending.  Returns false on the first violation.
template <int POL>
__device__ bool state_ok(const Ws &w, const Queue &q, int A, int end, int t, int need, int nextF, int py, int pm,
                         int pc, int filled) {
    const int lane = lane_id();
    bool bad = false;
    unsigned fmin = UINT_MAX;
    int cnt = 0, sum = 0;
    #pragma unroll 1
    for (int i = lane; i < filled; i += 32) {
        const int4 h = w.H[i];
        if (h.w < 0) {
            if (h.x != -1 || (POL == P_AMIN && w.K[i] != UINT_MAX)) bad = true;
            continue;
        }
        if (i >= end) bad = true;
        ++cnt;
        sum += h.z + t;
        fmin = min(fmin, unsigned(h.w));
        if ((POL == P_AMAX || POL == P_HSF || POL == P_AR) && h.w > h.x) bad = true;
        if (POL == P_AMIN && w.K[i] != unsigned(h.x - w.C[i].x + 1)) bad = true;
        if (h.x < t) continue;
        int v = 0;
        #pragma unroll 1
        for (int j = 0; j < end; ++j)
            if (w.H[j].x >= h.x) v += w.H[j].z + h.x;
        if (v != h.y + (unsigned(h.x) <= unsigned(py) ? pm * h.x + pc : 0)) bad = true;
    }
    if (int(__reduce_add_sync(FULL, unsigned(cnt))) != A || int(__reduce_add_sync(FULL, unsigned(sum))) != need) bad = true;
    #pragma unroll 1
    for (int i = lane; i + 1 < q.dn; i += 32)
        if (!qless(w.dq[i + 1], w.dq[i])) bad = true;
    if (q.mcb >= 0)
        #pragma unroll 1
        for (int i = q.mh + lane; i + 1 < min(q.me, q.mcb + kMc); i += 32)
            if (i >= q.mcb && !qless(w.mc[i - q.mcb], w.mc[i + 1 - q.mcb])) bad = true;
    fmin = __reduce_min_sync(FULL, fmin);
    if (A > 0 && fmin != unsigned(nextF)) bad = true;
    return __ballot_sync(FULL, bad) == 0;
}

// ---------------------------------------------------------------------------------------------
// One instance, simulated by one warp.  All lanes hold identical copies of the scalar state.
// INS: the instrumented copy, which also keeps the work counters of the per-step method and the
// batch-time sums; the plain copy has neither.
// All memory sums are at most M <= 2^26 where they are compared (V, need and a candidate's points
// belong to feasible schedules, a violated one exceeds M by one job's memory at most), so 32 bits
// hold them; steps stay below kMaxStep + 2^26.
// ---------------------------------------------------------------------------------------------
template <int POL, bool SMEM, bool INS>
__device__ __forceinline__ void sim_instance(const RunParams &P, const Ws &w0, int inst) {
    const int lane = lane_id();
    const InstInfo info = P.info[inst];
    // delta capacity for this instance: shifts in the delta cost O(capacity) per insertion, merges
    // into the main array O(n) per capacity insertions; a small delta suits a short queue
    Ws w = w0;
    w.dcap = min(w0.dcap, delta_cap(info.n));
    DevResult r;
    r.total_latency = r.makespan = r.peak_memory = r.evictions = r.steps = r.request_steps = 0;
    r.status = info.status;
    r.pad = 0;
    if (info.status == ST_OK && int64_t(info.n) > P.main_cap) r.status = ST_INVAL;  // larger than the queue buffers
    if (r.status != ST_OK || info.n == 0) {
        if (lane == 0) P.res[inst] = r;
        return;
    }
    const int n = info.n;
    const QEnt *rec = P.rec + info.base;
    const int32_t *ra = P.rec_a + info.base;
    const uint64_t tie_seed = (POL == P_AMIN && P.tie_seed) ? P.tie_seed[inst] : 0ull;
    const int M = int(P.M);
    const int64_t cap = info.cap;

    Queue q;
    q.mq = rec;
    q.mh = q.me = 0;
    q.lim = n;
    q.mbuf = -1;
    q.dn = 0;
    q.mcb = -1;
    // global-memory bytes moved by the queue (instrumented kernel); the merge adds through gbp
    int64_t gbq = 0;
    int64_t *const gbp = INS ? &gbq : nullptr;
    // work counters of the paper's per-step method (Theorem complexity), accumulated per step in
    // closed form: S2 adds (the active set), S3 compare-exchanges of the overflow sort
    // (A ceil(log2 A)^2), S5 endpoint evaluations of a binary-search admission
    // ((A' + k) ceil(log2(Q + 1))); k_step / ev_step: admitted / removed at the current step
    int64_t cS2 = 0, cS3 = 0, cS5 = 0;
    int k_step = 0, ev_step = 0;

    // Batch time (Section 6's linear batch-time model, coefficients given later): bx0..bx3 =
    // X0..X3, the sums over requests of the processed steps, batch sizes, step memories and
    // prefill tokens of the steps a_i .. C_i - 1 (an arrival at t subtracts the prefixes up to t,
    // a completion at C adds those up to C); bmem, bpf the prefixes of step memory and prefill
    // (steps and request steps have their own counters).
    const bool bt = INS && P.batch_time != nullptr;
    int64_t bx0 = 0, bx1 = 0, bx2 = 0, bx3 = 0, bmem = 0, bpf = 0;

    // A live jobs in the slots [0, end), the slots [0, filled) initialised; need: the memory of step
    // t; nextF, nextE: the smallest F and (A_ell) E; py, pm, pc: the pending update V += pm E + pc at
    // the endpoints E <= py (pm = 0: none)
    int A = 0, end = 0, filled = kPage, need = 0;
    unsigned nextF = UINT_MAX, nextE = UINT_MAX;
    int py = 0, pm = 0, pc = 0;
    free_page<POL>(w, 0);
    // steps processed = t - tb (tb moves with every idle gap); the instance stops at step tstop (the
    // step cap or kMaxStep); trare = min(tstop, next arrival)
    int t = ra[0], tb = t;
    const auto stop_at = [&]() { return int(min(int64_t(tb) + min(cap, int64_t(INT_MAX)), int64_t(kMaxStep) + 1)); };
    int tstop = stop_at();
    // arrival steps of the records [apb, apb + 32), one per lane
    int ap = 0, apb = 0, next_a = t, trare = t;
    int pa = lane < n ? ra[lane] : INT_MAX;
    int64_t sumC = 0, rsteps = 0, nev = 0;
    // 32 bits suffice (fewer live registers): makespan <= t + 1 with t <= kMaxStep + 1, and the peak
    // is a step's memory, <= M <= 2^26
    int makespan = 0, peak = 0;
    int ndone = 0;
    int status = ST_OK;

    // the head of R_t: entry h with projected length hL from the main (hsrc 0) or delta (1) part; it
    // does not fit before step fit_lb unless the set changes
    QEnt h;
    h.key = h.idx = INT_MAX;
    h.s = kNoHead;
    h.o = 0;
    int hL = 1, hsrc = 0, fit_lb = 0;
    // what the next iteration has to look at first
    enum { HEAD = 1, NEXTF = 2, SLOTS = 4, IDLE = 8 };
    int attn = 0;

    const auto load_head = [&](bool cached) {  // cached: w.mc covers q.mh (else h is reloaded before use)
        h = queue_head(w, q, hsrc);
        hL = h.key;
        if (POL == P_AR || POL == P_AELL) hL = cached && h.s != kNoHead ? proj_len<POL>(P, info.base, h) : 1;
    };

    // The conditions of all warp-uniform branches below are warp reductions: the compiler then knows
    // that they are uniform and emits plain jumps (about 12 cycles) instead of reconvergence blocks
    // (about 45, measured), and one reduction (29) decides several of them.  Single-value stores are
    // made by all lanes alike, for the same reason.
    for (;;) {
        if (!SMEM && P.debug && attn == 0 && !state_ok<POL>(w, q, A, end, t, need, int(nextF), py, pm, pc, filled)) {
            status = ST_STATE;  // a consistency check of SIM_OPT_DEBUG_CHECKS failed
            break;
        }
        unsigned fl = 0;
        if (attn != 0 || t >= trare || (POL == P_AELL && unsigned(t) > nextE)) fl |= 1u;
        if (POL == P_AMIN && need > M) fl |= 2u;
        if (t >= fit_lb && need + h.s < M) fl |= 4u;
        if (unsigned(t) == nextF) fl |= 8u;
        fl = __reduce_or_sync(FULL, fl);
        if (fl & 1u) {
            if (end >= min(filled, w.ca) || (attn & SLOTS)) {  // reclaim free slots, or take a new page
                if (end - A >= max(16, A >> 3) || (end >= w.ca && A < end)) {
                    compact<POL>(w, end);
                } else if (end >= w.ca) {
                    status = kStatusCapacity;
                    break;
                } else if (end >= filled) {
                    free_page<POL>(w, filled);
                    filled += kPage;
                    __syncwarp();
                }
            }
            if (t >= tstop) {
                status = ST_STEPCAP;
                break;
            }
            if (POL == P_AMIN && (attn & NEXTF)) {
                unsigned f = UINT_MAX;
                #pragma unroll 1
                for (int i = lane; i < end; i += 32) f = min(f, unsigned(w.H[i].w));
                nextF = __reduce_min_sync(FULL, f);
            }
            bool dirty = (attn & HEAD) != 0;
            attn = 0;
            // ---- S1: arrivals with a <= t join R_t (a sorted run of the staged records)
            if (next_a <= t) {
                int ae;
                if (__ldg(ra + n - 1) <= t) {
                    ae = n;
                    next_a = INT_MAX;
                } else {
                    ae = ap;
                    for (;;) {
                        const unsigned later = __ballot_sync(FULL, apb + lane >= ae && pa > t);
                        if (later) {
                            const int k = __ffs(later) - 1;
                            ae = apb + k;
                            next_a = __shfl_sync(FULL, pa, k);
                            break;
                        }
                        apb += 32;
                        ae = apb;
                        pa = apb + lane < n ? ra[apb + lane] : INT_MAX;
                    }
                }
                insert_run<POL>(w, q, rec, n, ap, ae, gbq, gbp);
                if (INS) gbq += int64_t(ae - ap) * 4;  // their arrival steps
                if (bt) {
                    const int64_t m = ae - ap;
                    bx0 -= m * (t - tb);
                    bx1 -= m * rsteps;
                    bx2 -= m * bmem;
                    bx3 -= m * bpf;
                }
                ap = ae;
                trare = min(tstop, next_a);
                dirty = true;
            }
            // ---- A_ell: jobs that used up their estimate unfinished (E < t) leave the batch and
            // re-enter the queue at its end with the estimate u (the delta orders their equal keys by
            // index)
            if (POL == P_AELL && unsigned(t) > nextE) {
                if (t > kAellMaxStep) {
                    status = ST_STEPCAP;
                    break;
                }
                unsigned f = UINT_MAX, e1 = UINT_MAX;
                #pragma unroll 1
                for (int b = 0; b < end; b += 32) {
                    const int4 hh = w.H[b + lane];
                    const bool out = unsigned(hh.x) < unsigned(t);
                    if (!out) {
                        f = min(f, unsigned(hh.w));
                        e1 = min(e1, unsigned(hh.x));
                    }
                    unsigned m = __ballot_sync(FULL, out);
                    #pragma unroll 1
                    while (m) {
                        const int pos = b + __ffs(m) - 1;
                        m &= m - 1;
                        const int4 j = w.H[pos];
                        const int2 pi = w.C[pos];
                        __syncwarp();
                        w.H[pos] = make_int4(-1, 0, 0, -1);
                        __syncwarp();
                        QEnt e;
                        e.key = 2 * t + 1;
                        e.idx = pi.y;
                        e.s = j.z + pi.x - 1;
                        e.o = j.w - pi.x + 1;
                        need -= j.z + t;
                        --A;
                        ++nev;
                        if (INS) ++ev_step;
                        delta_insert(w, q, e, gbp);
                    }
                }
                nextF = __reduce_min_sync(FULL, f);
                nextE = __reduce_min_sync(FULL, e1);
                dirty = true;
                fit_lb = 0;
            }
            if (dirty) {
                const int hi = h.idx, hk = h.key;
                if (q.mh < q.me) main_cache_at_head(w, q, gbq);
                load_head(true);
                if (h.idx != hi || h.key != hk) fit_lb = 0;
            }
            if (A == 0 && h.s == kNoHead) {
                if (ap >= n) {
                    status = ST_STATE;
                    break;
                }
                tb += next_a - t;  // idle: jump to the next arrival
                t = next_a;
                tstop = stop_at();
                trare = min(tstop, next_a);
            }
            continue;
        }
        // ---- S2/S3: A_min overflow of the next step -> cancel in ascending (estimate, tie key, index)
        if (POL == P_AMIN && (fl & 2u)) {
            if (INS) {
                const int lg = A > 1 ? 32 - __clz(A - 1) : 0;
                cS3 += int64_t(A) * lg * lg;
            }
            // Cancellation order (estimate, r, index), r the step's tie key (SplitMix64 of the seed
            // and t * 2^32 + index; under the index rule r = index, the same order).  A round
            // finds the smallest estimate and the first and last slot that hold it; only when these
            // differ does tie_position draw and compare the tied jobs' keys.  (On the 40960 x 2000
            // workload 1.3 % of the overflow steps have a tie at the smallest estimate.)
            #pragma unroll 1
            while (need > M) {
                unsigned bk = UINT_MAX;
                int lo = 0, hi = 0;
                #pragma unroll 1
                for (int p = 0; p < end; p += kPage) {
                    const int i = p + 4 * lane;
                    const uint4 k = *reinterpret_cast<const uint4 *>(w.K + i);
                    const unsigned m = min(min(k.x, k.y), min(k.z, k.w));
                    const int first = i + (k.x == m ? 0 : (k.y == m ? 1 : (k.z == m ? 2 : 3)));
                    const int last = i + (k.w == m ? 3 : (k.z == m ? 2 : (k.y == m ? 1 : 0)));
                    if (m < bk) lo = first;
                    if (m <= bk) hi = last;
                    bk = min(bk, m);
                }
                const unsigned mk = __reduce_min_sync(FULL, bk);
                int pos = int(__reduce_min_sync(FULL, bk == mk ? unsigned(lo) : UINT_MAX));
                const int pos2 = int(__reduce_max_sync(FULL, bk == mk ? unsigned(hi) : 0u));
                if (mk == UINT_MAX) {  // no live job
                    status = ST_STATE;
                    break;
                }
                if (pos != pos2) pos = tie_position(w.K, w.C, end, mk, tie_base(tie_seed, t), P.evict_index == 0);
                const int4 j = w.H[pos];
                const int2 pi = w.C[pos];
                __syncwarp();
                w.H[pos] = make_int4(-1, 0, 0, -1);
                w.K[pos] = UINT_MAX;
                __syncwarp();
                QEnt e;
                e.key = max(int(mk), t - pi.x);  // refined lower bound: max(estimate, tokens generated)
                e.idx = pi.y;
                e.s = j.z + pi.x - 1;
                e.o = j.w - pi.x + 1;
                need -= j.z + t;
                --A;
                ++nev;
                if (INS) ++ev_step;
                if (unsigned(j.w) == nextF) attn |= NEXTF;
                // endpoints before t need no update, and the update is left pending if none is
                const int do_sub = j.x < t ? 0 : (pm == 0 ? 1 : 2);
                if (__reduce_max_sync(FULL, do_sub) == 2) {
                    subtract_job(w, end, j.x, j.z);
                } else if (do_sub) {
                    py = j.x;
                    pm = -1;
                    pc = -j.z;
                }
                if (delta_insert(w, q, e, gbp)) attn |= HEAD;
                if (qless(e, h)) {  // the head of R_t is the smaller of the two
                    h = e;
                    hL = e.key;
                    hsrc = 1;
                }
            }
            if (status != ST_OK) break;
            fit_lb = 0;
            if (A == 0) attn |= IDLE;
            if (end - A >= max(16, A >> 3) && ((end - 1) ^ max(A - 1, 0)) >= kPage) attn |= SLOTS;
            continue;
        }
        // ---- S4/S5: admit the largest feasible prefix of R_t, one candidate at a time ((1) holds)
        if (fl & 4u) {
            const int y = t + hL - 1;
            const int c1 = h.s + 1 - M;
            int vy = 0, r2 = INT_MIN;
            unsigned em = UINT_MAX;
            #pragma unroll 1
            for (int p = 0; p < end; p += kPage) {
                int4 a[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) a[j] = w.H[p + 32 * j + lane];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (unsigned(a[j].x) <= unsigned(py)) {
                        a[j].y += pm * a[j].x + pc;
                        w.H[p + 32 * j + lane].y = a[j].y;
                    }
                    if (a[j].x >= y) vy += a[j].z + y;
                    em = min(em, unsigned(a[j].x - y));
                    // d = E - t: (2) asks V + d + s + 1 <= M; it holds from step t + (V + d + s + 1 - M)
                    // on, or once the endpoint has passed (t + d + 1)
                    const int d = a[j].x - t;
                    if (unsigned(d) < unsigned(hL)) r2 = max(r2, min(a[j].y + d + c1, d + 1));
                }
            }
            pm = pc = 0;
            vy = int(__reduce_add_sync(FULL, unsigned(vy)));
            em = __reduce_min_sync(FULL, em);
            // (3) at y; if it fails it cannot hold before y passes the next endpoint y + em
            if (vy + h.s + hL > M) r2 = max(r2, int(em) + 1);
            const int d = __reduce_max_sync(FULL, r2);
            if (d > 0) {
                // no fit before step t + d, and none at all if (1) fails there
                fit_lb = int64_t(need) + int64_t(A) * d + h.s + 1 > M ? INT_MAX : t + d;
            } else {
                // the pending update of its own admission adds the job's memory at y to its V
                __syncwarp();
                w.H[end] = make_int4(y, vy, h.s - t + 1, t + h.o - 1);
                w.C[end] = make_int2(t, h.idx);
                if (POL == P_AMIN) w.K[end] = unsigned(h.key);
                py = y;
                pm = 1;
                pc = h.s - t + 1;
                ++end;
                ++A;
                need += h.s + 1;
                nextF = min(nextF, unsigned(t + h.o - 1));
                if (POL == P_AELL) nextE = min(nextE, unsigned(y));
                if (INS) ++k_step;
                if (bt) bpf += h.s;  // prefill: the prompts of the admitted requests
                q.dn -= hsrc;
                q.mh += 1 - hsrc;
                const bool miss = q.mh < q.me && unsigned(q.mh - q.mcb) >= unsigned(kMc);
                if (miss) attn |= HEAD;
                if (end >= min(filled, w.ca)) attn |= SLOTS;
                load_head(!miss);
                fit_lb = 0;
                __syncwarp();
                continue;
            }
        }
        // ---- S6: process the batch
        if (fl & 8u) {
            if (need > M) status = ST_STATE;  // the step's memory; an internal error, reported at the end
            peak = max(peak, need);
            rsteps += A;
            if (bt) bmem += need;
            if (INS) {
                const int Qa = (q.me - q.mh) + q.dn;  // R_t after admission
                cS2 += A - k_step + ev_step;
                cS5 += int64_t(A) * (32 - __clz(Qa + k_step));
                k_step = ev_step = 0;
            }
            // the jobs with F = t complete (C = t + 1)
            if (P.completion) {
                #pragma unroll 1
                for (int i = lane; i < end; i += 32)
                    if (w.H[i].w == t) P.completion[info.base + w.C[i].y] = int64_t(t) + 1;
            }
            // A job that ends before its projected last step changes V: its slot keeps E (in place of
            // V) and B, and F = -2 - t tells it from the slots freed at other steps.
            constexpr bool kEarly = POL == P_AMAX || POL == P_AELL;
            int c = 0, sm = 0, ne = 0, ek = -1, bk = INT_MIN;
            unsigned f = UINT_MAX, e1 = UINT_MAX;
            #pragma unroll 1
            for (int p = 0; p < end; p += kPage) {
                int4 a[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) a[j] = w.H[p + 32 * j + lane];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool done = a[j].w == t, early = kEarly && done && a[j].x > t;
                    if (done) {
                        w.H[p + 32 * j + lane] = make_int4(-1, a[j].x, a[j].z, early ? -2 - t : -1);
                        if (POL == P_AMIN) w.K[p + 32 * j + lane] = UINT_MAX;
                        sm += a[j].z + t;
                        ++c;
                    } else {
                        f = min(f, unsigned(a[j].w));
                        if (POL == P_AELL) e1 = min(e1, unsigned(a[j].x));
                    }
                    if (early) {
                        ++ne;
                        ek = a[j].x;
                        bk = a[j].z;
                    }
                }
            }
            c = int(__reduce_add_sync(FULL, unsigned(c)));
            sm = int(__reduce_add_sync(FULL, unsigned(sm)));
            nextF = __reduce_min_sync(FULL, f);
            if (POL == P_AELL) nextE = __reduce_min_sync(FULL, e1);
            if (kEarly) {
                ne = int(__reduce_add_sync(FULL, unsigned(ne + (lane == 0 && pm != 0 ? 1 : 0))));
                ek = __reduce_max_sync(FULL, ek);
                bk = __reduce_max_sync(FULL, bk);
                if (ne == 1 && ek >= 0) {  // one such job, and no update pending: leave this one pending
                    py = ek;
                    pm = -1;
                    pc = -bk;
                }
                if (ne > 1 && ek >= 0) {
                    #pragma unroll 1
                    for (int b = 0; b < end; b += 32) {
                        const int4 x = w.H[b + lane];
                        unsigned m = __ballot_sync(FULL, x.w == -2 - t);
                        #pragma unroll 1
                        while (m) {
                            const int src = __ffs(m) - 1;
                            m &= m - 1;
                            subtract_job(w, end, __shfl_sync(FULL, x.y, src), __shfl_sync(FULL, x.z, src));
                        }
                    }
                }
            }
            A -= c;
            need += A - sm;
            ++t;
            makespan = t;
            sumC += int64_t(c) * t;
            if (bt) {
                bx0 += int64_t(c) * (t - tb);
                bx1 += int64_t(c) * rsteps;
                bx2 += int64_t(c) * bmem;
                bx3 += int64_t(c) * bpf;
            }
            ndone += c;
            fit_lb = 0;
            if (A == 0) attn |= IDLE;
            if (end - A >= max(16, A >> 3) && ((end - 1) ^ max(A - 1, 0)) >= kPage) attn |= SLOTS;
            if (ndone >= n) break;
        } else {
            // steps t .. tau-1 change nothing: no completion before nextF, no arrival before
            // trare, (A_min) no overflow, (A_ell) no promotion, and the head does not fit before fit_lb
            // (or at all, once (1) fails: need only grows while the set stays as it is)
            int tau = min(min(int(nextF), trare), need + h.s < M ? fit_lb : INT_MAX);
            if (POL == P_AELL) tau = min(tau, int(nextE) + 1);
            // the first step whose memory exceeds M
            if (POL == P_AMIN) tau = min(tau, t + int(unsigned(M - need) / unsigned(max(A, 1))) + 1);
            const int c = max(tau - t, 1);
            const int64_t mem = int64_t(need) + int64_t(A) * (c - 1);
            if (mem > M) status = ST_STATE;  // an internal error, reported at the end
            peak = max(peak, int(mem));
            rsteps += int64_t(A) * c;
            if (bt)  // steps t .. t+c-1 have memory need + A (x - t)
                bmem += c * int64_t(need) + int64_t(A) * (int64_t(c) * (c - 1) / 2);
            if (INS) {
                const int Qa = (q.me - q.mh) + q.dn;
                cS2 += int64_t(A) * c - k_step + ev_step;
                cS5 += int64_t(A) * (32 - __clz(Qa + k_step)) + int64_t(A) * (c - 1) * (32 - __clz(Qa));
                k_step = ev_step = 0;
            }
            need = int(mem) + A;
            t += c;
        }
    }
    if (lane == 0) {
        r.status = status;
        r.total_latency = sumC - info.sum_a;
        r.makespan = makespan;
        r.peak_memory = peak;
        r.evictions = nev;
        r.steps = t - tb;
        r.request_steps = rsteps;
        P.res[inst] = r;
        if (bt) {
            int64_t *o = P.batch_time + 6 * int64_t(inst);
            const bool ok = status == ST_OK;
            o[0] = ok ? bx0 : 0;
            o[1] = ok ? bx1 : 0;
            o[2] = ok ? bx2 : 0;
            o[3] = ok ? bx3 : 0;
            o[4] = ok ? bmem : 0;
            o[5] = ok ? bpf : 0;
        }
        if (INS && P.work_count) {
            int64_t *wc = P.work_count + 4 * int64_t(inst);
            wc[0] = cS2;
            wc[1] = cS3;
            wc[2] = cS5;
            wc[3] = gbq;
        }
    }
    __syncwarp();
}

template <int POL, bool SMEM, bool INS>
__global__ void __launch_bounds__(256, 2) k_run(RunParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id();
    const int wib = threadIdx.x >> 5;
    const int64_t slot = int64_t(blockIdx.x) * (blockDim.x >> 5) + wib;
    unsigned char *base;
    if (SMEM) base = smem_raw + size_t(wib) * ws_bytes(POL == P_AMIN, P.ca, P.dcap);
    else base = P.gws + slot * P.gws_stride;
    Ws w = carve_ws(base, P.ca, P.dcap);
    w.mb0 = P.mainbuf + slot * 2 * P.main_cap;
    w.mb1 = w.mb0 + P.main_cap;
    for (;;) {
        int k = 0;
        if (lane == 0) k = atomicAdd(P.counter, 1);
        k = __shfl_sync(FULL, k, 0);
        if (k >= P.n_work) break;
        const int inst = P.work ? P.work[k] : k;
        sim_instance<POL, SMEM, INS>(P, w, inst);
    }
}

using KernelFn = void (*)(RunParams);

template <int POL>
KernelFn pick(bool smem, bool ins) {
    if (smem) return ins ? k_run<POL, true, true> : k_run<POL, true, false>;
    return ins ? k_run<POL, false, true> : k_run<POL, false, false>;
}

KernelFn run_fn(int policy, const RunParams &p) {
    const bool smem = p.use_smem != 0, ins = p.work_count != nullptr || p.batch_time != nullptr;
    switch (policy) {
        case P_AMAX: return pick<P_AMAX>(smem, ins);
        case P_AMIN: return pick<P_AMIN>(smem, ins);
        case P_HSF: return pick<P_HSF>(smem, ins);
        case P_AR: return pick<P_AR>(smem, ins);
        default: return pick<P_AELL>(smem, ins);
    }
}

}  // namespace

cudaError_t run_blocks_per_sm(int policy, const RunParams &p, int warps_per_block, size_t smem_bytes, int *blocks) {
    const KernelFn fn = run_fn(policy, p);
    if (smem_bytes > 48 * 1024) {
        const cudaError_t e =
            cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem_bytes));
        if (e != cudaSuccess) return e;
    }
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, (const void *)fn, 32 * warps_per_block, smem_bytes);
}

cudaError_t launch_run(int policy, const RunParams &p, int blocks, int warps_per_block, size_t smem_bytes,
                       cudaStream_t st) {
    run_fn(policy, p)<<<dim3(blocks), dim3(32 * warps_per_block), smem_bytes, st>>>(p);
    return cudaGetLastError();
}

}  // namespace simgb
