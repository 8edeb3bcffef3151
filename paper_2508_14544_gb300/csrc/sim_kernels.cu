// Simulation kernel of the batched scheduler simulator (sm_103a): k_run<policy, shared, instrumented, wide, slots>.
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
//   W = V(E) + E       V(E) the projected memory of the whole set at step E, kept up to date (valid
//                      while E >= t)
//   B = s - p + 1      the job's memory at step x is B + x
//   F = p + o - 1      true last step (completion at step F, C = F + 1)
//   P = p, I = request index, K = the estimate (A_min cancellation key)
// A free slot has E = F = -1 and K = 2^32 - 1, which no test below selects, so a pass over the set
// reads whole half pages (64 slots) or pages (128) without bounds checks.  With V(x) = sum over E_j >= x of
// (B_j + x) the projected memory of the set at step x (eq. Constraint restricted to S'), a
// candidate (prompt s, estimate L) started at step t ends at y = t + L - 1 and fits iff
//   (1) need + s + 1 <= M, need = sum of (B_j + t), the memory of the coming step,
//   (2) V(E_i) + s + 1 + (E_i - t) <= M, i.e. W_i <= M - s - 1 + t, for every active endpoint
//       t <= E_i <= y,
//   (3) V(y) + s + L <= M at its own last step.
// Between endpoints V(x) grows, so these points decide every future step.  (2) and (3) are one pass
// over the slots and two warp reductions.  A job (E, B) that joins or leaves adds or subtracts
// B + E_i in W_i at every endpoint E_i <= E: one such update of each kind is left pending and applied by
// the next pass that reads the slots anyway (a candidate's test, A_min's scan for the smallest
// estimate), so an admission costs one pass, and a job that leaves at or after its E (every H-SF, A_r
// and A_min completion, every A_ell promotion) changes no W at all.  There are no sorted arrays, prefix
// sums or moves; freed slots are reclaimed by a compaction when that saves a page.  A candidate that
// fails yields the first later step at which (2) and (3) could hold with the set unchanged; the steps up
// to the next event (that step, a completion, an arrival, an A_min overflow, an A_ell promotion) are
// processed in closed form.  It also leaves a witness (c, V(c)): the violated step that would last longest.
// V(c) is carried along through admissions and completions (a job with E >= c counts B + c), and a head
// with t <= c <= y, the same or another, cannot fit before V(c) + s + 1 + (c - t) <= M or c has passed: a
// few instructions in place of most of the tests that fail after every change of the set.  A_max takes
// 5-17 % less with it (64 x 10^5 online 145 -> 129 ms, load sweep 1.61 -> 1.34, a tenth of the alpha sweep
// 4.43 -> 4.23), A_r 13 % (4.36 -> 3.80), A_ell 6 % (11.2 -> 10.5), H-SF 5-7 %, but 1 % more on 64 x 10^5
// online.  A_min, whose tests follow cancellations and mostly admit, took 0-4 % longer: it keeps none.
//
// What bounds it: every instance is a serial chain of events, each a few dependent warp operations
// (a shared-memory round trip, two reductions, a decision), so the time of an event is latency, and
// with many instances the issue slots (64-68 % used at 16 warps per SM).  Against the set kept sorted with
// suffix sums and prefix maxima: A_min on 40960 x 2000 248 -> 105 ms, A_max 50 -> 33, H-SF 38 -> 22;
// A_min's slowest instance of 1024 x 1000 alone 14.8 -> 7.9 ms; A_max on 64 x 10^5 402 -> 129 ms.
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
constexpr int kPage = kCaUnit;  // active-set slots per pass iteration (four per lane)
constexpr int kHalf = 64;   // sets whose slots end here are passed over in one half page (two per lane)
// s of the entry that stands for the head of an empty queue: never fits, greater than every entry
constexpr int kNoHead = 1 << 28;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ int64_t warp_slot() {
    return int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
}

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

// floor(a / b) for 0 <= a < 2^22, b >= 1, by a reciprocal and one correction each way (the estimate is
// off by less than one); a lower bound of it for larger a (there the estimate is off by less than 40).
// About half the latency of the integer division.
__device__ __forceinline__ int quotient_lb(int a, int b) {
    const int q = __float2int_rz(__fdividef(float(a), float(b)));
    const int r = a - q * b;
    return a >= (1 << 22) ? max(q - 40, 0) : q + (r >= b ? 1 : 0) - (r < 0 ? 1 : 0);
}

// Sums modulo 2^32.  W of a free slot or of an endpoint before t, and V of a witness that has passed, go on
// taking updates that nobody reads, and wrap on long streams.
__device__ __forceinline__ int plus(int a, int b) { return int(unsigned(a) + unsigned(b)); }
__device__ __forceinline__ int minus(int a, int b) { return int(unsigned(a) - unsigned(b)); }

__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// ---------------------------------------------------------------------------------------------
// Per-warp workspace (layout: ws_bytes in sim_internal.h)
// ---------------------------------------------------------------------------------------------
struct Ws {
    int2 *EW;        // active-set slots {E, W}, capacity ca (a multiple of kPage)
    int32_t *B, *F;  // and their B and F
    QEnt *dq;        // delta queue, dcap entries, sorted DESCENDING (head = dq[dn-1])
    QEnt *mc;        // cached head of the main queue, kMc entries
    int32_t *cnt;    // merge positions, dcap entries: the cache's space (a merge invalidates it)
    int2 *C;         // {P, I} per slot
    unsigned *K;     // A_min: the estimate per slot, UINT_MAX in a free one
    int32_t ca, dcap;
};

// The slot arrays and the head cache come first: with a capacity known at compile time they are constant
// offsets from one address.
__device__ __forceinline__ Ws carve_ws(unsigned char *base, int ca, int dcap) {
    Ws w;
    w.EW = reinterpret_cast<int2 *>(base);
    w.B = reinterpret_cast<int32_t *>(w.EW + ca);
    w.F = w.B + ca;
    w.C = reinterpret_cast<int2 *>(w.F + ca);
    w.mc = reinterpret_cast<QEnt *>(w.C + ca);
    w.cnt = reinterpret_cast<int32_t *>(w.mc);
    w.K = reinterpret_cast<unsigned *>(reinterpret_cast<unsigned char *>(w.mc) + kWsCacheBytes);
    w.dq = reinterpret_cast<QEnt *>(w.K + ca);
    w.ca = ca;
    w.dcap = dcap;
    return w;
}

// Position of the job A_min cancels when several jobs share the smallest estimate mk, the first of them
// at slot `first` and the last at `last`: the smallest (tie key, index) among them, the tie key drawn
// from `base` (tie_base of the step) or, under the index rule, the index itself.  Warp-wide; every
// lane gets the position.
__device__ __forceinline__ int tie_position(const unsigned *K, const int2 *C, int first, int last, unsigned mk,
                                            uint64_t base, int rnd) {
    unsigned br = UINT_MAX, bi = UINT_MAX;
    int bp = 0;
    int b = first & ~31;
    #pragma unroll 1
    do {
        const int i = b + lane_id();
        const unsigned id = unsigned(C[i].y);
        const unsigned r = rnd ? tie_key(base, int(id)) : id;
        const bool less = K[i] == mk && (r < br || (r == br && id < bi));
        br = less ? r : br;
        bi = less ? id : bi;
        bp = less ? i : bp;
        b += 32;
    } while (b <= last);
    const unsigned mr = __reduce_min_sync(FULL, br);
    const unsigned mi = __reduce_min_sync(FULL, br == mr ? bi : UINT_MAX);
    return int(__reduce_min_sync(FULL, br == mr && bi == mi ? unsigned(bp) : UINT_MAX));
}

// ---------------------------------------------------------------------------------------------
// Waiting set R_t: a sorted main array in global memory [mh, me) (a run of kMc entries from its head
// cached in the workspace) plus a small sorted delta array (descending, so the head is the last
// entry).  Together they hold R_t in (key, idx) order.  Inserts go to the delta; a full delta is
// merged into the main array.
// A_ell's queue is first in, first out: its main array is a run of the staged records that arrivals extend,
// and in place of the delta stand the promotions, appended to the instance's merge buffer (a request is
// promoted at most once) and read through a second cached run of kMc entries in the delta's space.  The
// projected lengths (l of an arrival, u of a promotion) are fetched with the cached runs, into K.
// ---------------------------------------------------------------------------------------------
struct Queue {
    const QEnt *mq;  // main array (global, ascending): the staged records or a merge buffer
    int mh, me;      // head / end
    int lim;         // entries of mq that may be read (the cache reads ahead of me up to here)
    int mbuf;        // -1: mq is the staged records; 0/1: ping-pong buffer in use
    int dn;          // delta size
    int dh, dce;     // A_ell: head of the promotions, end of their cached run (from dcb)
    int dcb;
    int mcb;         // main cache base: w.mc[i] = mq[mcb + i] for i < kMc; -1 invalid
};

// Make w.mc cover mq[mh].  The staged records are constant, so a cached run of them stays valid
// when later arrivals extend the main array.  gb counts the global-memory bytes the queue moves (a
// work counter of the instrumented kernel; a dead variable otherwise).  lu: A_ell's (l, u) table.
template <int POL>
__device__ __forceinline__ void main_cache_at_head(const Ws &w, Queue &q, const int2 *lu, int64_t &gb) {
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
    if (POL == P_AELL) {
        if (i0 < q.lim) w.K[lane] = unsigned(lu[a.idx].x);
        if (i1 < q.lim) w.K[32 + lane] = unsigned(lu[b.idx].x);
    }
    __syncwarp();
    q.mcb = q.mh;
}

// A_ell: make w.dq cover the head of the promotions `pl`, which must not be empty.
__device__ __forceinline__ void promo_cache_at_head(const Ws &w, Queue &q, const QEnt *pl, const int2 *lu, int64_t &gb) {
    if (q.dh < q.dce) return;
    const int lane = lane_id();
    const int m = min(q.dn, kMc);
    gb += int64_t(m) * int64_t(sizeof(QEnt));
    __syncwarp();
    #pragma unroll 1
    for (int i = lane; i < m; i += 32) {
        const QEnt e = pl[q.dh + i];
        w.dq[i] = e;
        w.K[kMc + i] = unsigned(lu[e.idx].y);
    }
    __syncwarp();
    q.dcb = q.dh;
    q.dce = q.dh + m;
}

// Merge the delta into the main array (into the other ping-pong buffer).  Rare (a full delta, or
// a long arrival run), so it is kept out of line.  Takes the few workspace pointers it needs by value and
// the queue by pointer; gb (null in the plain kernel) counts the global bytes moved.
// The delta is short and the main array long (up to the instance's requests): each delta entry finds
// its place in the main array by binary search, two searches per lane in flight, and the main array is
// then copied in coalesced runs of 128 entries, shifted by the number of delta entries before each.
// (More in flight costs registers, which count toward the simulation loop's: eight loads instead of four
// made the loop spill and every policy 25-60 % slower.)
__device__ __noinline__ void merge_delta(int32_t *pos, const QEnt *dq, QEnt *mb0, QEnt *mb1, Queue *qp, int64_t *gb) {
    const int lane = lane_id();
    Queue q = *qp;
    const int dn = q.dn;
    const int nx = q.me - q.mh;
    QEnt *out = (q.mbuf == 0) ? mb1 : mb0;
    const QEnt *X = q.mq + q.mh;
    #pragma unroll 1
    for (int j0 = lane; j0 < dn; j0 += 64) {
        const int j1 = j0 + 32;
        const int2 d0 = *reinterpret_cast<const int2 *>(&dq[dn - 1 - j0]);
        const int2 d1 = *reinterpret_cast<const int2 *>(&dq[j1 < dn ? dn - 1 - j1 : 0]);
        int lo0 = 0, hi0 = nx, lo1 = 0, hi1 = nx;
        #pragma unroll 1
        while (lo0 < hi0 || lo1 < hi1) {
            const int m0 = (lo0 + hi0) >> 1, m1 = (lo1 + hi1) >> 1;
            const int2 x0 = *reinterpret_cast<const int2 *>(&X[min(m0, nx - 1)]);
            const int2 x1 = *reinterpret_cast<const int2 *>(&X[min(m1, nx - 1)]);
            const bool l0 = x0.x < d0.x || (x0.x == d0.x && x0.y < d0.y);
            const bool l1 = x1.x < d1.x || (x1.x == d1.x && x1.y < d1.y);
            if (lo0 < hi0) {
                if (l0) lo0 = m0 + 1; else hi0 = m0;
            }
            if (lo1 < hi1) {
                if (l1) lo1 = m1 + 1; else hi1 = m1;
            }
        }
        pos[j0] = lo0;  // main entries before delta entry j (ascending)
        out[lo0 + j0] = dq[dn - 1 - j0];
        if (j1 < dn) {
            pos[j1] = lo1;
            out[lo1 + j1] = dq[dn - 1 - j1];
        }
    }
    __syncwarp();
    int r = 0;  // delta entries before main entry b
    #pragma unroll 1
    for (int b = 0; b < nx; b += 128) {
        QEnt x[4];
        int sh[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = b + 32 * k + lane;
            if (i < nx) x[k] = X[i];
            sh[k] = i + r;
        }
        #pragma unroll 1
        for (; r < dn && pos[r] < b + 128; ++r) {
            const int p = pos[r];
#pragma unroll
            for (int k = 0; k < 4; ++k) sh[k] += p <= b + 32 * k + lane ? 1 : 0;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (b + 32 * k + lane < nx) out[sh[k]] = x[k];
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

// The ping-pong buffers (of the warp's slot, or of the instance at its first request `base`) are found
// here, not held in registers.
__device__ __forceinline__ void merge_delta(const RunParams &P, const Ws &w, Queue &q, int64_t base, int n, int64_t *gb) {
    Queue qq = q;
    const bool slots = P.main_cap > 0;
    QEnt *mb = P.mainbuf + 2 * (slots ? warp_slot() * P.main_cap : base);
    merge_delta(w.cnt, w.dq, mb, mb + (slots ? P.main_cap : n), &qq, gb);
    q = qq;
}

// Insert one entry into the delta, which is not full.
__device__ __forceinline__ void delta_put(const Ws &w, Queue &q, const QEnt &e) {
    const int lane = lane_id();
    const int dn = q.dn;
    // the smaller entries move one place right: usually all of them are among the last 32
    const int base = max(dn - 32, 0), i0 = base + lane;
    const QEnt d = w.dq[i0];
    const bool in = i0 < dn;
    const unsigned gt = __ballot_sync(FULL, in && qless(e, d));
    if (gt != 0u || base == 0) {
        if (in && lane >= __popc(gt)) w.dq[i0 + 1] = d;
        w.dq[base + __popc(gt)] = e;
        __syncwarp();
        q.dn = dn + 1;
        return;
    }
    // otherwise: its place by one count over the keys, and the entries behind it moved from the back
    int greater = 0;
    #pragma unroll 2
    for (int i = lane; i < dn; i += 32) {
        const int2 k = *reinterpret_cast<const int2 *>(&w.dq[i]);
        greater += e.key < k.x || (e.key == k.x && e.idx < k.y) ? 1 : 0;
    }
    const int pos = int(__reduce_add_sync(FULL, unsigned(greater)));
    #pragma unroll 1
    for (int hi = dn; hi > pos; hi -= 32) {
        const int i = hi - 32 + lane;
        QEnt v;
        if (i >= pos) v = w.dq[i];
        __syncwarp();
        if (i >= pos) w.dq[i + 1] = v;
        __syncwarp();
    }
    w.dq[pos] = e;
    __syncwarp();
    q.dn = dn + 1;
}

// The same, merging the delta into main first if it is full.
__device__ __forceinline__ void delta_insert(const RunParams &P, const Ws &w, Queue &q, const QEnt &e, int64_t base, int n,
                                             int64_t *gb) {
    if (q.dn == w.dcap) merge_delta(P, w, q, base, n, gb);
    delta_put(w, q, e);
}

// Head of R_t (smallest (key, idx)), its projected length and which part holds it (src 0: main, 1: delta),
// or the kNoHead entry if R_t is empty.  The main cache must cover q.mh (A_ell: and w.dq q.dh).  No
// branches: both parts are read at a clamped position and an absent one is replaced by the kNoHead
// entry.  For A_max, A_min and H-SF the sort key is the projected length; A_r projects the true length.
template <int POL>
__device__ __forceinline__ QEnt queue_head(const Ws &w, const Queue &q, int &src, int &len) {
    const bool have_m = q.mh < q.me, have_d = q.dn > 0;
    const int im = have_m ? (q.mh - q.mcb) & (kMc - 1) : 0;
    const int id = POL == P_AELL ? (q.dh - q.dcb) & (kMc - 1) : (have_d ? q.dn - 1 : 0);
    QEnt hm = w.mc[im];
    QEnt hd = w.dq[id];
    if (!have_m) {
        hm.key = hm.idx = INT_MAX;
        hm.s = kNoHead;
    }
    if (!have_d) {
        hd.key = hd.idx = INT_MAX;
        hd.s = kNoHead;
    }
    src = qless(hd, hm) ? 1 : 0;
    const QEnt h = src ? hd : hm;
    len = POL == P_AELL ? int(w.K[src ? kMc + id : im]) : POL == P_AR ? h.o : h.key;
    return h;
}

// Arrival batch: the staged records [ap, ae), an ascending run.  It becomes the main array if that
// is empty and extends it under A_ell (FIFO keys, and it follows it in the staged records); a few entries
// go into the delta one by one; a long batch is copied into the emptied delta in chunks.
template <int POL>
__device__ __forceinline__ void insert_run(const RunParams &P, const Ws &w, Queue &q, int64_t base, int n, int ap,
                                           int ae, int64_t &gb, int64_t *gbp) {
    const QEnt *rec = P.rec + base;
    const int lane = lane_id();
    const int len = ae - ap;
    gb += int64_t(len) * int64_t(sizeof(QEnt));
    if (POL == P_AELL) {
        q.me = ae;
        return;
    }
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
    const QEnt *run = rec + ap;
    int done = 0;
    #pragma unroll 1
    while (done < len) {
        const int rem = len - done;
        if (rem <= 8) {
            #pragma unroll 1
            for (int j = 0; j < rem; ++j) delta_insert(P, w, q, run[done + j], base, n, gbp);
            break;
        }
        if (q.dn > 0) merge_delta(P, w, q, base, n, gbp);
        const int k = min(rem, w.dcap);
        #pragma unroll 1
        for (int j = lane; j < k; j += 32) w.dq[j] = run[done + k - 1 - j];  // descending
        __syncwarp();
        q.dn = k;
        done += k;
    }
}

template <int N>
struct Slots {
    static constexpr int value = N;
};

// body(Slots<N>, p) for the slots p + 32 j + lane, j < N, of every page in [0, end) (a half page when
// the caller knows, as a warp-uniform condition, that end <= kHalf).
template <class Body>
__device__ __forceinline__ void over_slots(bool half, int end, Body body) {
    if (half) {
        body(Slots<kHalf / 32>(), 0);
    } else {
        body(Slots<kPage / 32>(), 0);
        #pragma unroll 1
        for (int p = kPage; p < end; p += kPage) body(Slots<kPage / 32>(), p);
    }
}

// Passes (half pages) that over_slots makes over n slots.
__device__ __forceinline__ int slot_pages(int n) { return n <= kHalf ? 1 : 2 * ((n + kPage - 1) / kPage); }

// A job (e, b) leaves the set: W loses b + E at the endpoints E <= e (free slots compare greater).
__device__ __forceinline__ void subtract_job(const Ws &w, int end, int e, int b) {
    #pragma unroll 1
    for (int p = 0; p < end; p += kPage) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = p + 32 * j + lane_id();
            const int2 ew = w.EW[i];
            if (unsigned(ew.x) <= unsigned(e)) w.EW[i].y = minus(ew.y, b + ew.x);
        }
    }
}

// The same for two jobs in one pass (e = -2: none); W of free slots is not kept.
__device__ __forceinline__ void subtract_two(const Ws &w, int end, int e0, int b0, int e1, int b1) {
    const int most = max(e0, e1);
    #pragma unroll 1
    for (int p = 0; p < end; p += kPage) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = p + 32 * j + lane_id();
            int2 ew = w.EW[i];
            if (ew.x <= e0) ew.y = minus(ew.y, b0 + ew.x);
            if (ew.x <= e1) ew.y = minus(ew.y, b1 + ew.x);
            if (ew.x <= most) w.EW[i].y = ew.y;
        }
    }
}

template <int POL>
__device__ __forceinline__ void free_slot(const Ws &w, int i) {
    w.EW[i].x = -1;
    w.F[i] = -1;
    if (POL == P_AMIN) w.K[i] = UINT_MAX;
}

// Free the slots [from, from + kPage).
template <int POL>
__device__ __forceinline__ void free_page(const Ws &w, int from) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int i = from + 32 * j + lane_id();
        free_slot<POL>(w, i);
    }
}

// Move the live slots to the front, in place, and free the rest of their blocks.
template <int POL>
__device__ __forceinline__ void compact(const Ws &w, int &end) {
    const int lane = lane_id();
    const unsigned lt = (1u << lane) - 1u;
    int wpos = 0;
    #pragma unroll 1
    for (int b = 0; b < end; b += kHalf) {
        int2 e[2], c[2];
        int bb[2], f[2];
        unsigned k[2], m[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int i = b + 32 * j + lane;
            e[j] = w.EW[i];
            bb[j] = w.B[i];
            f[j] = w.F[i];
            c[j] = w.C[i];
            k[j] = POL == P_AMIN ? w.K[i] : 0u;
            m[j] = __ballot_sync(FULL, f[j] >= 0);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int d = wpos + __popc(m[j] & lt);
            if (f[j] >= 0) {
                w.EW[d] = e[j];
                w.B[d] = bb[j];
                w.F[d] = f[j];
                w.C[d] = c[j];
                if (POL == P_AMIN) w.K[d] = k[j];
            }
            wpos += __popc(m[j]);
        }
        __syncwarp();
    }
    #pragma unroll 1
    for (int i = wpos + lane; i < end; i += 32) {
        free_slot<POL>(w, i);
    }
    end = wpos;
    __syncwarp();
}

// Invariants of the simulation state between events (SIM_OPT_DEBUG_CHECKS; global-memory kernel
// only): the live slots number A and sum to need; nextF is their smallest F; W is the projected memory
// plus E at every endpoint not yet passed (with the pending updates); under A_max, H-SF and A_r no job runs
// past its projected last step; a witness not yet passed has V(ct) = cv; free slots are free; the delta
// queue is strictly descending (A_ell: the cached promotions ascending) and the cached head of the main
// array ascending.  Returns false on the first violation.
template <int POL>
__device__ bool state_ok(const Ws &w, const Queue &q, int A, int end, int t, int need, int nextF, int py, int pc,
                         int qy, int qc, int filled, int ct, int cv) {
    const int lane = lane_id();
    bool bad = false;
    unsigned fmin = UINT_MAX;
    int cnt = 0, sum = 0, vc = 0;
    #pragma unroll 1
    for (int i = lane; i < filled; i += 32) {
        const int4 h = make_int4(w.EW[i].x, w.EW[i].y, w.B[i], w.F[i]);
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
        if (h.x >= ct) vc += h.z + ct;
        int v = h.x;
        #pragma unroll 1
        for (int j = 0; j < end; ++j)
            if (w.EW[j].x >= h.x) v += w.B[j] + h.x;
        if (v != h.y + (h.x <= py ? h.x + pc : 0) - (h.x <= qy ? h.x + qc : 0)) bad = true;
    }
    if (int(__reduce_add_sync(FULL, unsigned(cnt))) != A || int(__reduce_add_sync(FULL, unsigned(sum))) != need) bad = true;
    #pragma unroll 1
    for (int i = lane; POL != P_AELL && i + 1 < q.dn; i += 32)
        if (!qless(w.dq[i + 1], w.dq[i])) bad = true;
    if (POL == P_AELL)
        #pragma unroll 1
        for (int i = q.dh - q.dcb + lane; i + 1 < q.dce - q.dcb; i += 32)
            if (!qless(w.dq[i], w.dq[i + 1])) bad = true;
    if (q.mcb >= 0)
        #pragma unroll 1
        for (int i = q.mh + lane; i + 1 < min(q.me, q.mcb + kMc); i += 32)
            if (i >= q.mcb && !qless(w.mc[i - q.mcb], w.mc[i + 1 - q.mcb])) bad = true;
    vc = int(__reduce_add_sync(FULL, unsigned(vc)));
    if (POL != P_AMIN && ct >= t && vc != cv) bad = true;
    fmin = __reduce_min_sync(FULL, fmin);
    if (A > 0 && fmin != unsigned(nextF)) bad = true;
    return __ballot_sync(FULL, bad) == 0;
}

// ---------------------------------------------------------------------------------------------
// One instance, simulated by one warp.  All lanes hold identical copies of the scalar state.
// INS: the instrumented copy, which also keeps the work counters of the per-step method and the
// batch-time sums; the plain copy has neither.
// All memory sums are at most M <= 2^26 where they are compared (V, need and a candidate's points
// belong to feasible schedules, a violated one exceeds M by one job's memory at most) and a projected
// step at most kMaxStep + 2^26, so 32 bits hold them and W <= 2^31 - 1 at the endpoints that are still to
// come (the sums that are not compared wrap: plus, minus).
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
    if (info.status == ST_OK && P.main_cap > 0 && int64_t(info.n) > P.main_cap) r.status = ST_INVAL;  // larger than the queue buffers
    if (r.status != ST_OK || info.n == 0) {
        if (lane == 0) P.res[inst] = r;
        return;
    }
    const int n = info.n;
    const int64_t base = info.base;
    const uint64_t tie_seed = (POL == P_AMIN && P.tie_seed) ? P.tie_seed[inst] : 0ull;
    const int M = int(P.M);

    Queue q;
    q.mq = P.rec + base;
    q.mh = q.me = 0;
    q.lim = n;
    q.mbuf = -1;
    q.dn = q.dh = q.dce = q.dcb = 0;
    q.mcb = -1;
    // global-memory bytes moved by the queue (instrumented kernel); the merge adds through gbp
    int64_t gbq = 0;
    int64_t *const gbp = INS ? &gbq : nullptr;
    // work counters of the paper's per-step method (Theorem complexity), accumulated per step in
    // closed form: S2 adds (the active set), S3 compare-exchanges of the overflow sort
    // (A ceil(log2 A)^2), S5 endpoint evaluations of a binary-search admission
    // ((A' + k) ceil(log2(Q + 1))); k_step / ev_step: admitted / removed at the current step
    int64_t cS2 = 0, cS3 = 0, cS5 = 0;
    int k_step = 0, ev_step = 0, ovf_t = -1;

    // Batch time (Section 6's linear batch-time model, coefficients given later): bx0..bx3 =
    // X0..X3, the sums over requests of the processed steps, batch sizes, step memories and
    // prefill tokens of the steps a_i .. C_i - 1 (an arrival at t subtracts the prefixes up to t,
    // a completion at C adds those up to C); bmem, bpf the prefixes of step memory and prefill
    // (steps and request steps have their own counters).
    const bool bt = INS && P.batch_time != nullptr;
    int64_t bx0 = 0, bx1 = 0, bx2 = 0, bx3 = 0, bmem = 0, bpf = 0;

    // A live jobs in the slots [0, end), the slots [0, filled) initialised; need: the memory of step
    // t; nextF, nextE: the smallest F and (A_ell) E; pending updates: W += E + pc at the endpoints
    // E <= py (the last job admitted) and W -= E + qc at those E <= qy (a job removed); -2: none
    int A = 0, end = 0, filled = kPage, need = 0;
    unsigned nextF = UINT_MAX, nextE = UINT_MAX;
    int py = -2, pc = 0, qy = -2, qc = 0;
    constexpr bool kSub = POL != P_HSF && POL != P_AR;
    free_page<POL>(w, 0);
    // steps processed = t - tb (tb moves with every idle gap); the instance stops at step tstop (the
    // step cap or kMaxStep); trare = min(tstop, next arrival)
    int t = P.rec_a[base], tb = t;
    const auto stop_at = [&]() { return int(min(int64_t(tb) + min(P.info[inst].cap, int64_t(INT_MAX)), int64_t(kMaxStep) + 1)); };
    int tstop = stop_at();
    // arrival steps of the records [apb, apb + 32), one per lane
    int ap = 0, apb = 0, next_a = t, trare = t;
    int pa = lane < n ? P.rec_a[base + lane] : INT_MAX;
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
    // the witness: the step ct that kept the last head that failed out for longest, and cv = V(ct), kept up
    // to date (see the top); no head whose own steps cover ct fits before bound()
    constexpr bool kWit = POL != P_AMIN;
    int ct = -1, cv = 0;
    const auto bound = [&]() {  // (the sum may wrap when there is no head: (1) fails then)
        if (!kWit) return 0;
        return unsigned(ct - t) < unsigned(hL) ? min(int(unsigned(cv - M + h.s + 1) + unsigned(ct)), ct + 1) : 0;
    };
    // what the next iteration has to look at first
    enum { HEAD = 1, NEXTF = 2, SLOTS = 4, IDLE = 8, MERGE = 16 };
    int attn = 0;

    const auto promotions = [&]() { return P.mainbuf + 2 * (P.main_cap > 0 ? warp_slot() * P.main_cap : base); };
    const auto load_head = [&]() { h = queue_head<POL>(w, q, hsrc, hL); };

    // The conditions of all branches below that the whole warp takes alike are results of warp reductions:
    // such a branch costs about 12 cycles, one on another value that the lanes happen to share about 45
    // (both measured), and one reduction (29) decides several of them.  Single-value stores are made by all
    // lanes alike, for the same reason.
    for (;;) {
        if (!SMEM && P.debug && attn == 0 &&
            !state_ok<POL>(w, q, A, end, t, need, int(nextF), py, pc, qy, qc, filled, ct, cv)) {
            status = ST_STATE;  // a consistency check of SIM_OPT_DEBUG_CHECKS failed
            break;
        }
        unsigned fl = 0;
        if (attn != 0 || t >= trare || (POL == P_AELL && unsigned(t) > nextE)) fl |= 1u;
        if (POL == P_AMIN && need > M) fl |= 2u;
        if (t >= fit_lb && need + h.s < M) fl |= 4u;
        if (unsigned(t) == nextF) fl |= 8u;
        if (end <= kHalf) fl |= 16u;
        fl = __reduce_or_sync(FULL, fl);
        const bool half = (fl & 16u) != 0;
        if (fl & 1u) {
            if (attn & SLOTS) {  // reclaim free slots, or take a new page
                if (end - A >= max(16, A >> 3) || (end >= w.ca && A < end)) {
                    compact<POL>(w, end);
                } else if (end >= w.ca) {
                    // a full set is no obstacle once every request has been admitted and none can return
                    if (POL == P_AMIN || POL == P_AELL || ndone + A < n) {
                        status = kStatusCapacity;
                        break;
                    }
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
                for (int i = lane; i < end; i += 32) f = min(f, unsigned(w.F[i]));
                nextF = __reduce_min_sync(FULL, f);
            }
            // (an admission that used up a cached run loaded the head from slots of the cache that hold no
            // entry of the queue: whatever they were, the head and its bound are new)
            const bool reload = (attn & HEAD) != 0;
            bool dirty = (attn & (HEAD | MERGE)) != 0;
            if (POL == P_AMIN && (attn & MERGE)) merge_delta(P, w, q, base, n, gbp);
            attn = 0;
            // ---- S1: arrivals with a <= t join R_t (a sorted run of the staged records)
            if (next_a <= t) {
                int ae;
                if (ap == 0 && P.rec_a[base + n - 1] <= t) {  // all at once
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
                        pa = apb + lane < n ? P.rec_a[base + apb + lane] : INT_MAX;
                    }
                }
                insert_run<POL>(P, w, q, base, n, ap, ae, gbq, gbp);
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
                if (ap < n) prefetch_l1(P.rec + base + min(ap + 8, n - 1));  // a line ahead of the next arrivals
            }
            // ---- A_ell: jobs that used up their estimate unfinished (E < t) leave the batch and
            // re-enter the queue at its end, in index order, with the estimate u
            if (POL == P_AELL && unsigned(t) > nextE) {
                if (t > kAellMaxStep) {
                    status = ST_STEPCAP;
                    break;
                }
                // their indices, in the space of K behind the cached lengths (or, for sets that do not
                // fit there, in the instance's second merge buffer), give each its place
                QEnt *pl = promotions() + q.dh + q.dn;
                int *ids = A <= w.ca - 2 * kMc
                               ? reinterpret_cast<int *>(w.K) + 2 * kMc
                               : reinterpret_cast<int *>(promotions() + (P.main_cap > 0 ? P.main_cap : int64_t(n)));
                int cnt = 0;
                #pragma unroll 1
                for (int b = 0; b < end; b += 32) {
                    const bool out = unsigned(w.EW[b + lane].x) < unsigned(t);
                    const unsigned m = __ballot_sync(FULL, out);
                    if (out) ids[cnt + __popc(m & ((1u << lane) - 1u))] = w.C[b + lane].y;
                    cnt += __popc(m);
                }
                __syncwarp();
                unsigned f = UINT_MAX, e1 = UINT_MAX;
                int sm = 0;
                #pragma unroll 1
                for (int b = 0; b < end; b += 32) {
                    const int i = b + lane;
                    const unsigned ei = unsigned(w.EW[i].x), fi = unsigned(w.F[i]);
                    if (ei >= unsigned(t)) {
                        f = min(f, fi);
                        e1 = min(e1, ei);
                    } else {
                        const int2 pi = w.C[i];
                        int place = 0;
                        #pragma unroll 1
                        for (int k = 0; k < cnt; ++k) place += ids[k] < pi.y ? 1 : 0;
                        QEnt e;
                        e.key = 2 * t + 1;
                        e.idx = pi.y;
                        e.s = w.B[i] + pi.x - 1;
                        e.o = int(fi) - pi.x + 1;
                        pl[place] = e;
                        sm += w.B[i] + t;
                        free_slot<POL>(w, i);
                    }
                }
                __syncwarp();
                __threadfence_block();
                need -= int(__reduce_add_sync(FULL, unsigned(sm)));
                A -= cnt;
                nev += cnt;
                q.dn += cnt;
                if (INS) {
                    ev_step += cnt;
                    gbq += int64_t(cnt) * int64_t(sizeof(QEnt));
                }
                nextF = __reduce_min_sync(FULL, f);
                nextE = __reduce_min_sync(FULL, e1);
                dirty = true;
                fit_lb = bound();
                if (end - A >= max(16, A >> 3) && slot_pages(end) > slot_pages(A)) attn |= SLOTS;
            }
            if (dirty) {
                const int hi = h.idx, hk = h.key;
                if (q.mh < q.me) main_cache_at_head<POL>(w, q, P.lu + base, gbq);
                if (POL == P_AELL && q.dn > 0) promo_cache_at_head(w, q, promotions(), P.lu + base, gbq);
                load_head();
                if (reload || h.idx != hi || h.key != hk) fit_lb = bound();
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
            if (INS && t != ovf_t) {  // (a full delta may interrupt the step's cancellations)
                const int lg = A > 1 ? 32 - __clz(A - 1) : 0;
                cS3 += int64_t(A) * lg * lg;
                ovf_t = t;
            }
            // Cancellation order (estimate, r, index), r the step's tie key (SplitMix64 of the seed
            // and t * 2^32 + index; under the index rule r = index, the same order).  A round
            // finds the smallest estimate and the first and last slot that hold it; only when these
            // differ does tie_position draw and compare the tied jobs' keys.  (On the 40960 x 2000
            // workload 1.3 % of the overflow steps have a tie at the smallest estimate.)
            #pragma unroll 1
            while (need > M && q.dn < w.dcap) {
                unsigned bk = UINT_MAX;
                int lo = 0, hi = 0;
                const int pq = max(py, qy);
                over_slots(half, end, [&](auto slots, int p) {
                    constexpr int N = decltype(slots)::value;
                    unsigned k[N], m = UINT_MAX;
                    int2 x[N];
#pragma unroll
                    for (int j = 0; j < N; ++j) {
                        k[j] = w.K[p + 32 * j + lane];
                        x[j] = w.EW[p + 32 * j + lane];
                    }
#pragma unroll
                    for (int j = 0; j < N; ++j) {
                        m = min(m, k[j]);
                        if (x[j].x <= py) x[j].y = plus(x[j].y, x[j].x + pc);
                        if (x[j].x <= qy) x[j].y = minus(x[j].y, x[j].x + qc);
                        if (x[j].x <= pq) w.EW[p + 32 * j + lane].y = x[j].y;
                    }
                    int first = 0, last = 0;
#pragma unroll
                    for (int j = 1; j < N; ++j) last = k[j] == m ? j : last;
#pragma unroll
                    for (int j = N - 1; j > 0; --j) first = k[j - 1] == m ? j - 1 : (j == N - 1 ? j : first);
                    if (m < bk) lo = p + 32 * first + lane;
                    if (m <= bk) hi = p + 32 * last + lane;
                    bk = min(bk, m);
                });
                const unsigned mk = __reduce_min_sync(FULL, bk);
                int pos = int(__reduce_min_sync(FULL, bk == mk ? unsigned(lo) : UINT_MAX));
                const int pos2 = int(__reduce_max_sync(FULL, bk == mk ? unsigned(hi) : 0u));
                if (mk == UINT_MAX) {  // no live job
                    status = ST_STATE;
                    break;
                }
                if (pos != pos2)
                    pos = tie_position(w.K, w.C, pos, pos2, mk, tie_base(tie_seed, t), P.evict_index == 0);
                const int ej = w.EW[pos].x, bj = w.B[pos], fj = w.F[pos];
                const int2 pi = w.C[pos];
                __syncwarp();
                free_slot<POL>(w, pos);
                __syncwarp();
                QEnt e;
                e.key = max(int(mk), t - pi.x);  // refined lower bound: max(estimate, tokens generated)
                e.idx = pi.y;
                e.s = bj + pi.x - 1;
                e.o = fj - pi.x + 1;
                need -= bj + t;
                --A;
                ++nev;
                if (INS) ++ev_step;
                if (unsigned(fj) == nextF) attn |= NEXTF;
                // the pass above applied the pending updates; this one waits for the next pass (endpoints
                // before t need none)
                py = -2;
                qy = ej < t ? -2 : ej;
                qc = bj;
                delta_put(w, q, e);
                if (qless(e, h)) {  // the head of R_t is the smaller of the two
                    h = e;
                    hL = e.key;
                    hsrc = 1;
                }
            }
            if (status != ST_OK) break;
            fit_lb = 0;
            if (A == 0) attn |= IDLE;
            if (q.dn == w.dcap) attn |= MERGE;
            if (end - A >= max(16, A >> 3) && slot_pages(end) > slot_pages(A)) attn |= SLOTS;
            // nothing else to look at: on to the head's test, or straight to the batch
            const unsigned st = __reduce_or_sync(FULL, (attn != 0 ? 1u : 0u) | (need + h.s < M ? 4u : 0u));
            if (st & 1u) continue;
            fl |= st;
        }
        // ---- S4/S5: admit the largest feasible prefix of R_t, one candidate at a time ((1) holds)
        if (fl & 4u) {
            // A candidate that fits is followed by the next one while nothing else needs a look; A_max,
            // whose admissions are mostly single, goes back to the top after each (with the inner loop
            // the load sweep takes 11 % longer, the online workloads 2-3 %; A_min takes 2-4 % less with it,
            // A_ell and H-SF 3 %).
            constexpr bool kBurst = POL != P_AMAX;
            const int A0 = A;
            unsigned st = fl & 8u;  // A_min: fl after the last admission, so that the batch can follow
            bool more;
            do {
                const int y = t + hL - 1;
                const int lim = M - h.s - 1 + t;
                int vy = 0, wm = INT_MIN;
                const int pq = kSub ? max(py, qy) : py;
                over_slots(half, end, [&](auto slots, int p) {
                    constexpr int N = decltype(slots)::value;
                    int2 x[N];
                    int bb[N];
#pragma unroll
                    for (int j = 0; j < N; ++j) {
                        x[j] = w.EW[p + 32 * j + lane];
                        bb[j] = w.B[p + 32 * j + lane];
                    }
#pragma unroll
                    for (int j = 0; j < N; ++j) {
                        if (x[j].x <= py) x[j].y = plus(x[j].y, x[j].x + pc);
                        if (kSub && x[j].x <= qy) x[j].y = minus(x[j].y, x[j].x + qc);
                        if (x[j].x <= pq) w.EW[p + 32 * j + lane].y = x[j].y;
                        if (x[j].x >= y) vy += bb[j] + y;
                        if (unsigned(x[j].x - t) < unsigned(hL)) wm = max(wm, x[j].y);
                    }
                });
                py = qy = -2;
                vy = int(__reduce_add_sync(FULL, unsigned(vy)));
                int d = max(wm, lim) - lim;      // > 0: (2) fails
                if (vy + h.s + hL > M) d = 1;    // (3) fails
                d = __reduce_max_sync(FULL, d);
                if (d > 0) {
                    // A second pass finds the first later step that could fit: W_i > lim violates (2) at
                    // endpoint i until the overlap has shrunk (W_i <= lim + tau - t) or the endpoint has
                    // passed, and (3) cannot hold before y has passed the next endpoint after it.  The witness
                    // is the endpoint that makes it so late, else y (all endpoints at one step have the same
                    // W; the endpoint with the largest W held heads out less: A_max +2 to +8 %; two witnesses
                    // cost more than they save, +3 %).  (In the same pass as the test it cost more than it
                    // saved, also where half of the tests fail.)
                    int r2 = 1, we = y, ww = vy + y;
                    unsigned em = UINT_MAX;
                    over_slots(half, end, [&](auto slots, int p) {
                        constexpr int N = decltype(slots)::value;
#pragma unroll
                        for (int j = 0; j < N; ++j) {
                            const int2 ew = w.EW[p + 32 * j + lane];
                            em = min(em, unsigned(ew.x - y));
                            const int r = unsigned(ew.x - t) < unsigned(hL) ? min(max(ew.y, lim) - lim, ew.x - t + 1) : 0;
                            if (kWit) we = r > r2 ? ew.x : we;
                            if (kWit) ww = r > r2 ? ew.y : ww;
                            r2 = max(r2, r);
                        }
                    });
                    em = __reduce_min_sync(FULL, em);
                    const int r1 = r2;
                    r2 = __reduce_max_sync(FULL, r2);
                    if (kWit) {
                        ct = __reduce_max_sync(FULL, r1 == r2 ? we : -1);
                        cv = __reduce_max_sync(FULL, r1 == r2 && we == ct ? ww : 0) - ct;
                    }
                    if (vy + h.s + hL > M) r2 = max(r2, int(em) + 1);
                    more = false;
                    // no fit before step t + r2, and none at all if (1) fails there
                    fit_lb = int64_t(need) + int64_t(A) * r2 + h.s + 1 > M ? INT_MAX : t + r2;
                } else {
                    // the pending update of its own admission adds the job's memory at y to its W
                    __syncwarp();
                    w.EW[end] = make_int2(y, vy + y);
                    w.B[end] = h.s - t + 1;
                    w.F[end] = t + h.o - 1;
                    w.C[end] = make_int2(t, h.idx);
                    if (POL == P_AMIN) w.K[end] = unsigned(h.key);
                    py = y;
                    pc = h.s - t + 1;
                    if (kWit) cv = plus(cv, y < ct ? 0 : pc + ct);
                    ++end;
                    ++A;
                    need += h.s + 1;
                    nextF = min(nextF, unsigned(t + h.o - 1));
                    if (POL == P_AELL) nextE = min(nextE, unsigned(y));
                    if (INS) ++k_step;
                    if (bt) bpf += h.s;  // prefill: the prompts of the admitted requests
                    q.dn -= hsrc;
                    if (POL == P_AELL) q.dh += hsrc;
                    q.mh += 1 - hsrc;
                    if (q.mh < q.me && unsigned(q.mh - q.mcb) >= unsigned(kMc)) attn |= HEAD;  // reloaded before use
                    if (POL == P_AELL && q.dn > 0 && q.dh >= q.dce) attn |= HEAD;
                    if (end == kHalf || (end & (kPage - 1)) == 0) attn |= SLOTS;
                    load_head();
                    fit_lb = bound();
                    __syncwarp();
                    more = false;
                    if (POL == P_AMIN) {
                        st = __reduce_or_sync(FULL, (attn != 0 || end == kHalf + 1 ? 1u : 0u) | (need + h.s < M ? 4u : 0u) |
                                                        (unsigned(t) == nextF ? 8u : 0u));
                        more = (st & 5u) == 4u;
                    } else if (kBurst) {
                        more = __reduce_max_sync(FULL, attn == 0 && t >= fit_lb && need + h.s < M && end != kHalf + 1);
                    }
                }
            } while (more);
            if (POL == P_AMIN) {
                if (st & 1u) continue;
                fl = st;
            } else if (A != A0) {
                continue;  // nextF may be this step now
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
            // A job that ends before its projected last step changes W: its slot keeps E (in place of
            // W) and B, and F = -2 - t tells it from the slots freed at other steps.
            constexpr bool kEarly = POL == P_AMAX || POL == P_AELL;
            int c = 0, sm = 0, ne = 0, ek = -1, bk = INT_MIN, dv = 0;
            unsigned f = UINT_MAX, e1 = UINT_MAX;
            over_slots(half, end, [&](auto slots, int p) {
                constexpr int N = decltype(slots)::value;
                int e[N], bb[N], fj[N];
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    fj[j] = w.F[p + 32 * j + lane];
                    bb[j] = w.B[p + 32 * j + lane];
                    if (kEarly) e[j] = w.EW[p + 32 * j + lane].x;
                }
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const int i = p + 32 * j + lane;
                    const bool done = fj[j] == t;
                    sm += done ? bb[j] + t : 0;
                    c += done ? 1 : 0;
                    f = min(f, done ? UINT_MAX : unsigned(fj[j]));
                    if (kEarly) {
                        const bool early = done && e[j] > t;
                        if (POL == P_AELL) e1 = min(e1, done ? UINT_MAX : unsigned(e[j]));
                        ne += early ? 1 : 0;
                        dv = plus(dv, early && e[j] >= ct ? bb[j] + ct : 0);
                        ek = early ? e[j] : ek;
                        bk = early ? bb[j] : bk;
                        if (done) w.EW[i] = make_int2(-1, e[j]);
                    } else if (done) {
                        w.EW[i].x = -1;
                    }
                    if (done) w.F[i] = kEarly ? -2 - t : -1;
                    if (POL == P_AMIN)
                        if (done) w.K[i] = UINT_MAX;
                    if (P.completion)
                        if (done) P.completion[base + w.C[i].y] = int64_t(t) + 1;
                }
            });
            c = int(__reduce_add_sync(FULL, unsigned(c)));
            sm = int(__reduce_add_sync(FULL, unsigned(sm)));
            nextF = __reduce_min_sync(FULL, f);
            if (POL == P_AELL) nextE = __reduce_min_sync(FULL, e1);
            if (kEarly) {
                // decided on reductions, as above; the first update is left pending if none is
                const int most = __reduce_max_sync(FULL, ne), tot = int(__reduce_add_sync(FULL, unsigned(ne)));
                const int e1st = __reduce_max_sync(FULL, ek), b1st = __reduce_max_sync(FULL, bk);
                const bool free_q = __reduce_max_sync(FULL, qy) < 0;
                cv = minus(cv, int(__reduce_add_sync(FULL, unsigned(dv))));
                if (tot == 1) {
                    if (free_q) {
                        qy = e1st;
                        qc = b1st;
                    } else {
                        subtract_job(w, end, e1st, b1st);
                    }
                } else if (most == 1) {  // one such job on each of several lanes
                    unsigned m = __ballot_sync(FULL, ne > 0);
                    int k = 0;
                    if (free_q) {
                        const int src = __ffs(m) - 1;
                        m &= m - 1;
                        qy = __shfl_sync(FULL, ek, src);
                        qc = __shfl_sync(FULL, bk, src);
                        k = 1;
                    }
                    #pragma unroll 1
                    for (; k < tot; k += 2) {
                        const int s0 = __ffs(m) - 1;
                        m &= m - 1;
                        const int s1 = __ffs(m) - 1;  // -1: no second one
                        m &= m - 1;
                        const int e2 = __shfl_sync(FULL, ek, s1 & 31);
                        subtract_two(w, end, __shfl_sync(FULL, ek, s0), __shfl_sync(FULL, bk, s0), s1 < 0 ? -2 : e2,
                                     __shfl_sync(FULL, bk, s1 & 31));
                    }
                } else if (most > 1) {  // several on one lane: found again by their mark
                    #pragma unroll 1
                    for (int b = 0; b < end; b += 32) {
                        const int xe = w.EW[b + lane].y, xb = w.B[b + lane];
                        unsigned m = __ballot_sync(FULL, w.F[b + lane] == -2 - t && xe > t);
                        #pragma unroll 1
                        while (m) {
                            const int src = __ffs(m) - 1;
                            m &= m - 1;
                            subtract_job(w, end, __shfl_sync(FULL, xe, src), __shfl_sync(FULL, xb, src));
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
            fit_lb = bound();
            if (A == 0) attn |= IDLE;
            if (end - A >= max(16, A >> 3) && slot_pages(end) > slot_pages(A)) attn |= SLOTS;
            if (ndone >= n) break;
        } else {
            // steps t .. tau-1 change nothing: no completion before nextF, no arrival before
            // trare, (A_min) no overflow, (A_ell) no promotion, and the head does not fit before fit_lb
            // (or at all, once (1) fails: need only grows while the set stays as it is)
            int tau = min(min(int(nextF), trare), need + h.s < M ? fit_lb : INT_MAX);
            if (POL == P_AELL) tau = min(tau, int(nextE) + 1);
            // the first step whose memory exceeds M
            if (POL == P_AMIN) tau = min(tau, t + quotient_lb(M - need, max(A, 1)) + 1);
            const int c = max(tau - t, 1);
            const int mem = need + A * (c - 1);  // of step tau - 1: feasible, so at most M
            if (mem > M) status = ST_STATE;      // an internal error, reported at the end
            peak = max(peak, mem);
            rsteps += int64_t(A) * c;
            if (bt)  // steps t .. t+c-1 have memory need + A (x - t)
                bmem += c * int64_t(need) + int64_t(A) * (int64_t(c) * (c - 1) / 2);
            if (INS) {
                const int Qa = (q.me - q.mh) + q.dn;
                cS2 += int64_t(A) * c - k_step + ev_step;
                cS5 += int64_t(A) * (32 - __clz(Qa + k_step)) + int64_t(A) * (c - 1) * (32 - __clz(Qa));
                k_step = ev_step = 0;
            }
            need = mem + A;
            t += c;
        }
    }
    if (lane == 0) {
        r.status = status;
        r.total_latency = sumC - P.info[inst].sum_a;
        r.makespan = makespan;
        r.peak_memory = peak;
        r.evictions = nev;
        r.steps = t - tb;
        r.request_steps = rsteps;
        P.res[inst] = r;
        if (status == kStatusCapacity && P.redo) P.redo[atomicAdd(P.redo_count, 1)] = inst;
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

// WIDE: up to 168 registers a thread (12 warps per SM), for launches whose time is one instance's serial
// chain; otherwise 128 (16 warps per SM), for launches with more instances than that.  On the
// 40960 x 2000 workload A_min takes 105 ms at 16 warps per SM and 131 at 12; the 256 x 10^4 online
// workload 26.2 ms with 168 registers and 28.5 with 128 (spills).
// CA: the slots per warp when fixed at compile time (the workspace arrays are then constant offsets from
// one address: 2-5 % on every policy), or 0 for P.ca (the global-memory kernel and other capacities).
template <int POL, bool SMEM, bool INS, bool WIDE, int CA>
__global__ void __launch_bounds__(WIDE ? 128 : 256, WIDE ? 3 : 2) k_run(RunParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = lane_id();
    const int ca = CA ? CA : P.ca;
    unsigned char *base;
    if (SMEM) base = smem_raw + size_t(threadIdx.x >> 5) * ws_bytes(ca, P.dcap);
    else base = P.gws + warp_slot() * P.gws_stride;
    Ws w = carve_ws(base, ca, P.dcap);
    const int n_work = P.n_work_dev ? *P.n_work_dev : P.n_work;
    // a warp's first instance is its slot's; the cursor hands out the rest, if there are any
    const int n_slots = int(gridDim.x * (blockDim.x >> 5));
    for (int k = int(warp_slot()); k < n_work;) {
        const int inst = P.work ? P.work[k] : k;
        sim_instance<POL, SMEM, INS>(P, w, inst);
        if (n_work <= n_slots) break;
        if (lane == 0) k = n_slots + atomicAdd(P.counter, 1);
        k = __shfl_sync(FULL, k, 0);
    }
}

using KernelFn = void (*)(RunParams);

template <int POL>
KernelFn pick(bool smem, bool ins, bool wide, int ca) {
    if (!smem) return ins ? k_run<POL, false, true, false, 0> : k_run<POL, false, false, false, 0>;
    if (wide && ca == kSmemCaDefault)
        return ins ? k_run<POL, true, true, true, kSmemCaDefault> : k_run<POL, true, false, true, kSmemCaDefault>;
    if (ins) return k_run<POL, true, true, false, 0>;
    if (!wide && ca == kDenseCa) return k_run<POL, true, false, false, kDenseCa>;
    return k_run<POL, true, false, false, 0>;
}

KernelFn run_fn(int policy, const RunParams &p, int warps_per_block) {
    const bool smem = p.use_smem != 0, ins = p.work_count != nullptr || p.batch_time != nullptr;
    const bool wide = p.wide != 0 && warps_per_block <= 4;
    switch (policy) {
        case P_AMAX: return pick<P_AMAX>(smem, ins, wide, p.ca);
        case P_AMIN: return pick<P_AMIN>(smem, ins, wide, p.ca);
        case P_HSF: return pick<P_HSF>(smem, ins, wide, p.ca);
        case P_AR: return pick<P_AR>(smem, ins, wide, p.ca);
        default: return pick<P_AELL>(smem, ins, wide, p.ca);
    }
}

}  // namespace

cudaError_t run_blocks_per_sm(int policy, const RunParams &p, int warps_per_block, size_t smem_bytes, int *blocks) {
    const KernelFn fn = run_fn(policy, p, warps_per_block);
    if (smem_bytes > 48 * 1024) {
        // to the device's limit, not to this launch's bytes: contexts with other launch shapes share the
        // kernel, also from other threads
        int dev = 0, most = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
    }
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, (const void *)fn, 32 * warps_per_block, smem_bytes);
}

cudaError_t launch_run(int policy, const RunParams &p, int blocks, int warps_per_block, size_t smem_bytes,
                       cudaStream_t st) {
    run_fn(policy, p, warps_per_block)<<<dim3(blocks), dim3(32 * warps_per_block), smem_bytes, st>>>(p);
    return cudaGetLastError();
}

}  // namespace simgb
