// sim.cu -- batched discrete-event simulation of request routing
// (ctr_simulate): Algorithm 1 of the paper inside the sec. III-D simulator,
// with the continuous decode batching of sec. VI, the marginal-cost score of
// sec. III-A and the sec. IV-C baselines.
//
// Layout: a row is (replica x cost-constant set x policy); a lane group of G
// lanes (a power of two >= the pool size: the next one in large launches, up to
// a whole warp in small ones, see sim_rows_per_warp) simulates one row, lane
// i < n_pre being prefill instance i and lane n_pre + d decode instance d, and
// a warp carries 32 / G rows side by side (the policies of one replica, which
// share arrival times).  Warps are persistent and pull row groups from an
// atomic counter in the workspace.  (Launches of very few rows take a block per
// row instead: sim_row_kernel.)  For every arrival k:
//   1. each decode lane takes its own instance's events up to t_k (the step
//      ends at which something changes, see Decode: completions, FCFS
//      admissions, step starts); each prefill lane retires prefills that
//      ended by t_k (or, with batched prefill, ends and starts its batches
//      first and hands the members' KV-ready times to the decode lanes);
//   2. every lane prices its instance for the row's policy, and two argmins
//      within the lane group (ties to the lowest lane) pick i_pre and i_dec;
//   3. the i_pre lane commits the prefill, broadcasts the KV-ready time when
//      it is known, and the i_dec lane queues the request.
// All time and cost arithmetic is int64 fixed point, so every decision is
// deterministic.  Instances never interact except through routing, so the
// per-lane event loops reproduce the global event order exactly (events at
// an arrival's own time are processed before it is routed).
//
// Per-lane structures live in the workspace slot of the warp, each lane's
// entries contiguous (a heap's top levels then share cache lines; the heaps
// are 4-ary, a node's four children two 16-byte words and a heap of n keys
// about log4 n levels deep, except with batched prefill: see heap_push_bin): a min-heap of
// pending KV-ready keys (t_ready << 23 | k) per decode lane (the prefill
// lanes use the same region as their in-flight ring of prefill end times,
// packed with the prompt length as end << 21 | p), a min-heap of active
// requests keyed by finishing step (finish << 23 | k), and a FIFO ring of
// KV-ready requests awaiting admission.  Heap tops are cached in registers,
// so a run of plain decode steps touches no memory.  The row checksum's
// routing terms are summed here; its first-token and completion terms are
// summed by hash_kernel from the outputs.
#include "ctr_internal.cuh"

namespace ctr {
namespace {

constexpr uint64_t kEmpty = ~0ull;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarpsPerBlock = 4;
constexpr int64_t kNever = INT64_MAX;
// an empty pending heap's top as a time: later than any event (the last one of a row that has not failed starts a step
// before 2^40, and a step lasts less than 2^38)
constexpr int64_t kIdle = (int64_t)(kEmpty >> kKeyBits);
constexpr int64_t kDrain = kIdle - 1;  // every event is at or before this
constexpr int64_t kBacklogClamp = int64_t(1) << 40;
constexpr uint64_t kPressureClamp = uint64_t(1) << 18;
constexpr int kRecipN = 1024;  // batch sizes with a tabulated reciprocal
constexpr int kRingPBits = 21;  // prefill ring entry: end << 21 | p (p <= 2^20)
constexpr int64_t kRingPMask = (int64_t(1) << kRingPBits) - 1;
constexpr int kRingKShift = 26;  // batched prefill ring entry: k << 26 | d << 21 | p

// ceil(2^64 / n) for n = 2..kRecipN, for the decode backlog's division by the
// batch size (built at compile time, read through the read-only path):
// floor(x / n) is the high word of x * v[n], exactly, while x < 2^54 (the
// product exceeds x / n by x e / (n 2^64) with e = v[n] n - 2^64 < n <= 2^10)
struct RecipTable {
    uint64_t v[kRecipN + 1];
};
constexpr RecipTable make_recip_table()
{
    RecipTable t{};
    for (int i = 2; i <= kRecipN; ++i) t.v[i] = ~0ull / (uint64_t)i + 1;
    return t;
}
__device__ const RecipTable kRecipTable = make_recip_table();

// floor(num / d) with r = floor((2^64 - 1) / d): the estimate is low by at most 2
__device__ __forceinline__ uint64_t div_recip(uint64_t num, uint64_t d, uint64_t recip)
{
    uint64_t q = __umul64hi(num, recip);
    uint64_t r = num - q * d;
    if (r >= d) {
        ++q;
        r -= d;
    }
    if (r >= d) ++q;
    return q;
}

// An estimate of x / d for 0 <= x < 2^31 and 1 <= d < 2^31 whose quotient is
// below 2^20, inv being recip_estimate(d): x and d rounded to fp32, a reciprocal
// good to a few 2^-24 and a product, so it is off by less than one unit either way.
__device__ __forceinline__ float recip_estimate(int32_t d)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__int2float_rn(d)));  // within 1 ulp
    return r;
}
__device__ __forceinline__ int32_t div_estimate(int32_t x, float inv)
{
    return __float2int_rz(__int2float_rn(x) * inv);
}

// floor(x / kv_div) for 0 <= x < 2^31, exact: kv_mul = ceil(2^(31 + s) / kv_div) with
// s = kv_shift the least with 2^s >= kv_div, so that x (kv_mul kv_div - 2^(31 + s)) < 2^31 2^s
__device__ __forceinline__ int32_t kv_term(int32_t x, const SimParams& P)
{
    return (int32_t)(__umulhi((uint32_t)x << 1, P.kv_mul) >> P.kv_shift);
}

// Entries per lane of a heap region holding up to cap keys.  The heaps are
// 4-ary: node j (0-based) sits at position j + 3, so its children 4j + 1 ..
// 4j + 4 sit at positions 4j + 4 .. 4j + 7, a 32-byte aligned block read as
// two 16-byte words; the region has cap + 3 entries rounded up to 4.
__host__ __device__ __forceinline__ int64_t heap_stride(int64_t cap) { return (cap + 6) & ~int64_t(3); }

constexpr int kHeapRoot = 3;

// min-heap of unique 64-bit keys; each lane's heap is contiguous
__device__ __forceinline__ void heap_push(uint64_t* h, int32_t& n, uint64_t& top, uint64_t key, int64_t lim,
                                          bool& bad)
{
    int i = kHeapRoot + n++;
    while (i > kHeapRoot) {
        const int parent = (i >> 2) + 2;
        const uint64_t pv = ck_ld(h, parent, lim, bad);
        if (pv < key) break;
        ck_st(h, i, lim, pv, bad);
        i = parent;
    }
    ck_st(h, i, lim, key, bad);
    if (i == kHeapRoot) top = key;
}

__device__ __forceinline__ void heap_pop(uint64_t* h, int32_t& n, uint64_t& top, int64_t lim, bool& bad)
{
    const int m = n--;  // the last key moves into the hole left at the root
    if (m == 1) {
        top = kEmpty;
        return;
    }
    const int lastp = kHeapRoot + m - 1;
    const uint64_t last = ck_ld(h, lastp, lim, bad);
    const int endp = lastp - 1;  // position of the last key that stays
    int i = kHeapRoot;
    for (;;) {
        const int c = (i - 2) << 2;  // first child
        if (c > endp) break;
        const ulonglong2 c01 = ck_ld2(h + c, 0, lim - c, bad);  // the block of four as two 16-byte words
        const ulonglong2 c23 = ck_ld2(h + c, 2, lim - c, bad);
        uint64_t cv = c01.x;
        int ci = c;
        if (c + 1 <= endp && c01.y < cv) {
            cv = c01.y;
            ci = c + 1;
        }
        if (c + 2 <= endp && c23.x < cv) {
            cv = c23.x;
            ci = c + 2;
        }
        if (c + 3 <= endp && c23.y < cv) {
            cv = c23.y;
            ci = c + 3;
        }
        if (last < cv) break;
        ck_st(h, i, lim, cv, bad);
        i = ci;
    }
    ck_st(h, i, lim, last, bad);
    top = ck_ld(h, kHeapRoot, lim, bad);
}

// Binary 1-based variants (children 2i and 2i + 1 in one 16-byte word), kept
// for batched prefill: its short-output document workload keeps decode batches
// small, where the extra compares of a 4-ary level cost more than the saved
// levels (4,096 x 2,000: 13.4 ms binary, 13.7 ms 4-ary; the replica sweep and
// the large pool were 2 % and 6 % faster 4-ary).  Same region stride.
__device__ __forceinline__ void heap_push_bin(uint64_t* h, int32_t& n, uint64_t& top, uint64_t key, int64_t lim,
                                              bool& bad)
{
    int i = ++n;
    while (i > 1) {
        const int parent = i >> 1;
        const uint64_t pv = ck_ld(h, parent, lim, bad);
        if (pv < key) break;
        ck_st(h, i, lim, pv, bad);
        i = parent;
    }
    ck_st(h, i, lim, key, bad);
    if (i == 1) top = key;
}

__device__ __forceinline__ void heap_pop_bin(uint64_t* h, int32_t& n, uint64_t& top, int64_t lim, bool& bad)
{
    const int m = n--;
    if (m == 1) {
        top = kEmpty;
        return;
    }
    const uint64_t last = ck_ld(h, m, lim, bad);
    const int sz = m - 1;
    int i = 1;
    for (;;) {
        const int c = 2 * i;
        if (c > sz) break;
        const ulonglong2 ch = ck_ld2(h, c, lim, bad);  // c even: a 16-byte word
        uint64_t cv = ch.x;
        int ci = c;
        if (c < sz && ch.y < cv) {
            cv = ch.y;
            ci = c + 1;
        }
        if (last < cv) break;
        ck_st(h, i, lim, cv, bad);
        i = ci;
    }
    ck_st(h, i, lim, last, bad);
    top = ck_ld(h, 1, lim, bad);
}

// 32-ary variants for a warp whose lanes all simulate the same instance (every
// lane calls with the same arguments and makes the same stores): a node's
// children, 32 consecutive entries, are one load of the warp and their minimum
// two redux.sync, so a level costs one child's worth of instructions instead of
// 32 and a heap of up to 33 keys has one.  Node j sits at position j + 3, its
// children at 32 j + 4 .. 32 j + 35: the 4-ary region's size serves.
// Nothing but a __syncwarp keeps the lanes of a warp in step, so what they share
// in memory follows one rule: a word has one lane that stores it, and a __syncwarp
// stands between that store and the other lanes' later loads, and between the
// other lanes' loads and a later store.  Every heap operation ends with one.
template <typename T, typename I>
__device__ __forceinline__ void lane_st(int lane, T* p, I i, int64_t lim, T v, bool& bad)
{
    if ((int)(threadIdx.x & 31) == lane) ck_st(p, i, lim, v, bad);
}

__device__ __forceinline__ void heap_push_warp(uint64_t* h, int32_t& n, uint64_t& top, uint64_t key, int64_t lim,
                                               bool& bad)
{
    int i = kHeapRoot + n++;
    while (i > kHeapRoot) {
        const int parent = ((i - 4) >> 5) + kHeapRoot;
        const uint64_t pv = parent == kHeapRoot ? top : ck_ld(h, parent, lim, bad);
        if (pv < key) break;
        __syncwarp();  // the parent has been read; it is stored to next
        lane_st(0, h, i, lim, pv, bad);
        i = parent;
    }
    lane_st(0, h, i, lim, key, bad);
    __syncwarp();
    if (i == kHeapRoot) top = key;
}

__device__ __forceinline__ void heap_pop_warp(uint64_t* h, int32_t& n, uint64_t& top, int64_t lim, bool& bad)
{
    const int m = n--;
    if (m == 1) {
        top = kEmpty;
        return;
    }
    const int lane = threadIdx.x & 31;
    const int lastp = kHeapRoot + m - 1;
    const uint64_t last = ck_ld(h, lastp, lim, bad);
    int i = kHeapRoot;
    int reader = 0;         // the only lane that has read position i
    uint64_t first = last;  // what comes to the root
    for (;;) {
        const int c = 32 * (i - kHeapRoot) + 4;  // first child
        if (c >= lastp) break;
        const uint64_t v = c + lane < lastp ? ck_ld(h, c + lane, lim, bad) : kEmpty;
        const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
        const uint32_t mhi = __reduce_min_sync(kFull, hi);
        const uint32_t mlo = __reduce_min_sync(kFull, hi == mhi ? lo : 0xffffffffu);
        const uint64_t cv = ((uint64_t)mhi << 32) | mlo;
        if (last < cv) break;
        if (i == kHeapRoot) first = cv;
        lane_st(reader, h, i, lim, cv, bad);
        reader = __ffs(__ballot_sync(kFull, v == cv)) - 1;
        i = c + reader;
    }
    lane_st(reader, h, i, lim, last, bad);
    __syncwarp();
    top = first;
}

// the heap operations of a kernel instantiation: binary with batched prefill, 32-ary where a whole warp
// simulates one instance, else 4-ary
template <int kArity>
__device__ __forceinline__ void hpush(uint64_t* h, int32_t& n, uint64_t& top, uint64_t key, int64_t lim, bool& bad)
{
    if constexpr (kArity == 2)
        heap_push_bin(h, n, top, key, lim, bad);
    else if constexpr (kArity == 32)
        heap_push_warp(h, n, top, key, lim, bad);
    else
        heap_push(h, n, top, key, lim, bad);
}
template <int kArity>
__device__ __forceinline__ void hpop(uint64_t* h, int32_t& n, uint64_t& top, int64_t lim, bool& bad)
{
    if constexpr (kArity == 2)
        heap_pop_bin(h, n, top, lim, bad);
    else if constexpr (kArity == 32)
        heap_pop_warp(h, n, top, lim, bad);
    else
        heap_pop(h, n, top, lim, bad);
}

// Accesses to an instance's other structures and to its requests' entries: plain ones of the lane that simulates it,
// or those of a warp that does together.  own_ld: its lanes have all read.
template <int kArity, typename T, typename I>
__device__ __forceinline__ T own_ld(const T* p, I i, int64_t lim, bool& bad)
{
    const T v = ck_ld(p, i, lim, bad);
    if constexpr (kArity == 32) __syncwarp();
    return v;
}
template <int kArity, typename T, typename I>
__device__ __forceinline__ void own_st(T* p, I i, int64_t lim, T v, bool& bad)
{
    if constexpr (kArity == 32)
        lane_st(0, p, i, lim, v, bad);
    else
        ck_st(p, i, lim, v, bad);
}
// what own_st has stored may be read from here on
template <int kArity>
__device__ __forceinline__ void own_stored()
{
    if constexpr (kArity == 32) __syncwarp();
}

// argmin over the lanes of 64-bit values (ties -> lowest lane)
__device__ __forceinline__ int warp_argmin(uint64_t v)
{
    const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
    const uint32_t mhi = __reduce_min_sync(kFull, hi);
    const uint32_t mlo = __reduce_min_sync(kFull, hi == mhi ? lo : 0xffffffffu);
    const uint32_t ball = __ballot_sync(kFull, hi == mhi && lo == mlo);
    return __ffs(ball) - 1;
}

// The row's slice of the trace and of the outputs: four pointers where
// registers allow (kPtr: 128 of them), else two offsets added on each access
// (pointers in every instantiation: single replica 4.72 -> 4.65 ms, but the
// replica sweep at 72 registers 137.0 -> 137.8).
template <bool kPtr, int kArity>
struct RowView {
    const SimParams& P;
    const int32_t *p_ = nullptr, *o_ = nullptr;
    int64_t *tf_ = nullptr, *td_ = nullptr;
    int64_t tb, ob;
    __device__ __forceinline__ RowView(const SimParams& P, int64_t tb, int64_t ob) : P(P), tb(tb), ob(ob)
    {
        if (kPtr) {
            p_ = P.trace.prompt_len + tb;
            o_ = P.trace.true_out + tb;
            tf_ = P.t_first + ob;
            td_ = P.t_done + ob;
        }
    }
    __device__ __forceinline__ int32_t p(uint32_t k, bool& bad) const
    {
        return kPtr ? ck_ldg(p_, k, P.n_req, bad) : ck_ldg(P.trace.prompt_len, tb + k, P.trace_len, bad);
    }
    __device__ __forceinline__ int32_t o(uint32_t k, bool& bad) const
    {
        return kPtr ? ck_ldg(o_, k, P.n_req, bad) : ck_ldg(P.trace.true_out, tb + k, P.trace_len, bad);
    }
    __device__ __forceinline__ int32_t o_hat(uint32_t k, bool& bad) const
    {
        return ck_ldg(P.trace.pred_out, tb + k, P.trace_len, bad);
    }
    __device__ __forceinline__ int64_t first(uint32_t k, bool& bad) const
    {
        return kPtr ? own_ld<kArity>(tf_, k, P.n_req, bad) : own_ld<kArity>(P.t_first, ob + k, P.out_len, bad);
    }
    __device__ __forceinline__ void set_first(uint32_t k, int64_t v, bool& bad) const
    {
        kPtr ? own_st<kArity>(tf_, k, P.n_req, v, bad) : own_st<kArity>(P.t_first, ob + k, P.out_len, v, bad);
    }
    __device__ __forceinline__ void set_done(uint32_t k, int64_t v, bool& bad) const
    {
        kPtr ? own_st<kArity>(td_, k, P.n_req, v, bad) : own_st<kArity>(P.t_done, ob + k, P.out_len, v, bad);
    }
};

// A decode lane's state.  Its next event is the end of a step at which
// something can change (a completion, an admission, the floor(KV / kv_div) term
// of the step time) or fail (the FIFO, the step budget), and the steps before it
// are a run of equal ones, left as they are until the event: the running step ends at step_end, `run` more of
// `step` us follow, and the event is at step_end + run * step.  An idle lane
// (n_act = 0) has run = 0 and step_end the time of its next KV-ready request
// (kIdle without one).  run * step stays below 2^31, so a time inside the run
// is a 32-bit offset from step_end.  step_idx, kv_res and a true-backlog sum
// are the values before the step that ends at step_end.
// `sum` is the one in-flight sum the row's policy reads: the true remaining
// output tokens R for the learned router on the true backlog, the predicted
// lengths o_hat for the length heuristic and the proxy's ledger
// (sum_is_o_hat), nothing for the others.
struct Decode {
    int64_t step_end, sum;
    int32_t run, step;
    float inv_step;          // about 1 / step (see div_estimate)
    int32_t step_idx;        // steps ended; the step budget keeps it and every completion step below 2^31
    int32_t kv_res, kv_rsv;  // resident <= reserved <= C < 2^31 tokens
    uint64_t pend_top, act_top;
    int32_t n_act, pend_n, w_head, w_n;  // n_act is also the active heap's size
    int32_t q;  // batched prefill: requests routed here and not completed (else the sum of the three counts, see in_flight)
};

// requests routed to a decode lane and not completed
template <bool kBat>
__device__ __forceinline__ int32_t in_flight(const Decode& s)
{
    return kBat ? s.q : s.n_act + s.pend_n + s.w_n;
}

__device__ __forceinline__ int64_t next_event(const Decode& s) { return s.step_end + (int64_t)s.run * s.step; }

// Steps of the run that have ended by t, for t before the next event: exact
// (the quotient is below run <= 2^20).
__device__ __forceinline__ int32_t ends_by(const Decode& s, int64_t t)
{
    const int32_t dt = (int32_t)(t - s.step_end);  // what follows from a time before step_end is not kept
    int32_t q = div_estimate(dt, s.inv_step);
    const int32_t r = dt - q * s.step;
    q += (r >= s.step) - (r < 0);
    return (s.n_act == 0) | (t < s.step_end) ? 0 : q + 1;
}

// A request becomes KV-ready at tp: the event moves up to the first step end at
// or after tp (or, where the estimate is one low, to the end before it, an event
// at which nothing changes).
__device__ __forceinline__ void cut_run(Decode& s, int64_t tp, bool when)
{
    const int64_t d = tp - s.step_end;
    if (when & (d < (int64_t)s.run * s.step)) {
        const int32_t rel = d > 0 ? (int32_t)d : 0;
        int32_t q = div_estimate(rel, s.inv_step);
        q += rel > q * s.step;
        s.run = q;
    }
}

// A new key of the pending heap (ready at key >> 23).  While requests wait for
// admission (w_n > 0) the next event does not depend on it -- either the head
// waits for a completion, or an event no later than this one is set already --
// unless it could overflow the FIFO, which counts from the step end at which it does.
template <int kArity>
__device__ __forceinline__ void push_pending(Decode& s, uint64_t* pend, uint64_t key, const SimParams& P, int64_t lim,
                                             bool& bad)
{
    hpush<kArity>(pend, s.pend_n, s.pend_top, key, lim, bad);
    const int64_t tp = (int64_t)(key >> kKeyBits);
    s.step_end = (s.n_act == 0) & (tp < s.step_end) ? tp : s.step_end;  // an idle instance's next event
    bool cut = s.w_n == 0;
    if (!cut) cut = s.w_n + s.pend_n > P.cap_wait;
    cut_run(s, tp, cut);
}

// Move every pending request whose KV is ready by t into the waiting FIFO, in
// (time, index) order; room is what the FIFO can still take.
template <int kArity>
__device__ __forceinline__ int flush_ready(Decode& s, int64_t t, int32_t room, const SimParams& P, uint64_t* pend,
                                           uint32_t* wait, bool& bad)
{
    const uint64_t by = (uint64_t)(t + 1) << kKeyBits;  // keys of requests KV-ready by t are below (kEmpty is not)
    while (s.pend_top < by) {
        const uint32_t k = (uint32_t)(s.pend_top & kKeyMask);
        hpop<kArity>(pend, s.pend_n, s.pend_top, heap_stride(P.cap_pr), bad);
        if (--room < 0) return CTR_EOVERFLOW;
        int pos = s.w_head + s.w_n;
        if (pos >= P.cap_wait) pos -= P.cap_wait;
        own_st<kArity>(wait, pos, P.cap_wait, k, bad);
        own_stored<kArity>();
        s.w_n += 1;
    }
    return CTR_OK;
}

// One event of a decode instance (at next_event): the run's steps end, requests
// that finish with the last one complete, those KV-ready by then are admitted
// strictly FCFS while the reservation fits, the next step starts and the next
// event is set.  The pending heap may hold requests already KV-ready (a
// KV-ready event while a step runs only matters at the step's end; while the
// FIFO's head waits for room, at the next completion); it has room for
// cap_pend + cap_wait + 1 entries, so a full heap means the waiting FIFO has
// overflowed.
template <int kArity, bool kPtr>
__device__ __forceinline__ int decode_event(Decode& s, int64_t tev, const SimParams& P, uint64_t* pend, uint64_t* act,
                                            uint32_t* wait, const RowView<kPtr, kArity>& V, bool sum_is_o_hat, bool& bad)
{
    {  // (1) run + 1 steps end (none of an idle instance): as many tokens for every active request
        const int32_t ends = s.n_act > 0 ? s.run + 1 : 0;
        const int32_t tokens = ends * s.n_act;  // within the reservation
        s.step_idx += ends;
        s.kv_res += tokens;
        if (!sum_is_o_hat) s.sum -= tokens;
    }
    while ((int32_t)(s.act_top >> kKeyBits) == s.step_idx) {  // never with an empty heap: its top is all ones
        const uint32_t k = (uint32_t)(s.act_top & kKeyMask);
        const int32_t pk = V.p(k, bad), ok = V.o(k, bad);
        int32_t gone = 0;
        if (sum_is_o_hat) gone = V.o_hat(k, bad);
        s.sum -= gone;
        V.set_done(k, tev, bad);
        hpop<kArity>(act, s.n_act, s.act_top, heap_stride(P.cap_act), bad);
        if constexpr (kArity == 2) s.q -= 1;
        s.kv_res -= pk + ok;
        s.kv_rsv -= pk + ok;
    }
    // (2) admission in FCFS order: the waiting FIFO, then the requests KV-ready by now in (time, index)
    // order, which join the FIFO once its head does not fit.  Before any admission the FIFO holds all of
    // them, so its room counts those admitted from the pending heap too.
    const uint64_t by = (uint64_t)(tev + 1) << kKeyBits;  // as in flush_ready
    int32_t room = P.cap_wait - s.w_n;
    int32_t admitted = 0;
    bool hold = false;  // the FIFO's head waits, and no further request can overflow the FIFO (see push_pending)
    uint32_t last = 0;  // the request admitted last; the others are chained through their t_first entries
    for (;;) {
        const bool fifo = s.w_n > 0;
        if (!fifo && s.pend_top >= by) break;
        const uint32_t k = fifo ? own_ld<kArity>(wait, s.w_head, P.cap_wait, bad) : (uint32_t)(s.pend_top & kKeyMask);
        const int32_t pk = V.p(k, bad), ok = V.o(k, bad);
        const bool fits = (uint32_t)s.kv_rsv + (uint32_t)(pk + ok) <= (uint32_t)P.kv_cap;  // < 2^31 + 2^21
        if (!fits || s.n_act == P.cap_act) {
            if (fits) return CTR_EOVERFLOW;
            const int rc = flush_ready<kArity>(s, tev, room, P, pend, wait, bad);
            if (rc != CTR_OK) return rc;
            hold = s.w_n + s.pend_n <= P.cap_wait;
            break;
        }
        if (fifo) {
            s.w_n -= 1;
            s.w_head = s.w_n == 0 || s.w_head + 1 == P.cap_wait ? 0 : s.w_head + 1;  // an empty ring restarts at 0
        } else {
            hpop<kArity>(pend, s.pend_n, s.pend_top, heap_stride(P.cap_pr), bad);
            --room;
        }
        s.kv_rsv += pk + ok;
        s.kv_res += pk;
        hpush<kArity>(act, s.n_act, s.act_top, ((uint64_t)(uint32_t)(s.step_idx + ok) << kKeyBits) | k,
                      heap_stride(P.cap_act), bad);
        if (admitted > 0) V.set_first(k, (int64_t)last, bad);
        last = k;
        admitted += 1;
    }
    // (3) the next step and the next event
    // the FIFO's room, the steps started on this instance, the time (its limit's low word is 0): a step that ended too
    // late was started within the budget
    if (room < 0 || s.step_idx + (s.n_act > 0) > (int32_t)P.max_steps ||
        (int32_t)(tev >> 32) >= (int32_t)(kTimeLimit >> 32))
        return room < 0 || (int32_t)(tev >> 32) >= (int32_t)(kTimeLimit >> 32) ? CTR_EOVERFLOW : CTR_ETIMEOUT;
    const int64_t tp = (int64_t)(s.pend_top >> kKeyBits);  // kIdle when empty
    const int32_t n = s.n_act;
    const bool idle = n == 0;  // then what follows computes nothing that is kept
    // dec_base <= 2^24 and a KV term below 2^31 add up in 32 bits
    const int64_t end = tev + (int64_t)((uint64_t)(uint32_t)P.dec_seq * (uint32_t)n) +
                        (int64_t)(uint64_t)((uint32_t)P.dec_base + (uint32_t)kv_term(s.kv_res, P));
    s.step_end = idle ? tp : end;
    if (kArity == 32 && admitted > 1) own_stored<kArity>();
    for (; admitted > 1; --admitted) {  // first token at the end of this step
        const uint32_t prev = (uint32_t)V.first(last, bad);
        V.set_first(last, s.step_end, bad);
        last = prev;
    }
    if (admitted == 1) V.set_first(last, s.step_end, bad);
    // after j of the run's ends the KV term is that of kv_res + j n, and it stays q1 while j n <= room1
    // (q1 + 1 <= 2^31 and kv_div <= 2^31; the sum is below 2^32)
    const int32_t q1 = kv_term(s.kv_res + n, P);
    const uint32_t room1 = (uint32_t)(q1 + 1) * (uint32_t)P.kv_div - 1u - (uint32_t)s.kv_res;
    // plain ends before the next completion or the end of the step budget, <= 2^20
    const int32_t fin = (int32_t)(s.act_top >> kKeyBits);
    int32_t m = (fin < (int32_t)P.max_steps ? fin : (int32_t)P.max_steps) - s.step_idx - 1;
    // the steps before the term changes, room1 / n (or one less): the estimate is within one where it is below m
    int32_t before = __float2int_rz(__uint2float_rn(room1) * recip_estimate(n));
    before -= (uint32_t)before * (uint32_t)n > room1;  // room1 < kv_div + n, so a product that matters fits
    m = before < m ? before : m;
    s.step = (int32_t)P.dec_base + (int32_t)P.dec_seq * n + q1;  // run_max = 0 where a step could reach 2^31 us
    s.inv_step = recip_estimate(s.step);
    s.run = idle ? 0 : m < P.run_max ? m : P.run_max;
    cut_run(s, tp, !hold);
    return CTR_OK;
}

// Advance one decode instance through every event at times <= T.  kSnap: when
// tsnap >= 0, also record in kv_snap the resident KV as it is after every event
// at times <= tsnap (an occupancy poll; tsnap <= T).
template <bool kSnap, int kArity, bool kPtr>
__device__ __forceinline__ int decode_advance(Decode& s, int64_t T, const SimParams& P, uint64_t* pend, uint64_t* act,
                                              uint32_t* wait, const RowView<kPtr, kArity>& V, int64_t tsnap, int64_t& kv_snap,
                                              bool sum_is_o_hat, bool& bad)
{
    for (;;) {
        const int64_t tev = next_event(s);
        if constexpr (kSnap) {
            if (tsnap >= 0 && tev > tsnap) {
                kv_snap = s.kv_res + ends_by(s, tsnap) * s.n_act;
                tsnap = -1;
            }
        }
        if (tev > T) return CTR_OK;
        const int rc = decode_event<kArity>(s, tev, P, pend, act, wait, V, sum_is_o_hat, bad);
        if (rc != CTR_OK) return rc;
    }
}

// A prefill lane keeps its state in decode fields it does not use (fewer live
// registers): step_end the end of its last prefill (of the running batch, when
// batched), act_top the ring's front entry (end << 21 | p, read while it holds
// any), sum the prompt tokens of the prefills in the ring, w_head / w_n the ring.
// Retire the serial prefills that ended by T.
template <bool kSig, int kArity>
__device__ __forceinline__ void retire_prefills(Decode& s, int64_t T, const SimParams& P, const int64_t* ring, bool& bad)
{
    const int64_t thr = ((T + 1) << kRingPBits) - 1;  // entries whose prefill ended by T
    while (s.w_n > 0 && s.act_top <= (uint64_t)thr) {
        if constexpr (kSig) s.sum -= s.act_top & kRingPMask;
        s.w_head = s.w_head + 1 == P.cap_ring ? 0 : s.w_head + 1;
        s.w_n -= 1;
        s.act_top = s.w_n > 0 ? (uint64_t)own_ld<kArity>(ring, s.w_head, P.cap_ring, bad) : (uint64_t)kNever;
    }
    if (s.w_n == 0) s.w_head = 0;
}

// Batched prefill: the running batch of run_n members (run_p tokens, ending at
// step_end); the queue behind it, cut FCFS into budget-limited batches, forms
// q_batches, the last of q_tail tokens.
struct BatchQueue {
    int32_t run_n, q_batches;
    int64_t run_p, q_tail;
};

// One request as the router sees it.
struct Request {
    int64_t k, T;
    uint32_t p, o_hat;
    int cls;
};

// The cost of instance `me` (of its pool) for a request under the row's policy
// (not round-robin), and kEmpty where the policy does not consider it.
template <bool kSig, bool kBat>
__device__ __forceinline__ uint64_t instance_cost(const SimParams& P, const ConstsDev& cc, int pol, bool is_pre, int me,
                                                  const Decode& s, const BatchQueue& bq, int64_t kv_seen,
                                                  const Request& rq)
{
    if (pol != CTR_POLICY_LEARNED && pol != CTR_POLICY_LEARNED_P2) {
        if (is_pre) return (uint64_t)s.w_n;
        return pol == CTR_POLICY_LENGTH_HEURISTIC && (int32_t)rq.o_hat >= P.heur_thresh ? (uint64_t)s.sum
                                                                                        : (uint64_t)in_flight<kBat>(s);
    }
    // backlog and own work of the instance, then the cost both kinds share
    // (feature ablation, sec. V-F, is in the constants: see ConstsDev)
    const int64_t T = rq.T;
    uint64_t b = 0, work;
    if (is_pre) {
        const int64_t rest = s.step_end > T ? s.step_end - T : 0;
        if (kSig && cc.proxy)  // the ledger: tau_pre0 + tau_pre p per prefill not yet ended
            b = (uint64_t)cc.tau_pre0 * (uint32_t)s.w_n + (uint64_t)cc.tau_pre * (uint64_t)s.sum;
        else if (kBat && P.pre_batch > 0)  // the running batch's rest, then the queue's batches
            b = (uint64_t)((bq.run_n > 0 ? rest : 0) + P.pre_base * (int64_t)bq.q_batches + P.pre_tok * (s.sum - bq.run_p));
        else
            b = (uint64_t)rest;
        work = (uint64_t)cc.tau_pre * rq.p + cc.tau_pre0;
    } else {
        const uint32_t oh_f = rq.o_hat & cc.oh_mask;
        int32_t kv = (int32_t)kv_seen;
        const bool polled = kSig && cc.poll_us > 0;
        if (!(kSig && cc.proxy && polled)) {
            const int32_t tokens = ends_by(s, T) * s.n_act;  // of the run's steps that have ended
            const int32_t kv_live = s.kv_res + tokens;
            if (!polled) kv = kv_live;
            if (!(kSig && cc.proxy)) {
                const uint64_t R = (uint64_t)(s.sum - tokens);
                const uint64_t step = (uint64_t)(P.dec_base + (int64_t)(int32_t)P.dec_seq * s.n_act + kv_term(kv_live, P));
                const uint32_t nd = (uint32_t)(s.n_act > 1 ? s.n_act : 1);
                if (((R | (step << 10)) >> 32) == 0 && nd <= (uint32_t)kRecipN) {
                    const uint64_t lo = (uint64_t)(uint32_t)R * (uint32_t)step;  // < 2^54
                    b = nd > 1 ? __umul64hi(lo, __ldg(&kRecipTable.v[nd])) : lo;
                } else {
                    const uint64_t lo = R * step;
                    b = __umul64hi(R, step) != 0 || lo >= (1ull << 62) ? (uint64_t)kBacklogClamp : lo / nd;
                }
            }
        }
        if (kSig && cc.proxy)  // the ledger: tau_dec o_hat per request routed here and not done
            b = (uint64_t)cc.ledger_tau * (uint64_t)s.sum;
        const uint32_t after = (uint32_t)kv + rq.p + oh_f;  // < 2^31 + 2^20 + 2^17
        uint64_t press;
        if (P.kv_cap_magic != 0) {
            const uint64_t lo = (uint64_t)after * (uint32_t)P.kv_cap_magic;
            press = ((uint64_t)after * (uint32_t)(P.kv_cap_magic >> 32) + (lo >> 32)) >> 16;
        } else {
            press = ((uint64_t)after << 16) / (uint64_t)P.kv_cap;
        }
        const uint32_t p18 = (press < kPressureClamp ? (uint32_t)press : (uint32_t)kPressureClamp) & cc.press_mask;
        const uint64_t own = (uint64_t)oh_f * cc.tau_dec;  // < 2^37
        work = own + ((((own * p18) >> 16) * cc.rho) >> 8);
    }
    if (b > (uint64_t)kBacklogClamp) b = (uint64_t)kBacklogClamp;
    const uint32_t queue = (uint32_t)(is_pre ? s.w_n : in_flight<kBat>(s));
    const uint64_t cost = (b * cc.w_b + work * cc.w_s) * cc.sigma[rq.cls] + cc.w_q16 * queue;
    if (pol == CTR_POLICY_LEARNED_P2) {
        // power of two choices: only two sampled candidates per pool are priced
        const Philox4 u = philox4x32_10((uint32_t)rq.k, (uint32_t)T, (uint32_t)((uint64_t)T >> 32), 0x5032u, 0x243F6A88u,
                                        0x85A308D3u);
        const uint32_t n_pool = is_pre ? (uint32_t)P.n_pre : (uint32_t)P.n_dec;
        const uint32_t a0 = is_pre ? u.v[2] : u.v[0], a1 = is_pre ? u.v[3] : u.v[1];
        const uint32_t c0 = (uint32_t)(((uint64_t)a0 * n_pool) >> 32);
        uint32_t c1 = c0;
        if (n_pool > 1) {
            c1 = c0 + 1 + (uint32_t)(((uint64_t)a1 * (n_pool - 1)) >> 32);
            if (c1 >= n_pool) c1 -= n_pool;
        }
        if ((uint32_t)me != c0 && (uint32_t)me != c1) return kEmpty;
    }
    return cost;
}

// the end of a serial prefill of p tokens that reaches, at T, an instance busy until `busy`
__device__ __forceinline__ int64_t prefill_end(const SimParams& P, int64_t busy, int64_t T, uint32_t p)
{
    const int64_t start = busy > T ? busy : T;
    return start + P.pre_base + (int64_t)(int32_t)P.pre_tok * (int32_t)p;
}

// Commit a serial prefill ending at `end` to its lane (the caller has checked the time limit).
template <bool kSig, int kArity>
__device__ __forceinline__ int push_prefill(Decode& s, int64_t end, uint32_t p, const SimParams& P, int64_t* ring,
                                            bool& bad)
{
    if (s.w_n == P.cap_ring) return CTR_EOVERFLOW;
    s.step_end = end;
    int pos = s.w_head + s.w_n;
    if (pos >= P.cap_ring) pos -= P.cap_ring;
    const int64_t e = (end << kRingPBits) | p;
    own_st<kArity>(ring, pos, P.cap_ring, e, bad);
    own_stored<kArity>();
    if (s.w_n == 0) s.act_top = (uint64_t)e;
    s.w_n += 1;
    if constexpr (kSig) s.sum += p;
    return CTR_OK;
}

// Commit a request to its decode lane at T: KV-ready at `ready` (-1: not known yet), `weight` its share of the
// lane's in-flight sum.
template <int kArity>
__device__ __forceinline__ int queue_decode(Decode& s, int64_t T, int64_t k, int64_t ready, int64_t weight,
                                            const SimParams& P, uint64_t* pend, uint32_t* wait, bool& bad)
{
    // requests routed here whose KV is not ready yet, exactly: first move
    // those already ready (kept in the heap until the step end) if it matters
    constexpr bool kBat = kArity == 2;
    if (in_flight<kBat>(s) - s.w_n - s.n_act >= P.cap_pend) {
        const int rc = flush_ready<kArity>(s, T, P.cap_wait - s.w_n, P, pend, wait, bad);
        if (rc != CTR_OK) return rc;
        if (in_flight<kBat>(s) - s.w_n - s.n_act == P.cap_pend) return CTR_EOVERFLOW;
    }
    if (kBat && ready >= 0 && s.pend_n == P.cap_pend_store) return CTR_EOVERFLOW;
    if (!kBat || ready >= 0)
        push_pending<kArity>(s, pend, ((uint64_t)ready << kKeyBits) | (uint64_t)k, P, heap_stride(P.cap_pr), bad);
    if constexpr (kBat) s.q += 1;
    s.sum += weight;
    return CTR_OK;
}

// One request's bounds and its place in arrival order (`before`: the previous one's arrival).
__device__ __forceinline__ bool request_valid(const SimParams& P, int64_t i, int64_t before, bool& bad)
{
    const int64_t t = ck_ld(P.trace.arrival_us, i, P.trace_len, bad);
    const int64_t p = ck_ld(P.trace.prompt_len, i, P.trace_len, bad);
    const int64_t o = ck_ld(P.trace.true_out, i, P.trace_len, bad);
    const int64_t oh = ck_ld(P.trace.pred_out, i, P.trace_len, bad);
    const int64_t c = ck_ld(P.trace.slo_class, i, P.trace_len, bad);
    return !(t < 0 || t >= kArrivalLimit || p < 0 || p > (1 << 20) || o < 1 || o > (1 << 20) || p + o > P.kv_cap ||
             oh < 0 || oh > (1 << 17) || c >= P.n_classes || t < before);
}

// Every request of a replica (CTR_EINVAL before anything is simulated); one warp.
__device__ __forceinline__ bool row_valid(const SimParams& P, int64_t tb, int lane, bool& bad)
{
    bool ok = true;
#pragma unroll 4
    for (int64_t k = lane; k < P.n_req; k += 32)
        ok = request_valid(P, tb + k, k > 0 ? ck_ld(P.trace.arrival_us, tb + k - 1, P.trace_len, bad) : 0, bad) && ok;
    return __all_sync(kFull, ok);
}

// argmin of 64-bit values within aligned groups of G lanes (ties -> lowest lane),
// returned as the lane index inside the group: a butterfly minimum, then one
// ballot for the lanes that hold it (every lane of the warp calls it)
template <int G>
__device__ __forceinline__ int group_argmin(uint64_t v, int gl)
{
    if constexpr (G == 32) {
        return warp_argmin(v);
    } else {
        uint64_t m = v;  // the group's minimum, then its lowest lane holding it
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) {
            const uint64_t o = __shfl_xor_sync(kFull, m, off, G);
            m = o < m ? o : m;
        }
        const uint32_t ball = __ballot_sync(kFull, v == m);
        return __ffs((ball >> ((threadIdx.x & 31) - gl)) & ((1u << G) - 1u)) - 1;
    }
}

// One warp carries 32 / G rows side by side: lanes [g*G, g*G + G) simulate
// row base_row + g, lane g*G + i being instance i of that row.  All rows of a
// workload have the same number of requests, so the groups walk their
// arrivals in lockstep (request k of every row at once, each at its own time);
// the per-lane event loops, the per-group argmins and the commits are
// independent across groups.  kMode 1 compiles in the deployed proxy's
// signals (ledger backlog, polled occupancy), kMode 2 batched prefill as
// well; the host launches the least instantiation a launch needs.
//
// Batched prefill: a prefill lane's ring holds its in-flight requests as
// k << 26 | d << 21 | p (running batch first, then the queue).  Before the
// decode lanes advance to an arrival, the prefill lanes end every batch that
// ends by then and start the next at that instant; each newly started batch
// (contiguous at the ring's head) is published to the group, and every
// decode lane copies its own members, now with known KV-ready times, into its
// pending heap.  Repeated until no prefill lane has another batch ending.
template <int G, int kMode, int kBlocksPerSM>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, kBlocksPerSM) sim_kernel(const __grid_constant__ SimParams P)
{
    constexpr bool kSig = kMode >= 1;  // the proxy's signals: ledger backlog, polled occupancy
    constexpr bool kBat = kMode == 2;  // batched prefill
    constexpr int kArity = kBat ? 2 : 4;  // heap arity: binary with batched prefill (see heap_push_bin)
    constexpr int kRowsPerWarp = 32 / G;
    const int lane = threadIdx.x & 31;
    const int grp = lane / G;
    const int gl = lane % G;
    const uint32_t gmask = G == 32 ? kFull : (((1u << G) - 1u) << (grp * G));
    const int64_t slot = (int64_t)blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    if (slot >= P.n_slots) return;
    unsigned char* sb = P.ws + slot * P.slot_bytes;
    const int64_t pr_stride = heap_stride(P.cap_pr);
    // the lane's place in the slot, which holds row_lanes lanes a row (lanes past a row's instances use none)
    const int sl = grp * P.row_lanes + gl;
    uint64_t* pend = reinterpret_cast<uint64_t*>(sb) + sl * pr_stride;  // decode lanes: 4-ary heap
    int64_t* ring = reinterpret_cast<int64_t*>(sb) + sl * pr_stride;    // prefill lanes: ring from 0
    uint64_t* act = reinterpret_cast<uint64_t*>(sb + P.off_act) + sl * heap_stride(P.cap_act);
    uint32_t* wait = reinterpret_cast<uint32_t*>(sb + P.off_wait) + sl * P.cap_wait;

    const bool is_pre = gl < P.n_pre;
    const bool is_dec = gl >= P.n_pre && gl < P.n_pre + P.n_dec;
    const int64_t per_rep = (int64_t)P.n_sets * P.n_pols;
    const int64_t n = P.n_req;

    for (;;) {
        uint32_t base32 = 0;
        if (lane == 0) base32 = atomicAdd(P.next_row, (uint32_t)kRowsPerWarp);
        const int64_t base_row = __shfl_sync(kFull, base32, 0);
        if (base_row >= P.n_rows) break;
        const int64_t row = base_row + grp;
        const bool has_row = row < P.n_rows;
        const int64_t rep = has_row ? row / per_rep : 0;
        const int set = has_row ? (int)((row / P.n_pols) % P.n_sets) : 0;
        const int pol = has_row ? P.pols[row % P.n_pols] : CTR_POLICY_ROUND_ROBIN;
        const ConstsDev& cc = P.sets[set];
        // the in-flight sum the row's decode pricing reads: predicted lengths for the length
        // heuristic and the proxy's ledger, else true remaining tokens (unread by JSQ / RR)
        const bool learned_row = pol == CTR_POLICY_LEARNED || pol == CTR_POLICY_LEARNED_P2;
        const bool sum_is_o_hat = pol == CTR_POLICY_LENGTH_HEURISTIC || (kSig && learned_row && cc.proxy);
        const int64_t tb = rep * n;
        const int64_t ob = row * n;
        const RowView<kBlocksPerSM <= 4, kArity> V(P, tb, ob);

        // per-request bounds, one row at a time with the whole warp
        bool oob = false;  // bounds-checked builds: an index of this lane fell outside its buffer
        bool valid = false;
        int64_t checked = -1;
        bool ok = false, oob_g = false;
        for (int g = 0; g < kRowsPerWarp; ++g) {
            const int64_t r = base_row + g;
            if (r >= P.n_rows) break;
            if (r / per_rep != checked) {  // the warp's rows are mostly one replica's
                checked = r / per_rep;
                oob_g = false;
                ok = row_valid(P, checked * n, lane, oob_g);
            }
            if (g == grp) oob = oob_g;
            if (g == grp) valid = ok;
        }
        bool live = has_row && valid;

        Decode s;
        s.step_end = is_dec ? kIdle : 0; s.run = 0; s.step = 1; s.inv_step = 1.0f;
        s.step_idx = 0; s.kv_res = 0; s.kv_rsv = 0; s.sum = 0;
        s.pend_top = kEmpty; s.act_top = kEmpty;
        s.n_act = 0; s.q = 0; s.pend_n = 0; s.w_head = 0; s.w_n = 0;
        // (a lane simulates a prefill or a decode instance, never both: see retire_prefills)
        int64_t& busy = s.step_end;
        int64_t& ring_sum_p = s.sum;
        int32_t& ring_head = s.w_head;
        int32_t& ring_n = s.w_n;
        int64_t kv_seen = 0, last_poll = -1;     // decode lanes: occupancy at the last poll instant
        int32_t rr_p = 0, rr_d = 0;
        uint64_t h = 0;
        int err = CTR_OK;
        BatchQueue bq = {0, 0, 0, 0};
        int32_t &run_n = bq.run_n, &q_batches = bq.q_batches;
        int64_t &run_p = bq.run_p, &q_tail = bq.q_tail;
        const bool batched = kBat && P.pre_batch > 0;

        // Batched prefill: end every batch that ends by T, start the next at that
        // instant, and hand the members' KV-ready times to their decode lanes
        // (warp-collective: every lane of the warp calls it).
        auto prefill_batches = [&](int64_t T) {
            for (;;) {
                int32_t pub_n = 0, pub_head = 0;
                int64_t pub_end = 0;
                if (live && err == CTR_OK && is_pre && run_n > 0 && busy <= T) {
                    ring_head += run_n;
                    if (ring_head >= P.cap_ring) ring_head -= P.cap_ring;
                    ring_n -= run_n;
                    ring_sum_p -= run_p;
                    run_n = 0;
                    run_p = 0;
                    if (ring_n > 0) {  // the next batch: the head, then FCFS while the budget holds
                        int pos = ring_head;
                        int64_t pmax = 0;
                        while (run_n < ring_n) {
                            const int64_t pj = ck_ld(ring, pos, (int64_t)P.cap_ring, oob) & kRingPMask;
                            if (run_n > 0 && run_p + pj > P.pre_batch) break;
                            run_p += pj;
                            pmax = pj > pmax ? pj : pmax;
                            run_n += 1;
                            pos = pos + 1 == P.cap_ring ? 0 : pos + 1;
                        }
                        busy += P.pre_base + P.pre_tok * run_p;
                        q_batches -= 1;
                        if (q_batches == 0) q_tail = 0;
                        if (busy + P.xfer_tok * pmax >= kTimeLimit) {
                            err = CTR_EOVERFLOW;
                        } else {
                            pub_n = run_n;
                            pub_head = ring_head;
                            pub_end = busy;
                        }
                    }
                }
                if (!__any_sync(kFull, pub_n > 0)) break;
                const int64_t* const rings = reinterpret_cast<const int64_t*>(sb);
                for (int i = 0; i < P.n_pre; ++i) {
                    const int src = grp * G + i;
                    const int32_t m_i = __shfl_sync(kFull, pub_n, src);
                    const int32_t h_i = __shfl_sync(kFull, pub_head, src);
                    const int64_t e_i = __shfl_sync(kFull, pub_end, src);
                    if (is_dec && live) {
                        int pos = h_i;
                        for (int32_t m = 0; m < m_i; ++m) {
                            const int64_t v = ck_ld(rings + (grp * P.row_lanes + i) * pr_stride, pos, (int64_t)P.cap_ring, oob);
                            if ((int)((v >> kRingPBits) & 31) == gl - P.n_pre) {
                                const int64_t ready = e_i + P.xfer_tok * (v & kRingPMask);
                                if (s.pend_n == P.cap_pend_store) {
                                    err = CTR_EOVERFLOW;  // the waiting FIFO has overflowed
                                } else {
                                    push_pending<kArity>(s, pend,
                                                         ((uint64_t)ready << kKeyBits) | (uint64_t)(v >> kRingKShift),
                                                         P, pr_stride, oob);
                                }
                            }
                            pos = pos + 1 == P.cap_ring ? 0 : pos + 1;
                        }
                    }
                }
            }
        };

        for (int64_t base = 0; base < n; base += G) {
            if (!__any_sync(kFull, live)) break;
            const int64_t kl = base + gl;
            const bool mine = live && kl < n;
            int64_t my_t = 0;
            uint32_t my_pc = 0, my_o = 0, my_oh = 0;
            if (mine) {
                my_t = ck_ld(P.trace.arrival_us, tb + kl, P.trace_len, oob);
                my_pc = (uint32_t)ck_ld(P.trace.prompt_len, tb + kl, P.trace_len, oob) |
                        ((uint32_t)ck_ld(P.trace.slo_class, tb + kl, P.trace_len, oob) << 24);
                my_o = (uint32_t)ck_ld(P.trace.true_out, tb + kl, P.trace_len, oob);
                my_oh = (uint32_t)ck_ld(P.trace.pred_out, tb + kl, P.trace_len, oob);
            }
            uint32_t my_route = 0;
            const int cnt = (int)(n - base < G ? n - base : G);
            for (int j = 0; j < cnt; ++j) {
                const int64_t T = __shfl_sync(kFull, my_t, j, G);

                // 1. advance every instance to the arrival time
                if constexpr (kBat) {
                    if (batched) prefill_batches(T);
                }
                if (live) {
                    if (is_dec) {
                        int64_t tsnap = -1;  // >= 0: the occupancy at this time is recorded on the way
                        if (kSig && cc.poll_us > 0) {
                            // the router sees the occupancy of the last poll instant floor(T / D) D,
                            // taken after every event at that instant, on the way to T
                            const int64_t tp = (int64_t)div_recip((uint64_t)T, (uint64_t)cc.poll_us, cc.poll_recip) *
                                               cc.poll_us;
                            if (tp > last_poll) {
                                tsnap = tp;
                                last_poll = tp;
                            }
                        }
                        if (err == CTR_OK)
                            err = decode_advance<kSig, kArity>(s, T, P, pend, act, wait, V, tsnap, kv_seen,
                                                               sum_is_o_hat, oob);
                    } else if (is_pre && !batched) {
                        retire_prefills<kSig, kArity>(s, T, P, ring, oob);
                    }
                }
                if (__ballot_sync(kFull, err != CTR_OK) & gmask) live = false;

                __syncwarp();  // the lanes leave their event loops at different passes: regroup
                // the request's features (read after the advance, which does not need them)
                const int64_t k = base + j;
                const uint32_t pc = __shfl_sync(kFull, my_pc, j, G);
                const int64_t pk = pc & 0xFFFFFFu;
                const int ck = (int)(pc >> 24);
                const int64_t ok = __shfl_sync(kFull, my_o, j, G);
                const int64_t ohk = __shfl_sync(kFull, my_oh, j, G);
                // 2. price the candidates and take the argmin of each pool
                uint64_t cost = kEmpty;
                if (live && pol != CTR_POLICY_ROUND_ROBIN && (is_pre || is_dec))
                    cost = instance_cost<kSig, kBat>(P, cc, pol, is_pre, is_pre ? gl : gl - P.n_pre, s, bq, kv_seen,
                                                     Request{k, T, (uint32_t)pk, (uint32_t)ohk, ck});
                int ip = rr_p, id = rr_d;
                if (G < 32 || pol != CTR_POLICY_ROUND_ROBIN) {  // a whole warp's row has one policy
                    const int amin_p = group_argmin<G>(is_pre ? cost : kEmpty, gl);
                    const int amin_d = group_argmin<G>(is_dec ? cost : kEmpty, gl);
                    if (pol != CTR_POLICY_ROUND_ROBIN) {
                        ip = amin_p;
                        id = amin_d - P.n_pre;
                    }
                }
                rr_p = rr_p + 1 == P.n_pre ? 0 : rr_p + 1;
                rr_d = rr_d + 1 == P.n_dec ? 0 : rr_d + 1;

                // 3. commit: FCFS prefill, KV transfer, queue at the decode instance
                int64_t ready = 0;
                if (batched && live && gl == ip) {
                    if (ring_n == P.cap_ring) {
                        err = CTR_EOVERFLOW;
                        ready = kTimeLimit;
                    } else {
                        int pos = ring_head + ring_n;
                        if (pos >= P.cap_ring) pos -= P.cap_ring;
                        ck_st(ring, pos, (int64_t)P.cap_ring, (k << kRingKShift) | ((int64_t)id << kRingPBits) | pk, oob);
                        ring_n += 1;
                        ring_sum_p += pk;
                        if (run_n == 0) {  // an idle instance starts a batch of this request at once
                            busy = T + P.pre_base + (int64_t)(int32_t)P.pre_tok * (int32_t)pk;
                            run_n = 1;
                            run_p = pk;
                            ready = busy + (int64_t)(int32_t)P.xfer_tok * (int32_t)pk;
                            if (ready >= kTimeLimit) err = CTR_EOVERFLOW;
                        } else {  // queued: its KV-ready time is known when its batch starts
                            if (q_batches > 0 && q_tail + pk <= P.pre_batch) {
                                q_tail += pk;
                            } else {
                                q_batches += 1;
                                q_tail = pk;
                            }
                            ready = -1;
                        }
                    }
                } else if (live && gl == ip) {
                    const int64_t end = prefill_end(P, busy, T, (uint32_t)pk);
                    ready = end + (int64_t)(int32_t)P.xfer_tok * (int32_t)pk;
                    err = ready >= kTimeLimit ? CTR_EOVERFLOW : push_prefill<kSig, kArity>(s, end, (uint32_t)pk, P, ring, oob);
                }
                if constexpr (kBat) __syncwarp();  // the decode lanes will read the ring entries stored here
                ready = __shfl_sync(kFull, ready, ip, G);
                if (live && gl == P.n_pre + id && ready < kTimeLimit && err == CTR_OK)
                    err = queue_decode<kArity>(s, T, k, ready, sum_is_o_hat ? ohk : ok, P, pend, wait, oob);
                if (gl == j) my_route = ((uint32_t)ip << 8) | (uint32_t)id;
                if (__ballot_sync(kFull, err != CTR_OK) & gmask) live = false;
            }
            if (mine && live) {
                // the routing term of the row checksum, all lanes at once (the
                // first-token and completion terms are added by hash_kernel)
                h += hterm(kl, 1, (uint64_t)my_route);
                if (P.i_pre) ck_st(P.i_pre, ob + kl, P.out_len, (uint8_t)(my_route >> 8), oob);
                if (P.i_dec) ck_st(P.i_dec, ob + kl, P.out_len, (uint8_t)(my_route & 0xFF), oob);
            }
        }
        // drain: every remaining batch, then every remaining event
        if constexpr (kBat) {
            if (batched) {
                prefill_batches(kDrain);
                if (__ballot_sync(kFull, err != CTR_OK) & gmask) live = false;
            }
        }
        if (live && is_dec) {
            err = decode_advance<false, kArity>(s, kDrain, P, pend, act, wait, V, -1, kv_seen, sum_is_o_hat,
                                                oob);
        }

#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) h += __shfl_xor_sync(kFull, h, off, G);
        int status = CTR_OK;
        if (__ballot_sync(kFull, err == CTR_ETIMEOUT) & gmask) status = CTR_ETIMEOUT;
        if (__ballot_sync(kFull, err == CTR_EOVERFLOW) & gmask) status = CTR_EOVERFLOW;
        if (has_row && !valid) status = CTR_EINVAL;
#if CTR_BOUNDS_CHECK
        if (__ballot_sync(kFull, oob) & gmask) status = CTR_EBOUNDS;
#endif
        if (gl == 0 && has_row) {
            P.row_status[row] = status;
            P.row_hash[row] = status == CTR_OK ? h : 0;
        }
    }
}

// One block per row, one warp per instance, for launches of few rows: all lanes
// of a warp simulate the same instance (same state, same control flow; what they
// share in memory follows heap_push_warp's rule), so no event waits for another instance's and the heaps are worked by
// the whole warp.  Every warp follows the row's arrivals.  Per arrival the
// instances' costs go through shared memory, one barrier, and each warp takes
// both argmins itself; the ends of all prefill queues ride along in every warp
// (lane i that of instance i), so the KV-ready time needs no second exchange and
// a round-robin row needs no barrier until its end.  Without batched prefill.
// Bound by its longest chain an arrival: about 3,600 cycles for the learned
// router; of 4,100 on an earlier source 2,500 were one instance's event, 800 its
// price and 600 the commit (cycle counters around each, 2P+6D).
constexpr uint64_t kFailed = kEmpty - 1;  // in place of a cost: the row has failed
template <int kMode, int kWarps>
__global__ void __launch_bounds__(kWarps * 32, 16 / kWarps) sim_row_kernel(const __grid_constant__ SimParams P)
{
    static_assert(kMode < 2, "no batched prefill");
    constexpr bool kSig = kMode == 1;
    constexpr int kArity = 32;
    __shared__ uint64_t cost_s[2][kWarps];  // arrivals alternate between the two
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int n_inst = P.n_pre + P.n_dec;  // the block's warps
    unsigned char* sb = P.ws + (int64_t)blockIdx.x * P.slot_bytes;
    const int64_t pr_stride = heap_stride(P.cap_pr);
    uint64_t* pend = reinterpret_cast<uint64_t*>(sb) + w * pr_stride;
    int64_t* ring = reinterpret_cast<int64_t*>(sb) + w * pr_stride;
    uint64_t* act = reinterpret_cast<uint64_t*>(sb + P.off_act) + w * heap_stride(P.cap_act);
    uint32_t* wait = reinterpret_cast<uint32_t*>(sb + P.off_wait) + w * P.cap_wait;
    const bool is_pre = w < P.n_pre;
    const int64_t per_rep = (int64_t)P.n_sets * P.n_pols;
    const int64_t n = P.n_req;

    for (int64_t row = blockIdx.x; row < P.n_rows; row += gridDim.x) {
        const int set = (int)((row / P.n_pols) % P.n_sets);
        const int pol = P.pols[row % P.n_pols];
        const ConstsDev& cc = P.sets[set];
        const bool learned_row = pol == CTR_POLICY_LEARNED || pol == CTR_POLICY_LEARNED_P2;
        const bool sum_is_o_hat = pol == CTR_POLICY_LENGTH_HEURISTIC || (kSig && learned_row && cc.proxy);
        const int64_t tb = row / per_rep * n, ob = row * n;
        const RowView<true, kArity> V(P, tb, ob);
        bool oob = false;  // bounds-checked builds: an index of this warp fell outside its buffer

        // per-request bounds and arrival order, a stretch of 32 requests per warp
        bool bad = false;
        for (int64_t k = (int64_t)w * 32 + lane; k < n; k += (int64_t)n_inst * 32)
            bad = bad || !request_valid(P, tb + k, k > 0 ? ck_ld(P.trace.arrival_us, tb + k - 1, P.trace_len, oob) : 0, oob);
        const bool valid = !__syncthreads_or(bad);

        Decode s;
        s.step_end = is_pre ? 0 : kIdle; s.run = 0; s.step = 1; s.inv_step = 1.0f;
        s.step_idx = 0; s.kv_res = 0; s.kv_rsv = 0; s.sum = 0;
        s.pend_top = kEmpty; s.act_top = kEmpty;
        s.n_act = 0; s.q = 0; s.pend_n = 0; s.w_head = 0; s.w_n = 0;
        const BatchQueue bq = {0, 0, 0, 0};
        int64_t kv_seen = 0, last_poll = -1;  // occupancy at the last poll instant
        int64_t busy = 0;                     // lane i: the end of prefill instance i's last prefill
        int ip = P.n_pre - 1, id = P.n_dec - 1;
        uint64_t h = 0;
        int err = CTR_OK;
        uint32_t failed_by = CTR_MAX_REQUESTS;  // round robin: the request by whose routing this instance had failed
        bool go = valid;  // the same in every thread of the block
        for (int64_t base = 0; go && base < n; base += 32) {
            const int64_t kl = base + lane;
            int64_t my_t = 0;
            uint32_t my_pc = 0, my_o = 0, my_oh = 0, my_route = 0;
            if (kl < n) {
                my_t = ck_ld(P.trace.arrival_us, tb + kl, P.trace_len, oob);
                my_pc = (uint32_t)ck_ld(P.trace.prompt_len, tb + kl, P.trace_len, oob) |
                        ((uint32_t)ck_ld(P.trace.slo_class, tb + kl, P.trace_len, oob) << 24);
                my_o = (uint32_t)ck_ld(P.trace.true_out, tb + kl, P.trace_len, oob);
                my_oh = (uint32_t)ck_ld(P.trace.pred_out, tb + kl, P.trace_len, oob);
            }
            const int cnt = (int)(n - base < 32 ? n - base : 32);
            for (int j = 0; go && j < cnt; ++j) {
                const int64_t k = base + j;
                const int64_t T = __shfl_sync(kFull, my_t, j);
                const uint32_t pc = __shfl_sync(kFull, my_pc, j);
                const uint32_t pk = pc & 0xFFFFFFu, ok = __shfl_sync(kFull, my_o, j), ohk = __shfl_sync(kFull, my_oh, j);
                // 1. the instance's events up to the arrival
                if (err == CTR_OK) {
                    if (is_pre) {
                        retire_prefills<kSig, kArity>(s, T, P, ring, oob);
                    } else {
                        int64_t tsnap = -1;  // >= 0: the occupancy at this time is recorded on the way
                        if (kSig && cc.poll_us > 0) {
                            const int64_t tp = (int64_t)div_recip((uint64_t)T, (uint64_t)cc.poll_us, cc.poll_recip) *
                                               cc.poll_us;
                            if (tp > last_poll) {
                                tsnap = tp;
                                last_poll = tp;
                            }
                        }
                        err = decode_advance<kSig, kArity>(s, T, P, pend, act, wait, V, tsnap, kv_seen, sum_is_o_hat, oob);
                    }
                }
                // 2. the costs of all instances and the argmin of each pool
                if (pol == CTR_POLICY_ROUND_ROBIN) {
                    if (err != CTR_OK && failed_by == CTR_MAX_REQUESTS) failed_by = (uint32_t)k;
                    ip = ip + 1 == P.n_pre ? 0 : ip + 1;
                    id = id + 1 == P.n_dec ? 0 : id + 1;
                } else {
                    uint64_t cost = kFailed;
                    if (err == CTR_OK)
                        cost = instance_cost<kSig, false>(P, cc, pol, is_pre, is_pre ? w : w - P.n_pre, s, bq, kv_seen,
                                                          Request{k, T, pk, ohk, (int)(pc >> 24)});
                    uint64_t* const slot = cost_s[k & 1];
                    if (lane == 0) slot[w] = cost;
                    __syncthreads();
                    const uint64_t c = lane < n_inst ? slot[lane] : kEmpty;
                    if (__any_sync(kFull, c == kFailed)) {  // every warp reads the same costs
                        go = false;
                        break;
                    }
                    ip = warp_argmin(lane < P.n_pre ? c : kEmpty);
                    id = warp_argmin(lane < P.n_pre ? kEmpty : c) - P.n_pre;
                }
                // 3. commit
                const int64_t end = prefill_end(P, __shfl_sync(kFull, busy, ip), T, pk);
                const int64_t ready = end + (int64_t)(int32_t)P.xfer_tok * (int32_t)pk;
                if (ready >= kTimeLimit) {  // the same in every warp
                    if (err == CTR_OK) err = CTR_EOVERFLOW;
                    go = false;
                    break;
                }
                if (lane == ip) busy = end;
                if (err == CTR_OK) {
                    if (w == ip)
                        err = push_prefill<kSig, kArity>(s, end, pk, P, ring, oob);
                    else if (w == P.n_pre + id)
                        err = queue_decode<kArity>(s, T, k, ready, sum_is_o_hat ? ohk : ok, P, pend, wait, oob);
                }
                if (lane == j) my_route = ((uint32_t)ip << 8) | (uint32_t)id;
            }
            if (go && w == 0 && kl < n) {  // the routing term of the row checksum
                h += hterm(kl, 1, (uint64_t)my_route);
                if (P.i_pre) ck_st(P.i_pre, ob + kl, P.out_len, (uint8_t)(my_route >> 8), oob);
                if (P.i_dec) ck_st(P.i_dec, ob + kl, P.out_len, (uint8_t)(my_route & 0xFF), oob);
            }
        }
        if (go && !is_pre && err == CTR_OK)  // drain: every remaining event
            err = decode_advance<false, kArity>(s, kDrain, P, pend, act, wait, V, -1, kv_seen, sum_is_o_hat, oob);

#pragma unroll
        for (int off = 16; off > 0; off >>= 1) h += __shfl_xor_sync(kFull, h, off);
        // The row's status is that of its first failure.  Costs that are exchanged end a row there, an overflow of the
        // commit before or of the same advance counting before a timeout; the warps of a round-robin row, which exchange
        // nothing, ran on, so the earliest of theirs is looked for.
        __syncthreads();  // the last costs have been read
        if (lane == 0) cost_s[0][w] = err == CTR_OK ? ~0u : 2 * failed_by + (err == CTR_ETIMEOUT);
        __syncthreads();  // (the next row's check has a barrier before its first cost)
        const uint32_t first = __reduce_min_sync(kFull, lane < n_inst ? (uint32_t)cost_s[0][lane] : ~0u);
        int status = first == ~0u ? CTR_OK : (first & 1u) != 0 ? CTR_ETIMEOUT : CTR_EOVERFLOW;
        if (!valid) status = CTR_EINVAL;
#if CTR_BOUNDS_CHECK
        if (__syncthreads_or(oob)) status = CTR_EBOUNDS;
#endif
        if (threadIdx.x == 0) {
            P.row_status[row] = status;
            P.row_hash[row] = status == CTR_OK ? h : 0;
        }
    }
}

// The first-token and completion terms of the row checksum, one block per
// row over the simulator's outputs (coalesced; cheaper than hashing inside
// the diverged event handlers).  Rows that failed keep the checksum 0.
constexpr int kHashThreads = 256;
__global__ void __launch_bounds__(kHashThreads) hash_kernel(const __grid_constant__ SimParams P, const uint64_t* kmix)
{
    __shared__ uint64_t part[kHashThreads / 32];
    for (int64_t row = blockIdx.x; row < P.n_rows; row += gridDim.x) {
        if (P.row_status[row] != CTR_OK) continue;  // block-uniform
        const int64_t ob = row * P.n_req;
        uint64_t h = 0;
#pragma unroll 4
        for (int64_t k = threadIdx.x; k < P.n_req; k += kHashThreads) {
            const int64_t tf = __ldcs(&P.t_first[ob + k]);
            const int64_t td = __ldcs(&P.t_done[ob + k]);
            if (kmix)  // the request-only halves, mixed once per call (launch_mix_table)
                h += mix64(__ldg(&kmix[k]) ^ (uint64_t)tf) + mix64(__ldg(&kmix[P.n_req + k]) ^ (uint64_t)td);
            else
                h += hterm(k, 2, (uint64_t)tf) + hterm(k, 3, (uint64_t)td);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) h += __shfl_xor_sync(kFull, h, off);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = h;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint64_t t = 0;
            for (int w = 0; w < kHashThreads / 32; ++w) t += part[w];
            P.row_hash[row] += t;
        }
        __syncthreads();  // part[] is reused by the next row
    }
}

}  // namespace

int64_t sim_slot_bytes(const ctr_sim_cfg& cfg, int lanes, int64_t* off_act, int64_t* off_wait, int32_t* cap_pr)
{
    const int64_t pend_store = (int64_t)cfg.cap_pending + cfg.cap_waiting + 1;  // pending heap entries
    const int64_t pr = pend_store > cfg.cap_prefill_ring ? pend_store : cfg.cap_prefill_ring;
    const int64_t a = heap_stride(pr) * 8 * lanes;
    const int64_t b = a + heap_stride(cfg.cap_active) * 8 * lanes;
    const int64_t c = b + (int64_t)cfg.cap_waiting * 4 * lanes;
    *off_act = a;
    *off_wait = b;
    *cap_pr = (int32_t)pr;
    return (c + 255) / 256 * 256;
}

int sim_group_width(int n_instances)
{
    return n_instances <= 4 ? 4 : n_instances <= 8 ? 8 : n_instances <= 16 ? 16 : 32;
}

// Rows of a launch are spread over more warps, fewer to a warp, while that
// leaves at most kSpreadWarps warps an SM: a warp of one row has fewer diverged
// event sequences to serialise, and as long as few warps share an SM a launch
// lasts as long as one warp.  With more of them the issue slots run out and
// packing wins.  1,500 requests on 2P+6D, four policies, with 1 / 2 / 4 rows to a
// warp: 1,536 rows take 3.6 / 3.8 / 4.1 ms, 2,048 take 3.9 / 3.8 / 4.1, 3,072
// take 5.0 / 4.3 / 4.7, 4,096 take 6.1 / 4.8 / 4.7; learned rows of 65 constant
// sets: 2,080 rows 4.2 / 4.6 / 5.3, 4,160 rows 6.7 / 5.7 / 6.1.
constexpr int kSpreadWarps = 14;
int sim_rows_per_warp(int width, int64_t n_rows)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 32 / width;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 32 / width;
    int rpw = 1;
    while (rpw < 32 / width && (n_rows + rpw - 1) / rpw > (int64_t)sms * kSpreadWarps) rpw *= 2;
    return rpw;
}

int sim_max_resident_warps(int* warps_per_block, int* blocks)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    // the launch bound of the instantiations with the fewest registers: every width and mode has 8 blocks an
    // SM, so one workspace size fits every launch
    *warps_per_block = kWarpsPerBlock;
    *blocks = sms * 8;
    return sms * 8 * kWarpsPerBlock;
}

namespace {

// The instantiation with the most registers at which all of the launch's
// persistent warps are resident at once (its launch bound promises that many
// blocks an SM): 4 blocks / up to 128 registers (90 to 105 are used) for launches
// of up to 16 warps an SM, which wait on their own chains and not for issue slots,
// so spills and constants re-read from the parameter bank cost time (against 7
// blocks, 1,500 requests: 2,048 document rows 4.8 -> 4.3 ms, 2,080 learned rows
// 4.5 -> 4.2); 7 blocks / 72 registers for one wave of up to 28; else 8 / 64,
// where more warps hide more latency.
template <int G, int kMode>
cudaError_t launch_width(const SimParams& p, int blocks, cudaStream_t stream)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
    const cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int64_t per_block = (int64_t)sms * kWarpsPerBlock;  // warps at one block an SM
    if (p.n_slots <= 4 * per_block)
        sim_kernel<G, kMode, 4><<<blocks, kWarpsPerBlock * 32, 0, stream>>>(p);
    else if (p.n_slots <= 7 * per_block)
        sim_kernel<G, kMode, 7><<<blocks, kWarpsPerBlock * 32, 0, stream>>>(p);
    else
        sim_kernel<G, kMode, 8><<<blocks, kWarpsPerBlock * 32, 0, stream>>>(p);
    return cudaGetLastError();
}

// A block per row, a warp per instance, where every block is resident at 128
// registers (16 warps an SM) and has at most 16 warps.  2,000 requests, four
// policies, 2P+6D: 152 rows 3.58 ms against 3.91 with a row per warp, 304 rows
// 3.95 / 3.91 (proxy's signals 3.38 / 3.73, baselines alone 2.23 / 2.65), 400 rows
// (a second wave; an earlier source) 5.55 / 4.03; 3P+9D, 152 rows: 3.63 / 3.81,
// 200 (a second wave): 5.11 / 3.82; 4P+12D, 152 rows: 3.66 / 3.75;
// 4P+28D (32 warps, 64 registers; an earlier source): 5.1 / 4.0.
constexpr int kRowWarpsPerSM = 16;
bool row_per_block(const SimParams& p, int sms)
{
    const int64_t n_inst = p.n_pre + p.n_dec;
    return p.pre_batch == 0 && n_inst <= 16 && p.n_rows * n_inst <= (int64_t)sms * kRowWarpsPerSM && p.n_slots >= p.n_rows &&
           p.rows_per_warp == 1;
}

template <int kMode>
cudaError_t launch_mode(const SimParams& p, int blocks, cudaStream_t stream)
{
    if constexpr (kMode < 2) {
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
        const cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if (row_per_block(p, sms)) {
            const unsigned threads = (unsigned)(p.n_pre + p.n_dec) * 32;
            if (threads <= 8 * 32)
                sim_row_kernel<kMode, 8><<<(unsigned)p.n_rows, threads, 0, stream>>>(p);
            else
                sim_row_kernel<kMode, 16><<<(unsigned)p.n_rows, threads, 0, stream>>>(p);
            return cudaGetLastError();
        }
    }
    switch (32 / p.rows_per_warp) {
    case 4: return launch_width<4, kMode>(p, blocks, stream);
    case 8: return launch_width<8, kMode>(p, blocks, stream);
    case 16: return launch_width<16, kMode>(p, blocks, stream);
    default: return launch_width<32, kMode>(p, blocks, stream);
    }
}

}  // namespace

cudaError_t launch_sim(const SimParams& p, int blocks, int warps_per_block, cudaStream_t stream)
{
    (void)warps_per_block;
    bool signals = false;  // the proxy's ledger backlog or polled occupancy in some constant set
    for (int i = 0; i < p.n_sets; ++i) signals = signals || p.sets[i].proxy != 0 || p.sets[i].poll_us > 0;
    const cudaError_t e = p.pre_batch > 0 ? launch_mode<2>(p, blocks, stream)
                          : signals       ? launch_mode<1>(p, blocks, stream)
                                          : launch_mode<0>(p, blocks, stream);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t launch_hash(const SimParams& p, const uint64_t* kmix, int blocks, cudaStream_t stream)
{
    if (p.n_rows == 0) return cudaSuccess;
    const int64_t hb = p.n_rows < (int64_t)blocks * 8 ? p.n_rows : (int64_t)blocks * 8;
    hash_kernel<<<(unsigned)hb, kHashThreads, 0, stream>>>(p, kmix);
    return cudaGetLastError();
}

}  // namespace ctr
