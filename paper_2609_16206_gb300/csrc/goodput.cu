// goodput.cu -- SLO goodput inputs per simulated row (ctr_goodput):
// the count of requests meeting both SLOs of their class (sec. IV-B targets,
// Table 2 goodput), the exact nearest-rank P99 TTFT and, on request, the
// exact nearest-rank P99 TPOT (Table 2 columns).
//
// One block per row.  A P99 needs the largest hundredth of its row only, so a
// sample of the row (256 or, of long rows, more evenly spaced groups of four
// neighbours, a memory sector each, in a histogram over logarithmic bins, 64 per
// octave) first gives a threshold that about 3 % of the values reach, and the one pass over the row
// then keeps those that do: per request the trace's arrival, output length and
// class and the row's t_first and t_done.  The P99 is the value of the remaining
// rank among the kept ones: their histogram over the same bins finds its bin,
// whose members are counted out or, if many, selected by their digits.  A row
// whose kept values are fewer than the rank needs or more than there is room for
// (thousands of equal values at the P99), or of 2^32 and more, takes an exact
// radix select over all its values read from global memory (row_rank).  A TPOT is compared
// without a division (floor(d / m) >= t is d >= t m) and divided only when kept,
// after the pass where there is room for the divisors: in the pass the few lanes
// that keep one would make their whole warp divide.
// Called from ctr_simulate with kHash, the pass also sums each row's checksum
// terms of first-token and completion times; the request-only half of those terms
// is read from the call's table (launch_mix_table) when ctr_simulate has one,
// else mixed in the pass.
#include "ctr_internal.cuh"

namespace ctr {
namespace {

constexpr int kMaxThreads = 512;  // of a block: 128 in launches of many rows
constexpr int kLogBins = 2112;  // bin 0: a value of 0; then 64 per octave of [1, 2^32)
constexpr int kHistWords = kLogBins / 2;  // two 16-bit counts a word (no more than the sample or kMaxCand are counted)
constexpr int kMinSampleLog2 = 10, kMaxSampleLog2 = 13;  // sampled requests of a row (all of a shorter one)
constexpr int kMaxCand = 8192;  // most values kept
constexpr int kFew = 128;       // members of the rank's bin counted out directly
constexpr int kDigit = 10;      // radix select
constexpr int kBins = 1 << kDigit;
constexpr int kSubBins = 256;   // parts of a crowded bin (see finer_threshold)
static_assert(kBins <= kHistWords, "the radix select takes the place of a 16-bit histogram");

// Monotone bin of a value in [0, 2^32): the exponent and the top 6 mantissa bits
// of its fp32 value rounded toward zero (exact integer to float conversion
// order is kept by round-toward-zero, so x <= y gives bin(x) <= bin(y)); values
// outside go to the end bins.
__device__ __forceinline__ uint32_t log_bin(int64_t x)
{
    if (x <= 0) return 0u;
    if (x >= (int64_t(1) << 32)) return kLogBins - 1;
    return (__float_as_uint(__uint2float_rz((uint32_t)x)) >> 17) - (126u << 6);
}
// the least value of a bin, the least of all for bin 0
__device__ __forceinline__ int64_t bin_floor(uint32_t b)
{
    return b == 0 ? INT64_MIN : (int64_t)ceilf(__uint_as_float((b + (126u << 6)) << 17));
}

template <typename T, typename Op>
__device__ T block_reduce(T v, T identity, Op op, T* scratch)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, off));
    if (lane == 0) scratch[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < (int)blockDim.x / 32 ? scratch[lane] : identity;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, off));
        if (lane == 0) scratch[0] = v;
    }
    __syncthreads();
    const T r = scratch[0];
    __syncthreads();
    return r;
}

// The bin holding 0-based rank `rank` among the counts of nb bins, and the count
// of the bins before it, to every thread in pick[0] and pick[1]: each thread sums
// a contiguous run of bins, a block scan of the sums finds the run, its thread
// walks it.  at(b) is the count of bin b.
template <typename At>
__device__ void find_rank_bin(const At& at, int nb, int64_t rank, uint32_t* pick, uint32_t* wsum)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int per = (nb + (int)blockDim.x - 1) / (int)blockDim.x;
    const int b0 = tid * per, b1 = b0 + per < nb ? b0 + per : nb;
    uint32_t sum = 0;
#pragma unroll 4
    for (int b = b0; b < b1; ++b) sum += at(b);
    uint32_t incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    uint32_t before = 0;
    for (int w = 0; w < wid; ++w) before += wsum[w];
    const uint32_t excl = before + incl - sum;
    if ((int64_t)excl <= rank && rank < (int64_t)(excl + sum)) {  // exactly one thread
        uint32_t acc = excl;
        int bin = b0;
        for (int b = b0; b < b1; ++b) {
            const uint32_t c = at(b);
            if ((int64_t)(acc + c) > rank) {
                bin = b;
                break;
            }
            acc += c;
        }
        pick[0] = (uint32_t)bin;
        pick[1] = acc;
    }
    __syncthreads();
}

// Shared scratch of the selections.
struct SelScratch {
    int64_t red64[kMaxThreads / 32];
    uint32_t wsum[kMaxThreads / 32];
    uint32_t pick[2];
    uint32_t n_few;
    uint32_t few[kFew];
};

// 16-bit counts, two to a word
__device__ __forceinline__ void count16(uint32_t* h, uint32_t b, bool& bad)
{
    if (ck_ok(b, kLogBins, bad)) atomicAdd(&h[b >> 1], (b & 1u) ? 0x10000u : 1u);
}
__device__ __forceinline__ uint32_t at16(const uint32_t* h, int b) { return (h[b >> 1] >> ((b & 1) * 16)) & 0xffffu; }

#if CTR_BOUNDS_CHECK
#define CTR_CK_FLAG_PARAM , bool& bad
#define CTR_CK_FLAG_ARG , bad
#else  // the plain build's function keeps its plain signature
#define CTR_CK_FLAG_PARAM
#define CTR_CK_FLAG_ARG
#endif

// use(v) for each value of src over k < n, a few loaded before any is made up
template <typename Src, typename Use>
__device__ __forceinline__ void for_each_value(const Src& src, int64_t n, const Use& use)
{
    constexpr int kBatch = 4;
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int64_t k0 = tid; k0 < n; k0 += kBatch * nt) {
        typename Src::Raw raw[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) raw[u] = src.load(k0 + u * nt < n ? k0 + u * nt : k0);
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            int64_t v;
            if (k0 + u * nt < n && src.value(raw[u], v)) use(v);
        }
    }
}

// Exact radix select: the value of 0-based rank `rank` among those of src that lie in [lo, lo + 2^bits), all of which
// fit in it when bits is 64 (10-bit digits, most significant first).  Block-collective; every thread returns it.
template <typename Src>
__device__ int64_t radix_rank(const Src& src, int64_t n, int64_t rank, int64_t lo, int bits, uint32_t* hist,
                              SelScratch& S CTR_CK_FLAG_PARAM)
{
#if !CTR_BOUNDS_CHECK
    bool bad = false;  // dead: the accessors below compile to plain accesses
#endif
    const int tid = threadIdx.x, nt = blockDim.x;
    uint64_t prefix = 0;  // chosen high bits of (value - lo)
    for (int shift = bits; shift > 0;) {
        const int dbits = shift < kDigit ? shift : kDigit;
        const int above = shift;  // candidates agree with prefix on bits >= above
        shift -= dbits;
        for (int i = tid; i < kBins; i += nt) hist[i] = 0;
        __syncthreads();
        const uint32_t dmask = (1u << dbits) - 1u;
        for_each_value(src, n, [&](int64_t tv) {
            const uint64_t v = (uint64_t)tv - (uint64_t)lo;
            const bool match = above >= 64 || (v >> above) == (prefix >> above);
            if (match) {
                const uint32_t b = (uint32_t)(v >> shift) & dmask;
                if (ck_ok(b, kBins, bad)) atomicAdd(&hist[b], 1u);
            }
        });
        __syncthreads();
        find_rank_bin([&](int b) { return hist[b]; }, kBins, rank, S.pick, S.wsum);
        prefix |= (uint64_t)S.pick[0] << shift;
        rank -= S.pick[1];
        __syncthreads();
    }
    return (int64_t)((uint64_t)lo + prefix);
}
__device__ __forceinline__ int bits_of(uint64_t range) { return range == 0 ? 0 : 64 - __clzll((long long)range); }

// (t_done - t_first) / (o - 1) of o >= 2 tokens, toward zero: 32-bit where it may be
__device__ __forceinline__ int64_t tpot_value(int64_t dec, int32_t o)
{
    return (uint64_t)dec < (uint64_t(1) << 32) ? (int64_t)((uint32_t)dec / (uint32_t)(o - 1)) : dec / (int64_t)(o - 1);
}

// A row's values in memory: x - y, or with kTpot (x - y) / (o - 1) where o >= 2.
template <bool kTpot>
struct RowValues {
    const int64_t *x, *y;
    const int32_t* o;
    int64_t n;
    bool& bad;
    struct Raw {
        int64_t d;
        int32_t o;
    };
    __device__ __forceinline__ Raw load(int64_t k) const
    {
        return {ck_ldg(x, k, n, bad) - ck_ldg(y, k, n, bad), kTpot ? ck_ldg(o, k, n, bad) : 2};
    }
    __device__ __forceinline__ bool value(const Raw& r, int64_t& v) const
    {
        v = r.d;
        if (kTpot && r.o >= 2) v = tpot_value(r.d, r.o);
        return !kTpot || r.o >= 2;
    }
};
// Kept values.
struct KeptValues {
    const uint32_t* cand;
    using Raw = uint32_t;
    __device__ __forceinline__ Raw load(int64_t k) const { return cand[k]; }
    __device__ __forceinline__ bool value(Raw r, int64_t& v) const
    {
        v = r;
        return true;
    }
};

// The value of rank `rank` among all of a row.  A first count over logarithmic bins, 32 per octave, leaves a range whose
// digits the radix select takes (10,000 TPOTs near 15 ms: two passes over memory in all, TTFTs near 1 s: three); a rank
// among values below 1 or from 2^32 on starts from the least and the greatest value.  Block-collective.
template <bool kTpot>
__device__ __noinline__ int64_t row_rank(const int64_t* x, const int64_t* y, const int32_t* o, int64_t n, int64_t rank,
                                         uint32_t* hist, SelScratch& S CTR_CK_FLAG_PARAM)
{
#if !CTR_BOUNDS_CHECK
    bool bad = false;
#endif
    const int tid = threadIdx.x, nt = blockDim.x;
    const RowValues<kTpot> src = {x, y, o, n, bad};
    for (int i = tid; i < kHistWords; i += nt) hist[i] = 0;
    __syncthreads();
    for_each_value(src, n, [&](int64_t v) {
        const uint32_t b = log_bin(v) >> 1;
        if (ck_ok(b, kHistWords, bad)) atomicAdd(&hist[b], 1u);
    });
    __syncthreads();
    find_rank_bin([&](int b) { return hist[b]; }, kHistWords, rank, S.pick, S.wsum);
    const int b = (int)S.pick[0];
    const int64_t before = (int64_t)S.pick[1];
    __syncthreads();
    if (b > 0 && b < kHistWords - 1) {
        const int64_t lo = bin_floor(2 * b);
        return radix_rank(src, n, rank - before, lo, bits_of((uint64_t)(bin_floor(2 * b + 2) - lo - 1)), hist, S CTR_CK_FLAG_ARG);
    }
    int64_t mn = INT64_MAX, mx = INT64_MIN;
    for_each_value(src, n, [&](int64_t v) {
        mn = v < mn ? v : mn;
        mx = v > mx ? v : mx;
    });
    mn = block_reduce<int64_t>(mn, INT64_MAX, [](int64_t a, int64_t b) { return a < b ? a : b; }, S.red64);
    mx = block_reduce<int64_t>(mx, INT64_MIN, [](int64_t a, int64_t b) { return a > b ? a : b; }, S.red64);
    return radix_rank(src, n, rank, mn, bits_of((uint64_t)mx - (uint64_t)mn), hist, S CTR_CK_FLAG_ARG);
}

// the nearest rank of the P99 among m values, 0-based
__device__ __forceinline__ int64_t p99_rank(int64_t m) { return (99 * m + 99) / 100 - 1; }

// The request of sample i: all of a row of up to 2^log2, else evenly spaced groups of four neighbours.
__device__ __forceinline__ int64_t sample_at(int i, int64_t n, int log2)
{
    return n <= (int64_t(1) << log2) ? i : ((((int64_t)(i >> 2) * n) >> (log2 - 2)) & ~int64_t(3)) + (i & 3);
}
// The sampled TTFTs, read again (they are in the L2); the sampled TPOTs, whose division is not repeated, are kept.
struct SampledTtfts {
    RowValues<false> row;
    int log2;
    using Raw = RowValues<false>::Raw;
    __device__ __forceinline__ Raw load(int64_t i) const { return row.load(sample_at((int)i, row.n, log2)); }
    __device__ __forceinline__ bool value(const Raw& r, int64_t& v) const { return row.value(r, v); }
};

// Within bin B (neither the first nor the last), which holds in_bin of src's `taken` samples, the floor of the part that
// holds their want-th largest, by the next 8 bits; the floor of the part above where that leaves more than `most` of
// them.  Block-collective.
template <typename Src>
__device__ __noinline__ int64_t finer_threshold(const Src src, int taken, uint32_t B, int32_t in_bin, int32_t want,
                                                int32_t most, uint32_t* hist, SelScratch& S CTR_CK_FLAG_PARAM)
{
#if !CTR_BOUNDS_CHECK
    bool bad = false;
#endif
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int i = tid; i < kSubBins; i += nt) hist[i] = 0;
    __syncthreads();
    for_each_value(src, taken, [&](int64_t v) {
        if (log_bin(v) != B) return;
        const uint32_t sub = (__float_as_uint(__uint2float_rz((uint32_t)v)) >> 9) & (kSubBins - 1);
        if (ck_ok(sub, kSubBins, bad)) atomicAdd(&hist[sub], 1u);
    });
    __syncthreads();
    find_rank_bin([&](int b) { return hist[b]; }, kSubBins, want < in_bin ? in_bin - want : 0, S.pick, S.wsum);
    uint32_t bits = ((B + (126u << 6)) << 17) + (S.pick[0] << 9);
    if (in_bin - (int32_t)S.pick[1] > most) bits += 1u << 9;
    __syncthreads();  // pick and wsum are free again
    return (int64_t)ceilf(__uint_as_float(bits));
}

// A threshold that at least the top m - p99_rank(m) of about m values reach, from the histogram of `taken`
// samples of them: the floor of the bin of the sample's j-th largest, j six standard deviations above the
// expected count (neighbours are alike; exactly the count when every value is in the sample).  Where that bin holds so
// many that the kept values could outgrow their room (a fifth of a row's TPOTs may lie within 1 %), a finer one: of 352
// simulated rows of 10,000 and 40,000 none needs the radix select with this at 0.6 of the room, five do at 0.9 and 170
// without.  Equal values that are still too many are left out, as the radix select would be sure with them.  src: n_src
// values, the samples among them.  Block-collective.
template <typename Src>
__device__ __forceinline__ int64_t threshold(uint32_t* hist, int32_t taken, int64_t m, uint32_t room, const Src& src, int n_src,
                                             SelScratch& S CTR_CK_FLAG_PARAM)
{
    if (taken <= 0) return INT64_MAX;
    const int64_t top = m - p99_rank(m);
    int32_t j = (int32_t)top;
    if (taken < m) {
        const float e = (float)taken * ((float)top / (float)m);
        j = (int32_t)(e + 6.0f * sqrtf(e)) + 2;
    }
    find_rank_bin([&](int b) { return at16(hist, b); }, kLogBins, j < taken ? taken - j : 0, S.pick, S.wsum);
    const uint32_t B = S.pick[0];
    const int32_t reach = taken - (int32_t)S.pick[1], in_bin = (int32_t)at16(hist, (int)B);
    __syncthreads();  // pick and wsum are free again, and hist is
    if (10 * reach * m <= 6 * (int64_t)taken * room || B == 0 || B == kLogBins - 1) return bin_floor(B);
    const int32_t above = reach - in_bin;
    return finer_threshold<Src>(src, n_src, B, in_bin, j - above, (int32_t)(9 * (int64_t)taken * room / (10 * m)) - above, hist,
                                S CTR_CK_FLAG_ARG);
}

// entries i and i + 1 as one load (bounds-checked builds also check its alignment)
template <typename V, typename T>
__device__ __forceinline__ V ck_ldg_pair(const T* p, int64_t i, int64_t len, bool& bad)
{
    static_assert(sizeof(V) == 2 * sizeof(T), "a pair");
    if (CTR_CK_OUT(i, len - 1, bad)) return V();
#if CTR_BOUNDS_CHECK
    if (reinterpret_cast<uintptr_t>(p + i) % sizeof(V) != 0) {
        bad = true;
        return V();
    }
#endif
    return __ldg(reinterpret_cast<const V*>(p + i));
}

// The value of rank `rank` among c kept ones (c <= kMaxCand).  Block-collective.
__device__ int64_t kept_rank(const uint32_t* cand, int c, int64_t rank, uint32_t* hist, SelScratch& S CTR_CK_FLAG_PARAM)
{
#if !CTR_BOUNDS_CHECK
    bool bad = false;
#endif
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int i = tid; i < kHistWords; i += nt) hist[i] = 0;
    if (tid == 0) S.n_few = 0;
    __syncthreads();
    for (int i = tid; i < c; i += nt) count16(hist, log_bin(cand[i]), bad);
    __syncthreads();
    find_rank_bin([&](int b) { return at16(hist, b); }, kLogBins, rank, S.pick, S.wsum);
    const uint32_t B = S.pick[0];
    const int64_t r_in = rank - (int64_t)S.pick[1];  // among the bin's members
    for (int i = tid; i < c; i += nt) {
        if (log_bin(cand[i]) == B) {
            const uint32_t j = atomicAdd(&S.n_few, 1u);
            if (j < (uint32_t)kFew) S.few[j] = cand[i];
        }
    }
    __syncthreads();
    const int m = (int)S.n_few;
    if (m > kFew) {
        __syncthreads();  // n_few has been read (a bin of a single value has no digits to select by, so no barrier there)
        const int64_t lo = B == 0 ? 0 : bin_floor(B);
        return radix_rank(KeptValues{cand}, c, r_in, lo, B == 0 ? 0 : bits_of((uint64_t)(bin_floor(B + 1) - lo - 1)), hist,
                          S CTR_CK_FLAG_ARG);
    }
    for (int i = tid; i < m; i += nt) {  // the member whose position in (value, slot) order is the rank
        const uint32_t v = S.few[i];
        int pos = 0;
        for (int j = 0; j < m; ++j) pos += S.few[j] < v || (S.few[j] == v && j < i);
        if (pos == r_in) S.pick[0] = v;
    }
    __syncthreads();
    const uint32_t v = S.pick[0];
    __syncthreads();
    return v;
}

// Bound by the pass: about 110 warp-instructions for 32 requests (64-bit times,
// the SLO tables, one kept value in 30) and the bytes in flight.  Eight blocks
// of 128 threads an SM overlap one row's sample and selection with the others'
// passes.  4,096 rows x 20,000: 445 us with the P99 TPOT, 305 us without; 873 and
// 400 us when every request's logarithmic bin was counted and staged in shared
// memory and the TPOT took two more passes of its own.  Those TPOTs are spread out;
// 2,048 simulated rows x 10,000, whose TPOTs crowd within a few percent, take 139 to
// 154 us with the P99 TPOT (mixed lengths, loads 0.1 to 0.85; 262 to 395 with the two
// passes, 403 to 575 while crowded bins outgrew the room of the kept values), and 383
// where most rows have thousands of equal times (502 with the two passes).
template <bool kHash, bool kTpot, bool kLater>
__global__ void __launch_bounds__(kMaxThreads, 2) goodput_kernel(const GoodputParams P)
{
    __shared__ uint32_t hist_s[kHistWords];  // of the TTFTs, then of the kept values
    __shared__ SelScratch S;
    __shared__ uint32_t n_cand[2];
    // kept TTFTs, then TPOTs (with kLater decode times, then output lengths less 1), cap each; before the pass the
    // TPOTs' histogram, then the sampled TPOTs.  Little shared memory leaves the pass more L1 for its loads in flight.
    extern __shared__ uint32_t cand_s[];
    uint32_t* const hist[2] = {hist_s, cand_s};
    const int tid = threadIdx.x, nt = blockDim.x;
    const int64_t n = P.n_req;
    const int64_t trace_len = (P.n_rows / P.rows_per_replica) * n, out_len = P.n_rows * n;  // entries of trace and outputs
    const uint32_t cap = (uint32_t)P.cand_cap;

    for (int64_t row = blockIdx.x; row < P.n_rows; row += gridDim.x) {
        const int64_t tb = (row / P.rows_per_replica) * n, ob = row * n;
        bool bad = false;  // bounds-checked builds: an index of this thread fell outside its buffer

        // ---- the sample and the thresholds
        for (int i = tid; i < kHistWords; i += nt) {
            hist[0][i] = 0;
            if (kTpot) hist[1][i] = 0;
        }
        if (tid < 2) n_cand[tid] = 0;
        const int sample = 1 << P.sample_log2;
        const int taken = n < sample ? (int)n : sample;
        uint32_t* const tpot_s = cand_s + kHistWords;
        int32_t taken_many = 0;
        __syncthreads();
        constexpr int kBatch = 4;  // samples a thread loads before it uses any
        for (int i0 = tid; i0 < taken; i0 += kBatch * nt) {
            int64_t ttft[kBatch], dec[kBatch];
            int32_t o[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                const int i = i0 + j * nt < taken ? i0 + j * nt : i0;
                const int64_t k = sample_at(i, n, P.sample_log2);
                const int64_t tf = ck_ldg(P.t_first, ob + k, out_len, bad);
                ttft[j] = tf - ck_ldg(P.trace.arrival_us, tb + k, trace_len, bad);
                if (kTpot) {
                    o[j] = ck_ldg(P.trace.true_out, tb + k, trace_len, bad);
                    dec[j] = ck_ldg(P.t_done, ob + k, out_len, bad) - tf;
                }
            }
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                if (i0 + j * nt >= taken) continue;
                count16(hist[0], log_bin(ttft[j]), bad);
                if (kTpot) {
                    const int64_t v = o[j] >= 2 ? tpot_value(dec[j], o[j]) : 0;
                    // (in the first and the last bin, which have no finer threshold, values may be cut and others be among them)
                    ck_st(tpot_s, i0 + j * nt, sample, v <= 0 ? 0u : v >> 32 ? ~0u : (uint32_t)v, bad);
                    if (o[j] >= 2) {
                        ++taken_many;
                        count16(hist[1], log_bin(v), bad);
                    }
                }
            }
        }
        if (kTpot) taken_many = block_reduce<int32_t>(taken_many, 0, [](int32_t a, int32_t b) { return a + b; },
                                                      reinterpret_cast<int32_t*>(S.red64));
        else
            __syncthreads();
        const SampledTtfts again = {{P.t_first + ob, P.trace.arrival_us + tb, nullptr, n, bad}, P.sample_log2};
        const int64_t t_ttft = threshold(hist[0], taken, n, cap, again, taken, S CTR_CK_FLAG_ARG);
        uint32_t t_tpot = 0;  // 0: none
        if (kTpot && taken_many > 0) {
            const int64_t t = threshold(hist[1], taken_many,
                                        n <= sample ? taken_many : ((int64_t)taken_many * n) >> P.sample_log2, cap,
                                        KeptValues{tpot_s}, taken, S CTR_CK_FLAG_ARG);
            t_tpot = t > 0 ? (uint32_t)t : 0;  // below 2^32
        }

        // ---- the pass over the row
        int32_t met = 0;
        uint64_t h = 0;     // kHash: the row's first-token and completion checksum terms
        int32_t many = 0;   // kTpot: requests of two tokens or more
        int32_t wide = 0;   // a kept TTFT or decode time of 2^32 or more
        auto request = [&](int64_t k, int64_t ta, int32_t o, int c, int64_t tf, int64_t td) {
            if (c >= P.n_classes) c = P.n_classes - 1;
            const int64_t ttft = tf - ta, dec = td - tf;
            met += ttft <= P.ttft[c] && (o == 1 || dec <= P.tpot[c] * ((int64_t)o - 1));
            if (ttft >= t_ttft) {
                const uint32_t i = atomicAdd(&n_cand[0], 1u);
                if ((uint64_t)ttft >> 32) wide = 1;
                if (i < cap) cand_s[i] = (uint32_t)ttft;
            }
            if (kTpot && o >= 2) {
                ++many;
                if (dec >= (int64_t)((uint64_t)t_tpot * (uint32_t)(o - 1))) {
                    const uint32_t i = atomicAdd(&n_cand[1], 1u);
                    if ((uint64_t)dec >> 32) wide = 1;
                    if (i < cap && kLater) {
                        cand_s[cap + i] = (uint32_t)dec;
                        cand_s[2 * cap + i] = (uint32_t)(o - 1);
                    } else if (i < cap) {
                        cand_s[cap + i] = (uint32_t)dec / (uint32_t)(o - 1);
                    }
                }
            }
            if (kHash) {
                const uint64_t m2 = P.kmix ? ck_ldg(P.kmix, k, 2 * n, bad) : mix64((uint64_t(2) << 56) ^ (uint64_t)k);
                const uint64_t m3 = P.kmix ? ck_ldg(P.kmix, n + k, 2 * n, bad) : mix64((uint64_t(3) << 56) ^ (uint64_t)k);
                h += mix64(m2 ^ (uint64_t)tf) + mix64(m3 ^ (uint64_t)td);
            }
        };
        // kU requests a thread, every load issued before any is used: neighbours in pairs, one 16-byte load of
        // each array, where rows are aligned (an even n), else one by one
        constexpr int kU = 4;
        for (int64_t base = 0; base < n; base += kU * nt) {
            int64_t k[kU], a[kU], f[kU], d[kU];
            int32_t o[kU];
            int c[kU];
            if (P.pairs) {
#pragma unroll
                for (int u = 0; u < kU; u += 2) {
                    k[u] = base + u * nt + 2 * tid;
                    k[u + 1] = k[u] + 1;
                    const int64_t e = k[u] < n ? k[u] : 0;
                    const longlong2 a2 = ck_ldg_pair<longlong2>((const long long*)P.trace.arrival_us, tb + e, trace_len, bad);
                    const int2 o2 = ck_ldg_pair<int2>(P.trace.true_out, tb + e, trace_len, bad);
                    const uchar2 c2 = ck_ldg_pair<uchar2>(P.trace.slo_class, tb + e, trace_len, bad);
                    const longlong2 f2 = ck_ldg_pair<longlong2>((const long long*)P.t_first, ob + e, out_len, bad);
                    const longlong2 d2 = ck_ldg_pair<longlong2>((const long long*)P.t_done, ob + e, out_len, bad);
                    a[u] = a2.x; a[u + 1] = a2.y;
                    o[u] = o2.x; o[u + 1] = o2.y;
                    c[u] = c2.x; c[u + 1] = c2.y;
                    f[u] = f2.x; f[u + 1] = f2.y;
                    d[u] = d2.x; d[u + 1] = d2.y;
                }
            } else {
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    k[u] = base + u * nt + tid;
                    const int64_t e = k[u] < n ? k[u] : 0;
                    a[u] = ck_ldg(P.trace.arrival_us, tb + e, trace_len, bad);
                    o[u] = ck_ldg(P.trace.true_out, tb + e, trace_len, bad);
                    c[u] = ck_ldg(P.trace.slo_class, tb + e, trace_len, bad);
                    f[u] = ck_ldg(P.t_first, ob + e, out_len, bad);
                    d[u] = ck_ldg(P.t_done, ob + e, out_len, bad);
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (k[u] < n) request(k[u], a[u], o[u], c[u], f[u], d[u]);
        }
        auto add = [](int64_t a, int64_t b) { return (int64_t)((uint64_t)a + (uint64_t)b); };  // mod 2^64
        // met and (below it) the multi-token requests, both at most 2^23, and the threads with a wide value: 2^23 met
        // requests are the top bit, so the word is read unsigned
        const uint64_t sums = (uint64_t)block_reduce<int64_t>(((int64_t)met << 40) + ((int64_t)many << 16) + wide, 0, add,
                                                              S.red64);  // its barriers publish the kept values
        many = (int32_t)((sums >> 16) & 0xffffffu);
        const bool packs = (sums & 0xffff) == 0;
        if (kHash) {
            h = (uint64_t)block_reduce<int64_t>((int64_t)h, 0, add, S.red64);
            if (tid == 0 && P.row_status[row] == CTR_OK) P.row_hash[row] += h;  // a failed row keeps 0
        }

        // ---- the rank among the kept values, or among all
        int64_t p99 = -1, p99_tpot = -1;
        if (n > 0) {
            const int64_t below = n - (int64_t)n_cand[0], rank = p99_rank(n);
            if (n_cand[0] <= cap && rank >= below && packs) {
                p99 = kept_rank(cand_s, (int)n_cand[0], rank - below, hist[0], S CTR_CK_FLAG_ARG);
            } else {
                p99 = row_rank<false>(P.t_first + ob, P.trace.arrival_us + tb, nullptr, n, rank, hist[0], S CTR_CK_FLAG_ARG);
            }
        }
        if (kTpot && many > 0) {
            const int64_t below = many - (int64_t)n_cand[1], rank = p99_rank(many);
            if (t_tpot > 0 && n_cand[1] <= cap && rank >= below && packs) {
                if (kLater)
                    for (int i = tid; i < (int)n_cand[1]; i += nt) cand_s[cap + i] /= cand_s[2 * cap + i];
                // (its barriers order the divided values)
                p99_tpot = kept_rank(cand_s + cap, (int)n_cand[1], rank - below, hist[0], S CTR_CK_FLAG_ARG);
            } else {
                p99_tpot = row_rank<true>(P.t_done + ob, P.t_first + ob, P.trace.true_out + tb, n, rank, hist[0],
                                    S CTR_CK_FLAG_ARG);
            }
        }
#if CTR_BOUNDS_CHECK
        const bool out = __syncthreads_or(bad);  // a row whose pass left a buffer: both outputs say so
#endif
        if (tid == 0) {
            P.met[row] = (int64_t)(sums >> 40);
            P.p99[row] = p99;
            if (kTpot) P.p99_tpot[row] = p99_tpot;
#if CTR_BOUNDS_CHECK
            if (out) P.met[row] = P.p99[row] = CTR_EBOUNDS;
#endif
        }
        __syncthreads();  // the shared arrays are free for the next row
    }
}

__global__ void __launch_bounds__(256) mix_table_kernel(uint64_t* t, int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 2 * n; i += (int64_t)gridDim.x * blockDim.x) {
        const bool first = i < n;
        const int64_t k = first ? i : i - n;
        t[i] = mix64(((first ? uint64_t(2) : uint64_t(3)) << 56) ^ (uint64_t)k);
    }
}

constexpr int64_t kLongRow = 30000, kHugeRow = 65536;  // see launch_rows

template <bool kHash, bool kTpot>
cudaError_t launch_rows(const GoodputParams& p, int sms, cudaStream_t stream)
{
    // 128 threads a row, which overlap best (4,096 rows of 20,000 with the P99 TPOT, as all figures here, TPOTs divided
    // in the pass: 481 us, 521 with 256), except
    // - while that leaves an SM's 1,024 threads partly idle (4 rows of 2,000: 15 us with 512, 21 with 128; 32 rows of
    //   50,000: 62 and 169);
    // - for long rows, as the eight rows of an SM drift apart and read their replica's trace again, and their kept
    //   values leave room for fewer blocks (4,096 rows, 128 / 256 / 512 threads: 28,000 requests 637 / 674 / 748 us,
    //   32,000 763 / 756 / 821, 60,000 1,782 / 1,342 / 1,338; 1,824 rows of 90,000 1,243 / 911 / 837);
    // - where eight rows an SM at a time leave the last turn so empty that four at a time take clearly fewer row
    //   times (2,500 rows of 20,000: 343 us with 128, 318 with 256; 1,300: 231 and 196; 3,040 even; rows of 5,000
    //   lose up to 10 %).
    const auto turns = [&](int64_t rows_at_once) {  // row times of an SM
        const int64_t slots = sms * rows_at_once;
        return (p.n_rows + slots - 1) / slots * rows_at_once;
    };
    int threads = 128;
    if (p.n_rows <= (int64_t)sms * 2 || p.n_req >= kHugeRow)
        threads = 512;
    else if (p.n_rows <= (int64_t)sms * 4 || p.n_req >= kLongRow || (p.n_req >= 10000 && 20 * turns(8) > 23 * turns(4)))
        threads = 256;
    // TPOTs are divided after the pass while their divisors leave L1 60 KB of the SM's 256 (with 128 threads up to
    // rows of 23,400, with 256 of 56,000, with 512 of 120,000; with the P99 TPOT, us without / with: 4,096 rows of
    // 20,000 483 / 459, 3,040 of 20,000 384 / 365, 4,096 of 40,000 894 / 848; past it 4,096 of 28,000 633 / 683,
    // 4,096 of 60,000 1,338 / 1,428)
    const size_t block_bytes = sizeof(SelScratch) + kHistWords * 4 + 1024;
    const bool later = kTpot && (kMaxThreads * 2 / threads) * (block_bytes + (size_t)p.cand_cap * 12) <= 196 * 1024;
    const auto k = later ? goodput_kernel<kHash, kTpot, kTpot> : goodput_kernel<kHash, kTpot, false>;
    size_t dyn_bytes = (size_t)p.cand_cap * 4 * (later ? 3 : kTpot ? 2 : 1);
    const size_t sampled = (kHistWords + (size_t(1) << p.sample_log2)) * 4;
    if (kTpot && dyn_bytes < sampled) dyn_bytes = sampled;
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxCand * 12);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, dyn_bytes);
    if (err != cudaSuccess) return err;
    const int64_t cap = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    const int64_t blocks = p.n_rows < cap ? p.n_rows : cap;
    k<<<(unsigned)blocks, threads, dyn_bytes, stream>>>(p);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_mix_table(uint64_t* t, int64_t n, cudaStream_t stream)
{
    if (n <= 0) return cudaSuccess;
    int64_t blocks = (2 * n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    mix_table_kernel<<<(unsigned)blocks, 256, 0, stream>>>(t, n);
    return cudaGetLastError();
}

cudaError_t launch_goodput(const GoodputParams& given, cudaStream_t stream)
{
    if (given.n_rows == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    GoodputParams p = given;
    p.pairs = p.n_req % 2 == 0 &&
              ((uintptr_t)p.trace.arrival_us | (uintptr_t)p.t_first | (uintptr_t)p.t_done) % 16 == 0 &&
              (uintptr_t)p.trace.true_out % 8 == 0 && (uintptr_t)p.trace.slo_class % 2 == 0;
    // one request in 32 to 64 of a long row, so that the kept values, 3 % of a row at 1,024 samples, still have room:
    // 1,200 rows of 200,000: 1,093 us, 3,980 with 1,024 samples (past kMaxCand a row takes the radix select)
    p.sample_log2 = kMinSampleLog2;
    while (p.sample_log2 < kMaxSampleLog2 && (int64_t(64) << p.sample_log2) < p.n_req) ++p.sample_log2;
    // room for a sixteenth of the row (3 % is expected, more where a bin holds many)
    const int64_t room = p.n_req / 16 + 64;
    p.cand_cap = (int32_t)(room < 512 ? 512 : room > kMaxCand ? kMaxCand : room);
    if (p.row_hash) return launch_rows<true, false>(p, sms, stream);
    return p.p99_tpot ? launch_rows<false, true>(p, sms, stream) : launch_rows<false, false>(p, sms, stream);
}

}  // namespace ctr
