// trace.cu -- synthetic request trace on the GPU (ctr_gen_trace).
//
// A warp takes 32 consecutive requests of a replica (a chunk), one to a lane.
// Per request: two Philox4x32-10 blocks (Salmon et al., SC'11), rounded
// lognormal prompt / output lengths (Table 1 profiles), a predicted output
// length with multiplicative lognormal noise (sec. III-C, sec. V-G), an SLO
// class, and an integer unit-rate exponential gap.  An int64 inclusive scan
// turns gaps into cumulative work (exact in any order); Poisson arrivals divide
// by the rate, MMPP arrivals find their state interval among windows of 32.
// With many replicas a warp walks one replica's chunks in order
// (trace_kernel); with few, a cluster of blocks shares one replica
// (trace_split_kernel).
//
// Bit-identity with the CPU reference construction rests on doing only IEEE
// basic operations in a fixed order, in fp32 (the precision the integer
// lengths and gaps are defined in; GB300's fp64 rate would bound the kernel):
// every operation below is an explicit round-to-nearest intrinsic (no
// contraction into FMA; the file is also compiled with -fmad=false), and
// log / exp / the normal quantile are written here from their published
// methods rather than taken from CUDA's math library.
#include <cooperative_groups.h>

#include "ctr_internal.cuh"

namespace cg = cooperative_groups;

namespace ctr {
namespace {

using U32x4 = Philox4;
__device__ __forceinline__ U32x4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                        uint32_t k1)
{
    return philox4x32_10(c0, c1, c2, c3, k0, k1);
}

// ------------------------------------------------------------- fp32 helpers
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float dvd(float a, float b) { return __fdiv_rn(a, b); }

// Integer <-> float conversions without the 64-bit conversion instructions
// (GB300 runs those on its narrow fp64 pipe).  rn_u33(n): n < 2^33 rounded
// once to fp32 -- the exact sum of two exactly representable parts, rounded by
// one fp32 addition; trunc_pos(v): the integer part of a non-negative finite
// float below 2^63, read off its exponent and mantissa.
__device__ __forceinline__ float rn_u33(uint64_t n)
{
    const float hi = __uint2float_rn((uint32_t)(n >> 9));   // < 2^24: exact
    const float lo = __uint2float_rn((uint32_t)(n & 511u));  // exact
    return add(mul(hi, 512.0f), lo);
}

__device__ __forceinline__ int64_t trunc_pos(float v)
{
    const uint32_t b = __float_as_uint(v);
    const int e = (int)((b >> 23) & 0xffu) - 127;  // -0.0 (from ln 1) has e < 0 and gives 0
    if (e < 0) return 0;
    const uint64_t mant = (uint64_t)((b & 0x007FFFFFu) | 0x00800000u);
    return (int64_t)(e >= 23 ? mant << (e - 23) : mant >> (23 - e));
}

// (u + 1/2) 2^-32 rounded once to fp32; 1 - U is the same of ~u
__device__ __forceinline__ float u01(uint32_t u)
{
    return mul(rn_u33(2ull * u + 1ull), 0x1p-33f);
}

// Natural log of a positive normal x: x = m 2^e with m in (sqrt(1/2), sqrt(2)],
// s = (m - 1)/(m + 1), ln m = 2 s sum_{i=0..5} s^(2i) / (2i + 1) by Horner,
// ln x = e * ln2_hi + (e * ln2_lo + ln m)  (ln2_hi has 16 significant bits).
__device__ float det_logf(float x)
{
    const float inv_odd[6] = {0x1p+0f, 0x1.555556p-2f, 0x1.99999ap-3f, 0x1.24924ap-3f, 0x1.c71c72p-4f, 0x1.745d18p-4f};
    const uint32_t bits = __float_as_uint(x);
    int e = (int)((bits >> 23) & 0xffu) - 127;
    float m = __uint_as_float((bits & 0x007FFFFFu) | 0x3F800000u);
    if (m > 0x1.6a09e6p+0f) {
        m = mul(m, 0.5f);
        e += 1;
    }
    const float f = sub(m, 1.0f);
    const float s = dvd(f, add(m, 1.0f));
    const float z = mul(s, s);
    float acc = inv_odd[5];
#pragma unroll
    for (int i = 4; i >= 0; --i) acc = add(mul(acc, z), inv_odd[i]);
    const float ln_m = mul(add(s, s), acc);
    const float ed = __int2float_rn(e);
    return add(mul(ed, 0x1.62e4p-1f), add(mul(ed, 0x1.7f7d1cp-20f), ln_m));
}

// Two fp32 operations in one instruction, each rounded to nearest on its own.
struct F2 {
    uint64_t v;
};
__device__ __forceinline__ F2 pack(float lo, float hi)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack(F2 a, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v)); }
__device__ __forceinline__ F2 add2(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
// The product as a fused multiply-add of -0, which rounds a b alone and keeps its sign.  The zeros come from
// the kernel's parameters: where the assembler sees a plain product, or knows the zeros, it contracts it into
// the add.rn.f32x2 that follows, and one request in 3,000 got another length.
__device__ __forceinline__ F2 mul2(F2 a, F2 b, uint64_t minus_zeros)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(minus_zeros));
    return r;
}

// exp: k = nearest integer to x / ln2 (halves away from zero),
// r = (x - k ln2_hi) - k ln2_lo, e^r by its degree-7 Taylor polynomial, times
// 2^k through the exponent field.  x is clamped to [-87, 88].
__device__ float det_expf(float x)
{
    const float inv_fact[8] = {0x1p+0f, 0x1p+0f, 0x1p-1f, 0x1.555556p-3f, 0x1.555556p-5f, 0x1.111112p-7f,
                               0x1.6c16c2p-10f, 0x1.a01a02p-13f};
    if (x > 88.0f) x = 88.0f;
    if (x < -87.0f) x = -87.0f;
    const float kf = mul(x, 0x1.715476p+0f);
    const int k = __float2int_rz(kf >= 0.0f ? add(kf, 0.5f) : sub(kf, 0.5f));
    const float kd = __int2float_rn(k);
    const float r = sub(sub(x, mul(kd, 0x1.62e4p-1f)), mul(kd, 0x1.7f7d1cp-20f));
    float acc = inv_fact[7];
#pragma unroll
    for (int i = 6; i >= 0; --i) acc = add(mul(acc, r), inv_fact[i]);
    return mul(acc, __uint_as_float((uint32_t)(k + 127) << 23));
}

// exp of two values, operation by operation the same (k ln2 is negated to subtract it by an addition)
__device__ __forceinline__ void det_expf2(float x0, float x1, uint64_t mz, float& e0, float& e1)
{
    const float inv_fact[8] = {0x1p+0f, 0x1p+0f, 0x1p-1f, 0x1.555556p-3f, 0x1.555556p-5f, 0x1.111112p-7f,
                               0x1.6c16c2p-10f, 0x1.a01a02p-13f};
    if (x0 > 88.0f) x0 = 88.0f;
    if (x0 < -87.0f) x0 = -87.0f;
    if (x1 > 88.0f) x1 = 88.0f;
    if (x1 < -87.0f) x1 = -87.0f;
    const F2 x = pack(x0, x1);
    float f0, f1;
    unpack(mul2(x, pack(0x1.715476p+0f, 0x1.715476p+0f), mz), f0, f1);
    const int k0 = __float2int_rz(add(f0, copysignf(0.5f, f0))), k1 = __float2int_rz(add(f1, copysignf(0.5f, f1)));
    const F2 kd = pack(__int2float_rn(k0), __int2float_rn(k1));
    const F2 r = add2(add2(x, mul2(kd, pack(-0x1.62e4p-1f, -0x1.62e4p-1f), mz)),
                      mul2(kd, pack(-0x1.7f7d1cp-20f, -0x1.7f7d1cp-20f), mz));
    F2 acc = pack(inv_fact[7], inv_fact[7]);
#pragma unroll
    for (int i = 6; i >= 0; --i) acc = add2(mul2(acc, r, mz), pack(inv_fact[i], inv_fact[i]));
    unpack(mul2(acc, pack(__uint_as_float((uint32_t)(k0 + 127) << 23), __uint_as_float((uint32_t)(k1 + 127) << 23)), mz), e0,
           e1);
}

// Wichura (1988), algorithm AS241 PPND16 in fp32: rational approximations of
// degree 7 in r = 0.180625 - q^2 (|q| <= 0.425, q = U - 1/2) or in
// r = sqrt(-ln min(U, 1 - U)) shifted by 1.6 (r <= 5) or by 5.  The numerator
// and the denominator go through Horner's scheme as one pair.
__device__ __forceinline__ void ratio7(const float* num, const float* den, float r, uint64_t mz, float& n,
                                       float& d)
{
    const F2 rr = pack(r, r);
    F2 acc = pack(num[7], den[7]);
#pragma unroll
    for (int i = 6; i >= 0; --i) acc = add2(mul2(acc, rr, mz), pack(num[i], den[i]));
    unpack(acc, n, d);
}

// 2^33 (U - 1/2) = 2 u + 1 - 2^32 (odd, below 2^32 in magnitude) as q = U - 1/2 rounded once
__device__ __forceinline__ float centred(uint32_t u)
{
    const bool neg = (u & 0x80000000u) == 0;
    const uint32_t mag = neg ? ~(u << 1) : (u << 1) + 1u;  // |2 u + 1 - 2^32|
    const float m = __uint2float_rn(mag);
    return mul(neg ? -m : m, 0x1p-33f);
}

constexpr float kCentre = 0x1.b33334p-2f;  // |q| up to here: the central approximation

// the central approximation of three words, side by side so that each coefficient pair is fetched once
__device__ __forceinline__ void ndtri_centre3(const float (&q)[3], uint64_t mz, float (&z)[3])
{
    const float a[8] = {0x1.b18d92p+1f, 0x1.0a4888p+7f, 0x1.ece5d2p+10f, 0x1.ad1d8cp+13f,
                        0x1.66c3e8p+15f, 0x1.06c1c6p+16f, 0x1.052d26p+15f, 0x1.39a296p+11f};
    const float b[8] = {0x1p+0f, 0x1.5281b4p+5f, 0x1.5797fp+9f, 0x1.512322p+12f,
                        0x1.4b772ep+14f, 0x1.3317cap+15f, 0x1.c0e458p+14f, 0x1.46a7ecp+12f};
    F2 rr[3], acc[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float r = sub(0x1.71eb86p-3f, mul(q[i], q[i]));
        rr[i] = pack(r, r);
        acc[i] = pack(a[7], b[7]);
    }
#pragma unroll
    for (int j = 6; j >= 0; --j) {
        const F2 c = pack(a[j], b[j]);
#pragma unroll
        for (int i = 0; i < 3; ++i) acc[i] = add2(mul2(acc[i], rr[i], mz), c);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float n, d;
        unpack(acc[i], n, d);
        z[i] = dvd(mul(q[i], n), d);
    }
}

__device__ float ndtri_tail(uint32_t u, uint64_t mz)
{
    const float c[8] = {0x1.6c666p+0f, 0x1.285774p+2f, 0x1.713f72p+2f, 0x1.d2ecb2p+1f,
                        0x1.453ccp+0f, 0x1.ef2abcp-3f, 0x1.744eb6p-6f, 0x1.9615acp-11f};
    const float d[8] = {0x1p+0f, 0x1.06cefcp+1f, 0x1.ad278ep+0f, 0x1.61293p-1f,
                        0x1.2f5124p-3f, 0x1.f207a8p-7f, 0x1.1f18ccp-11f, 0x1.20d3f6p-30f};
    const float e[8] = {0x1.aa1b1cp+2f, 0x1.5daea6p+2f, 0x1.c8ea64p+0f, 0x1.2fad94p-2f,
                        0x1.b2b412p-6f, 0x1.45c19p-10f, 0x1.c6ec6cp-16f, 0x1.afb74ep-23f};
    const float f[8] = {0x1p+0f, 0x1.331d34p-1f, 0x1.186eb2p-3f, 0x1.e76f94p-7f,
                        0x1.9c8bcap-11f, 0x1.35c2c4p-16f, 0x1.31447p-23f, 0x1.269cp-49f};
    const bool neg = (u & 0x80000000u) == 0;
    const float r = __fsqrt_rn(-det_logf(u01(neg ? u : ~u)));
    float n, m;
    if (r <= 5.0f)
        ratio7(c, d, sub(r, 0x1.99999ap+0f), mz, n, m);
    else
        ratio7(e, f, sub(r, 5.0f), mz, n, m);
    const float v = dvd(n, m);
    return neg ? -v : v;
}

// The normal quantiles of three words per lane, warp-collective.  15 % of the
// words lie in the tails, so nearly every warp would run the tail path (a
// logarithm, a square root, a rational) once for each of the three with a few
// lanes active; instead the tail words of all lanes queue up in shared memory
// (the warp's 96 entries at `q`) and are done together, 32 at a time: 14.4 of
// them on average, so one pass.
__device__ __forceinline__ void ndtri3(const uint32_t (&u)[3], float (&z)[3], uint64_t mz, uint32_t* q,
                                       int lane)
{
    uint32_t m[3], pos[3];
    uint32_t total = 0;
    const uint32_t below = (1u << lane) - 1u;
    float c[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        c[i] = centred(u[i]);
        const bool tail = fabsf(c[i]) > kCentre;
        const uint32_t b = __ballot_sync(0xffffffffu, tail);
        pos[i] = total + __popc(b & below);
        total += __popc(b);
        m[i] = tail;
        if (m[i]) q[pos[i]] = u[i];
    }
    ndtri_centre3(c, mz, z);
    __syncwarp();
    for (uint32_t i = lane; i < total; i += 32) q[i] = __float_as_uint(ndtri_tail(q[i], mz));
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if (m[i]) z[i] = __uint_as_float(q[pos[i]]);
    __syncwarp();  // the queue is free for the next chunk
}

// clip(floor(v + 1/2), lo, hi) for v >= 0 (NaN / inf / huge -> hi); hi <= 2^20, exact in fp32
__device__ __forceinline__ int32_t round_clip(float v, const TraceParams::Clip& c)
{
    const float y = add(v, 0.5f);
    const int32_t t = __float2int_rz(y);
    return !(y < c.hi_f) ? c.hi : t < c.lo ? c.lo : t;
}

// floor(num / d) for num >= 0 with recip = floor((2^64 - 1) / d): the estimate is low by at most 2
__device__ __forceinline__ int64_t div_rate(int64_t num, int64_t d, uint64_t recip)
{
    uint64_t q = __umul64hi((uint64_t)num, recip);
    uint64_t r = (uint64_t)num - q * (uint64_t)d;
    if (r >= (uint64_t)d) {
        ++q;
        r -= (uint64_t)d;
    }
    if (r >= (uint64_t)d) ++q;
    return (int64_t)q;
}

// The replica's Philox key and sub-stream.
struct Stream {
    uint32_t k0, k1, sub_id;
};
__device__ __forceinline__ Stream stream_of(const TraceParams& P, int64_t r)
{
    const int64_t g = P.replica_offset + r;
    const uint64_t seed = P.seed + (uint64_t)(g % P.n_seeds);
    return {(uint32_t)seed, (uint32_t)(seed >> 32), (uint32_t)(g / P.n_seeds)};
}

// Request k's lengths and class, written to its place; returns its gap (0 past
// the end).  Warp-collective.
__device__ __forceinline__ int64_t request(const TraceParams& P, const Stream& S, int64_t row, int64_t k, uint32_t* q,
                                           int lane)
{
    const U32x4 x = philox((uint32_t)k, S.sub_id, 0u, 0u, S.k0, S.k1);
    const U32x4 y = philox((uint32_t)k, S.sub_id, 0u, 1u, S.k0, S.k1);
    const uint32_t u[3] = {x.v[0], x.v[2], x.v[3]};
    float z[3];
    ndtri3(u, z, P.minus_zeros, q, lane);
    if (k >= P.n_req) return 0;
    const bool is_short = (uint64_t)x.v[1] < P.mix_short_thr;
    const float mu = is_short ? P.short_mu : P.long_mu;
    const float sg = is_short ? P.short_sigma : P.long_sigma;
    float ep, eo;
    det_expf2(add(P.prompt_mu, mul(P.prompt_sigma, z[0])), add(mu, mul(sg, z[1])), P.minus_zeros, ep, eo);
    const int32_t p = round_clip(ep, P.prompt), o = round_clip(eo, P.outlen);
    const int32_t oh = round_clip(mul(__int2float_rn(o), det_expf(mul(P.noise_sigma, z[2]))), P.pred);
    // the cumulative thresholds at or below the word: those of 0 always are, t is at or below it when t - 1 is less
    const int c = P.class_base + (y.v[0] > P.class_below[0]) + (y.v[0] > P.class_below[1]) + (y.v[0] > P.class_below[2]);
    P.out.prompt_len[row + k] = p;
    P.out.true_out[row + k] = o;
    P.out.pred_out[row + k] = oh;
    P.out.slo_class[row + k] = (uint8_t)c;
    return trunc_pos(mul(-det_logf(u01(y.v[1])), 0x1.dcd65p+29f));
}

// inclusive warp scan of 64-bit integers (sums mod 2^64)
__device__ __forceinline__ uint64_t scan32(uint64_t v, int lane)
{
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint64_t w = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += w;
    }
    return v;
}

// Arrival times from cumulative work, for one warp whose lam never decreases.
// MMPP: lane l holds interval j0 + l of a window of 32, its start time and the
// work done before it; the window after starts at (t_next, a_next), and
// (ti, ai, end, par) is the interval found last.  A dwell longer than any trace
// counts as 2^58 of work, so no sum leaves 64 bits (lam stays below 2^23 gaps of
// 2.3e10 < 2^58) and no later interval is looked at.
struct Arrivals {
    int64_t j0, t, t_next, ti;
    uint64_t a, a_next, ai, end;
    int par;

    __device__ __forceinline__ void window(const TraceParams& P, const Stream& S, int lane)
    {
        const U32x4 x = philox((uint32_t)(j0 + lane), S.sub_id, 1u, 0u, S.k0, S.k1);
        const uint64_t d = (uint64_t)trunc_pos(mul(-det_logf(u01(x.v[0])), P.dwell_mean_f));
        uint64_t w = (uint64_t)P.rate[lane & 1] * d;  // below 2^62; j0 is even
        if (w > (uint64_t(1) << 58)) w = uint64_t(1) << 58;
        const uint64_t td = scan32(d, lane), aw = scan32(w, lane);
        t = t_next + (int64_t)(td - d);
        a = a_next + aw - w;
        t_next += (int64_t)__shfl_sync(0xffffffffu, td, 31);
        a_next += __shfl_sync(0xffffffffu, aw, 31);
    }
    __device__ __forceinline__ void start(const TraceParams& P, const Stream& S, int lane)
    {
        j0 = t = t_next = ti = 0;
        a = a_next = ai = end = 0;  // an empty interval: the first call looks its own up
        par = 0;
        if (P.arrival_kind == 1) window(P, S, lane);
    }
    // each lane's arrival for its lam (unused where !live); warp-collective
    __device__ __forceinline__ int64_t time(const TraceParams& P, const Stream& S, uint64_t lam, bool live, int lane)
    {
        if (P.arrival_kind == 0) return div_rate((int64_t)lam, P.rate[0], P.rate_recip[0]);
        int64_t out = 0;
        bool done = !live;
        for (;;) {
            if (!done && lam < end) {
                out = ti + div_rate((int64_t)(lam - ai), P.rate[par], P.rate_recip[par]);
                done = true;
            }
            const uint32_t left = __ballot_sync(0xffffffffu, !done);
            if (left == 0) return out;
            // the interval of the first lane left: the last one that starts at or before its lam
            const uint64_t lf = __shfl_sync(0xffffffffu, lam, __ffs(left) - 1);
            while (lf >= a_next) {
                j0 += 32;
                window(P, S, lane);
            }
            const int i = 31 - __clz(__ballot_sync(0xffffffffu, a <= lf));  // a never decreases over the lanes
            const uint64_t up = __shfl_sync(0xffffffffu, a, (i + 1) & 31);
            ai = __shfl_sync(0xffffffffu, a, i);
            ti = __shfl_sync(0xffffffffu, t, i);
            end = i < 31 ? up : a_next;
            par = i & 1;
        }
    }
};

// One warp per replica.  Bound by instruction issue (Philox, the fp32 variates): 4,096 x 20,000 MMPP requests took
// 2.95 ms (980 warp-instructions a chunk of 32) with a tail path per variate, scalar polynomials and one dwell at a
// time, and take 2.26 ms (804, 0.72 of the issue slots); 21 B a request are 0.76 TB/s of stores.  At 64 registers the
// 27 warps an SM of that size are one wave.
constexpr int kWalkWarps = 4;
__global__ void __launch_bounds__(kWalkWarps * 32, 7) trace_kernel(const TraceParams P)
{
    __shared__ uint32_t queue[kWalkWarps][96];
    const int lane = threadIdx.x & 31;
    uint32_t* q = queue[threadIdx.x >> 5];
    const int64_t warp = (int64_t)blockIdx.x * kWalkWarps + (threadIdx.x >> 5);
    const int64_t n_warps = (int64_t)gridDim.x * kWalkWarps;
    for (int64_t r = warp; r < P.n_replicas; r += n_warps) {
        const Stream S = stream_of(P, r);
        const int64_t row = r * P.n_req;
        uint64_t carry = 0;  // cumulative unit-rate work before this chunk (nano-events)
        Arrivals arr;
        arr.start(P, S, lane);
        for (int64_t base = 0; base < P.n_req; base += 32) {
            const int64_t k = base + lane;
            const uint64_t lam = carry + scan32((uint64_t)request(P, S, row, k, q, lane), lane);
            carry = __shfl_sync(0xffffffffu, lam, 31);
            const int64_t t = arr.time(P, S, lam, k < P.n_req, lane);
            if (k < P.n_req) P.out.arrival_us[row + k] = t;
        }
    }
}

// A cluster of blocks per replica, each warp a contiguous run of its chunks.
// Pass 1 writes every request's lengths, and its work within the run into its
// arrival's place; the totals of the runs before it, of its block's warps and of
// the cluster's blocks (read from their shared memory), give each run its start;
// pass 2 turns the work into arrival times, each thread reading back what it
// wrote itself.  Bound by the chain of a chunk (Philox, quantile, logarithm) and
// the two cluster barriers: 1 x 10,000 requests take 7.9 us (Poisson) and 12.2 us
// (MMPP: every warp steps over the windows before its run), 356 and 430 us with
// one warp.  Nothing but the totals is shared: with every chunk's total in shared
// memory (8 bytes each, 128 KB for the longest) 650 x 450,000 took 13.6 ms, 10.3 now.
constexpr int kSplitWarps = 8;
constexpr int kMaxCluster = 16;
__global__ void __launch_bounds__(kSplitWarps * 32) trace_split_kernel(const TraceParams P)
{
    __shared__ uint32_t queue[kSplitWarps][96];
    __shared__ uint64_t warp_sum[kSplitWarps];
    __shared__ uint64_t block_sum;
    cg::cluster_group cluster = cg::this_cluster();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t blocks = (int64_t)cluster.num_blocks(), rank = (int64_t)cluster.block_rank();
    const int64_t r = blockIdx.x / blocks;
    const int64_t n_chunks = (P.n_req + 31) / 32, runs = blocks * kSplitWarps, run = rank * kSplitWarps + wid;
    const int64_t c0 = n_chunks * run / runs, c1 = n_chunks * (run + 1) / runs;
    const Stream S = stream_of(P, r);
    const int64_t row = r * P.n_req;

    uint64_t work = 0;  // of the run so far
    for (int64_t c = c0; c < c1; ++c) {
        const int64_t k = c * 32 + lane;
        const uint64_t lam = work + scan32((uint64_t)request(P, S, row, k, queue[wid], lane), lane);
        if (k < P.n_req) P.out.arrival_us[row + k] = (int64_t)lam;
        work = __shfl_sync(0xffffffffu, lam, 31);
    }
    if (lane == 0) warp_sum[wid] = work;
    __syncthreads();
    uint64_t offset = 0;
    for (int w = 0; w < wid; ++w) offset += warp_sum[w];
    if (wid == kSplitWarps - 1 && lane == 0) block_sum = offset + work;
    cluster.sync();  // every block's sum is there
    uint64_t others = lane < rank ? *cluster.map_shared_rank(&block_sum, lane) : 0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) others += __shfl_xor_sync(0xffffffffu, others, off);
    offset += others;

    Arrivals arr;
    arr.start(P, S, lane);
    for (int64_t c = c0; c < c1; ++c) {
        const int64_t k = c * 32 + lane;
        const bool live = k < P.n_req;
        const uint64_t lam = live ? offset + (uint64_t)P.out.arrival_us[row + k] : 0;
        const int64_t t = arr.time(P, S, lam, live, lane);
        if (live) P.out.arrival_us[row + k] = t;
    }
    cluster.sync();  // no block leaves while another may still read its sum
}

}  // namespace

cudaError_t launch_trace(const TraceParams& p, cudaStream_t stream)
{
    if (p.n_replicas == 0 || p.n_req == 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    // Split replicas while a warp each leaves the GPU idle or waiting on one warp's chain (1.4 us a chunk): 64 x 10,000
    // requests 446 -> 35 us.  Short traces leave a block's warps idle and stay with one warp a replica unless there are
    // very few of them: 1,000 x 64 takes 6.8 us there, 6.9 split; 152 x 128 9.0 and 6.1.  The fewer its chunks, the fewer
    // replicas pay for a block's barriers and uneven runs (MMPP, split / whole: 512 requests 1,520 replicas 32 / 36 us,
    // 1,824 38 / 36, 3,040 59 / 49; 1,000 requests 2,280 77 / 79, 2,432 81 / 79; 2,500 requests 2,736 200 / 226, 3,040
    // 221 / 227; 4,000 requests 3,040 339 / 355, 3,344 371 / 416; 20,000 requests 3,040 1,632 / 1,744, 4,096 2,180 /
    // 2,354): the lines of the longer traces are where the split crossed with its chunks' totals in shared memory, and
    // on the safe side of where it would now.
    const int64_t n_chunks = (p.n_req + 31) / 32;
    const int64_t most = (int64_t)sms * (n_chunks < 32 ? 10 : n_chunks < 64 ? 15 : n_chunks < 100 ? 18 : 20);
    if (p.n_replicas <= most && n_chunks >= (p.n_replicas <= sms ? 4 : 16)) {
        // blocks per replica: up to 8 blocks an SM in all, at least 2 chunks a block; clusters of 16 only for a few
        // replicas, as they are slow to place (16 x 10,000: 19.6 us with 8 blocks, 16.8 with 16; 64 x 10,000: 34 us
        // with 4 or 8, 40 with 16)
        int cluster = 1;
        while (cluster < kMaxCluster && p.n_replicas * cluster * 2 <= (cluster < 8 ? sms * 8 : sms * 2) &&
               n_chunks >= cluster * 4)
            cluster *= 2;
        err = cudaFuncSetAttribute(trace_split_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (err != cudaSuccess) return err;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(p.n_replicas * cluster));
        cfg.blockDim = dim3(kSplitWarps * 32);
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cluster;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int fit = 1;
        if (cluster > 8 && (cudaOccupancyMaxActiveClusters(&fit, trace_split_kernel, &cfg) != cudaSuccess || fit < 1)) {
            (void)cudaGetLastError();  // more than the portable 8 blocks: not on every device (the query takes 0.2 us)
            cfg.gridDim.x = (unsigned)(p.n_replicas * 8);
            attr[0].val.clusterDim.x = 8;
        }
        err = cudaLaunchKernelEx(&cfg, trace_split_kernel, p);
        if (err != cudaSuccess) return err;
        return cudaGetLastError();
    }
    // small blocks spread one warp per replica evenly over the SMs (the kernel is
    // issue-bound, so the SM holding the most warps sets its time)
    int64_t blocks = (p.n_replicas + kWalkWarps - 1) / kWalkWarps;
    const int64_t cap = (int64_t)sms * 16;
    if (blocks > cap) blocks = cap;
    trace_kernel<<<(unsigned)blocks, kWalkWarps * 32, 0, stream>>>(p);
    return cudaGetLastError();
}

}  // namespace ctr
