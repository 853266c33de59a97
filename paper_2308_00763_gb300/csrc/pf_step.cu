// pf_step.cu -- the fused per-frame SIR step for sm_103a.
//
// One launch per frame for a whole batch of trackers.  A tile is kTile consecutive
// particles k of one tracker's previous frame.  Per tile (in ticket order):
//   1. resampling of the previous frame (Sec. IV, "Normalizing" and "Resampling"):
//      e_k = exp(L_k - M) (Eq. 5 with the max of the previous step), a block scan, and a
//      decoupled lookback over the tracker's earlier tiles give the inclusive prefix
//      P_k; C_k = P_k * (1/S) (the reciprocal saved by the previous step); the strata
//      j with C_{k-1} < u_j <= C_k are the offspring of k.  The tile's offspring form a
//      contiguous range of j, and their ancestors all lie in the tile, so the gather of
//      ancestor positions is a read of the tile's own particles staged in shared memory.
//   2. propagation (Eq. 1-2) of every offspring j with Philox draws keyed by (j, t),
//   3. likelihood (Eq. 3; Eq. 4 scaled half form in F16/BF16) on the new frame.  The
//      likelihood is a function of the particle's pixel only, so each tile first tabulates
//      it in shared memory over the window its offspring can reach (the ancestors'
//      bounding box widened by the drift and the largest draw the 23-bit Box-Muller can
//      produce), from a copy of the frame region staged in shared memory, and each
//      offspring reads its pixel's value; a pixel outside the window is evaluated directly
//      from global memory by the same arithmetic in the same order, so the two routes
//      give identical bits.
//   4. per-tile (max L, sum e, sum e*dx, sum e*dy), merged with rescaling,
//   5. the tile that completes a tracker merges its tiles' partials in index order:
//      M, S, 1/S and the estimate of the frame (the weighted mean of the propagated
//      particles).
// Frame t = 0 has no resampling: every particle starts at the initial position.
//
// Multinomial trackers (Sec. IV: each ancestor drawn from the categorical distribution of
// the weights) are not in the step kernel's launch; they take two other launches per
// frame (the same code in other modes): the CDF kernel runs phase 1 up to the CDF and writes it to
// T.cdf; the pull kernel then gives each offspring j the first particle whose CDF value
// reaches an independent uniform v_j (a search of T.cdf in three levels), gathers the ancestors'
// positions of its tile's offspring into shared memory, sizes the likelihood window by
// them and runs phases 2-5 as the step kernel does.  Gumbel-max trackers (the log-domain
// form of the same draw, Sec. IV), Metropolis and rejection trackers (Sec. III) skip the CDF
// kernel: the pull kernel reads the ancestors their kernel (pf_gumbel.cu, pf_metropolis.cu,
// pf_rejection.cu) wrote to T.anc instead of searching.
//
// Scan boundaries.  The prefix between tiles is an exact 128-bit fixed-point sum of
// the tiles' aggregates, so every tile obtains the same boundary value whichever
// predecessors its lookback visits.  Inside a tile the prefix is an FP scan made
// non-decreasing by a running max and clamped to the exact value at the tile's end.
// Hence C is non-decreasing, the strata ranges of consecutive tiles meet exactly, and
// every j is written by exactly one tile.
#include <cuda_runtime.h>
#include <float.h>
#include <stddef.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "pf_device.cuh"
#include "pf_internal.h"
#include "pf_ref64.cuh"

// The pull kernel's offspring have no likelihood table (window width 0), so its bounds
// tests against the window compare unsigned values with a constant 0.
#pragma nv_diag_suppress 186

namespace pfk {

namespace {

constexpr int kWarps = kThreads / 32;
constexpr int kRoiMax = 2 * kTableMax;     // staged frame pixels (window + template margin)
// Row sums of the half-form table: words (a half2 of two neighbouring cells, or a float)
constexpr int kRowWords = 3 * kTile / 2;
constexpr int kMapMax = 2 * kTile;         // offspring of a tile served by the ancestor map
constexpr uint32_t kSpinLimit = 1u << 22;  // bounded waits: ~1 s with backoff
// Half-width of the likelihood window in standard deviations of the transition noise.
// Every draw is below sqrt(-2 ln 2^-24) = 5.77 in magnitude (kDrawMax, rounded up).  When
// that window has more cells than the block has threads, a window of 3.5 sigma is used:
// a tile's few offspring beyond it (probability 4.7e-4 per coordinate) are cheaper to
// evaluate directly (same arithmetic, same bits) than a window twice as wide.
constexpr float kDrawMax = 5.7683f;
constexpr float kWindowSigmas = 3.5f;

__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t atom_add_acq_rel(uint32_t *p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

__device__ __forceinline__ bool timed_out(const TrackerState *st) {
    return (ld_relaxed_u32(&st->status) & kStatusTimeout) != 0u;
}

// Checked builds (-DPF_CHECKED): every index below that is in range by construction is
// tested; one out of range raises the tracker's bounds bit and is redirected to element 0
// (the host then reports the step as failed).  Other builds use the index as it is.
#ifdef PF_CHECKED
__device__ __forceinline__ int checked_index(int i, int n, TrackerState *st) {
    if (static_cast<unsigned>(i) >= static_cast<unsigned>(n)) {
        atomicOr(&st->status, kStatusBounds);
        return 0;
    }
    return i;
}
#define PF_IDX(i, n) checked_index((i), (n), st)
#else
#define PF_IDX(i, n) (i)
#endif

// The normalised CDF value of a prefix P: P * (1/S) with the reciprocal saved by the
// previous step (the paper's saved constant); the naive study build (-DPF_NAIVE_RESAMPLE)
// divides by S for every element instead.
#ifdef PF_NAIVE_RESAMPLE
#define PF_NORM(P) div_rn((P), Sdiv)
#else
#define PF_NORM(P) mul_rn((P), invS)
#endif

// ---- lookback descriptor words (see LookbackDesc): 16-bit launch tag | 48-bit payload
constexpr uint64_t kPayload48 = (1ull << 48) - 1ull;

__device__ __forceinline__ uint64_t desc_tag(uint32_t ep) {   // never 0 (cleared memory)
    return static_cast<uint64_t>(ep % 65535u + 1u) << 48;
}

__device__ __forceinline__ void st_relaxed_v2(uint64_t *p, uint64_t a, uint64_t b) {
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void st_relaxed_u64(uint64_t *p, uint64_t a) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(a) : "memory");
}
__device__ __forceinline__ void ld_relaxed_v2(const uint64_t *p, uint64_t &a, uint64_t &b) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

// Publish a tile's aggregate (which = 0) or inclusive prefix (which = 1).
__device__ __forceinline__ void desc_publish(LookbackDesc *d, int which, U128 v, uint64_t tag) {
    const uint64_t w0 = (v.lo & kPayload48) | tag;
    const uint64_t w1 = (((v.lo >> 48) | (v.hi << 16)) & kPayload48) | tag;
    const uint64_t w2 = (v.hi >> 32) | tag;
    st_relaxed_v2(&d->w[2 * which], w0, w1);
    st_relaxed_u64(&d->w[4 + which], w2);
}

__device__ __forceinline__ U128 desc_value(uint64_t w0, uint64_t w1, uint64_t w2) {
    U128 v;
    v.lo = (w0 & kPayload48) | (w1 << 48);
    v.hi = ((w1 & kPayload48) >> 16) | ((w2 & kPayload48) << 32);
    return v;
}

// Wait (bounded) until a predecessor tile has published this launch's inclusive prefix
// (returns 2) or aggregate (returns 1), with its value in v.  Returns 0 on timeout (and
// raises the tracker's timeout bit).
__device__ uint32_t wait_desc(const LookbackDesc *d, uint64_t tag, TrackerState *st, U128 &v,
                              uint32_t limit = kSpinLimit) {
    uint32_t ns = 8;
    for (uint32_t it = 0; it < limit; ++it) {
        // all six words in one round trip (the predecessor has usually published only its
        // aggregate when the tiles of a wave look back together)
        uint64_t a0, a1, i0, i1, w4, w5;
        ld_relaxed_v2(&d->w[0], a0, a1);
        ld_relaxed_v2(&d->w[2], i0, i1);
        ld_relaxed_v2(&d->w[4], w4, w5);
        const uint64_t hm = ~kPayload48;
        if ((i0 & hm) == tag && (i1 & hm) == tag && (w5 & hm) == tag) { v = desc_value(i0, i1, w5); return 2u; }
        if ((a0 & hm) == tag && (a1 & hm) == tag && (w4 & hm) == tag) { v = desc_value(a0, a1, w4); return 1u; }
        if ((it & 1023u) == 1023u && timed_out(st)) return 0u;   // another wait already gave up
        __nanosleep(ns);
        if (ns < 256) ns <<= 1;
    }
    atomicOr(&st->status, kStatusTimeout);
    return 0u;
}

// Tile partials of the FP32/FP16/BF16 kernels: 32-bit launch tag | float bits per word.
__device__ __forceinline__ uint64_t partial_tag(uint32_t ep) {   // never 0 (cleared memory)
    return static_cast<uint64_t>(ep % 0x7fffffffu + 1u) << 32;
}

// Wait (bounded) until the words of a tile partial (statistics, and the bounding box when
// the launch tracks it) carry this launch's tag; on timeout the tracker's timeout bit is
// raised and the words read last are returned.
__device__ void wait_partial(const TilePartial *p, uint64_t tag, TrackerState *st, uint64_t (&q)[8], bool with_box,
                             uint32_t limit = kSpinLimit) {
    uint32_t ns = 8;
    const uint64_t hm = 0xffffffff00000000ull;
    q[4] = q[5] = q[6] = q[7] = tag;
    for (uint32_t it = 0; it < limit; ++it) {
        ld_relaxed_v2(&p->w[0], q[0], q[1]);
        ld_relaxed_v2(&p->w[2], q[2], q[3]);
        if (with_box) {
            ld_relaxed_v2(&p->b[0], q[4], q[5]);
            ld_relaxed_v2(&p->b[2], q[6], q[7]);
        }
        if ((q[0] & hm) == tag && (q[1] & hm) == tag && (q[2] & hm) == tag && (q[3] & hm) == tag &&
            (q[4] & hm) == tag && (q[5] & hm) == tag && (q[6] & hm) == tag && (q[7] & hm) == tag)
            return;
        if ((it & 1023u) == 1023u && timed_out(st)) return;
        __nanosleep(ns);
        if (ns < 64) ns <<= 1;
    }
    atomicOr(&st->status, kStatusTimeout);
}

// exp(d) for d <= 0.  CUDA's single-precision expf and __expf return exactly 1 at +-0 and 0 for
// every d below -104 (checked over all of them on this part), so they need no shortcuts of their
// own: two comparisons and selections each, at 2.5 exponentials a particle.  2^20 particles F16
// 21.8 -> 20.0 us a frame, F32 23.6 -> 21.6; 2^24 F16 244 -> 229.
__device__ __forceinline__ double exp_le0(double d) {
    return exp_table_takes(d) ? exp_table(d) : (d < -746.0 ? 0.0 : exp(d));
}
__device__ __forceinline__ float exp_le0(float d) {
    return expf(d);
}
// The FP16/BF16 filters weigh with the hardware exp2 approximation (their likelihoods
// carry ~11 bits); the scan and the statistics use the same function, so they agree.
template <bool kFast, typename A> __device__ __forceinline__ A wexp(A d) { return exp_le0(d); }
template <> __device__ __forceinline__ float wexp<true, float>(float d) {
    return __expf(d);
}

// fmax / fmin of prefixes and CDF values, which are never negative; a NaN loses to any value, as
// with fmax and fmin.  In FP64 on the bits, whose unsigned order is that of the values (an FP64
// comparison costs as much as ten of these instructions): 200003 particles 75.9 -> 70.3 us a
// frame, 2^20 224 -> 214.
__device__ __forceinline__ float prefix_max(float a, float b) { return fmax(a, b); }
__device__ __forceinline__ float prefix_min(float a, float b) { return fmin(a, b); }
__device__ __forceinline__ double prefix_max(double a, double b) {
    constexpr unsigned long long kInf = 0x7ff0000000000000ull;
    const unsigned long long x = static_cast<unsigned long long>(__double_as_longlong(a));
    const unsigned long long y = static_cast<unsigned long long>(__double_as_longlong(b));
    return x > kInf ? b : (y > kInf ? a : (x > y ? a : b));
}
__device__ __forceinline__ double prefix_min(double a, double b) {   // (a NaN's bits are above every value's)
    const unsigned long long x = static_cast<unsigned long long>(__double_as_longlong(a));
    const unsigned long long y = static_cast<unsigned long long>(__double_as_longlong(b));
    return x < y ? a : b;
}

// A likelihood of weight 0 (the elements past a tile's end).
template <typename L> __device__ __forceinline__ L no_weight();
template <> __device__ __forceinline__ double no_weight<double>() { return neg_inf<double>(); }
template <> __device__ __forceinline__ float no_weight<float>() { return neg_inf<float>(); }
template <> __device__ __forceinline__ __half no_weight<__half>() { return __ushort_as_half(0xfc00u); }
template <> __device__ __forceinline__ __nv_bfloat16 no_weight<__nv_bfloat16>() { return __ushort_as_bfloat16(0xff80u); }

template <typename A>
struct Stats {
    A m, s, sx, sy;
};

// Merge of two partial (max, sums) with rescaling to the larger max.  Symmetric:
// stats_merge(a, b) and stats_merge(b, a) give the same bits (no fused multiply-add).
template <bool F, typename A>
__device__ __forceinline__ Stats<A> stats_merge(const Stats<A> &a, const Stats<A> &b) {
    const A m = a.m > b.m ? a.m : b.m;
    if (m == neg_inf<A>()) return a;
    const A sa = (a.m == neg_inf<A>()) ? static_cast<A>(0) : wexp<F>(a.m - m);
    const A sb = (b.m == neg_inf<A>()) ? static_cast<A>(0) : wexp<F>(b.m - m);
    Stats<A> r;
    r.m = m;
    r.s = add_rn(mul_rn(a.s, sa), mul_rn(b.s, sb));
    r.sx = add_rn(mul_rn(a.sx, sa), mul_rn(b.sx, sb));
    r.sy = add_rn(mul_rn(a.sy, sa), mul_rn(b.sy, sb));
    return r;
}

// Order, equality with -inf and narrowing of FP64 values on their words: an FP64 comparison or
// conversion takes as long as ten integer operations.  (-0 orders below +0; no NaN.)  The FP64
// step issued 95 FP64 operations a particle, 21 of them comparisons and conversions; with these,
// the pixel by integers, no exponential of the maximum itself and nothing issued by warps past
// a tile's end: 200003 particles 70.0 -> 58.8 us a frame, 2^20 214 -> 190, 1000 43.6 -> 35.0,
// the same bits.
__device__ __forceinline__ long long order_key(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ bool above(double a, double b) { return order_key(a) > order_key(b); }
__device__ __forceinline__ bool above(float a, float b) { return a > b; }
__device__ __forceinline__ bool is_neg_inf(double v) {
    return static_cast<unsigned long long>(__double_as_longlong(v)) == 0xfff0000000000000ull;
}
__device__ __forceinline__ bool is_neg_inf(float v) { return v == neg_inf<float>(); }
__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(double v) {   // rounded to nearest, as the conversion does
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(v)), lo = static_cast<uint32_t>(__double2loint(v));
    const uint32_t e = (hi >> 20) & 0x7ffu;
    if (e < 897u || e > 1149u) return static_cast<float>(v);   // (zero, FP32 subnormal or beyond)
    const uint32_t f = (hi & 0x80000000u) | ((((hi & 0x7fffffffu) - 0x38000000u) << 3) | (lo >> 29));
    const uint32_t rem = lo & 0x1fffffffu;
    return __uint_as_float(f + (rem > 0x10000000u || (rem == 0x10000000u && (f & 1u)) ? 1u : 0u));
}
// A weight above 2^-30 of the largest (weights are never negative).
__device__ __forceinline__ bool counts_in_box(float w) { return w > 9.3132257461547852e-10f; }
__device__ __forceinline__ bool counts_in_box(double w) { return __double_as_longlong(w) > 0x3e10000000000000ll; }

// Two particles at once (a particle whose flag is false is skipped).  The rescale to a new
// maximum is applied without a branch: when the maximum does not move the factor is
// wexp(0) = 1 exactly (and 1 while no particle has been seen), so the sums are unchanged,
// the same bits as skipping it.
template <bool F, typename A>
__device__ __forceinline__ void stats_add2(Stats<A> &a, bool v0, A L0, A dx0, A dy0, bool v1, A L1, A dx1, A dy1) {
    const A l0 = v0 ? L0 : neg_inf<A>(), l1 = v1 ? L1 : neg_inf<A>();
    A e0, e1;
    if constexpr (sizeof(A) == 8) {
        // FP64: a factor of 1 or a weight of 1 costs more than the branch around it
        const bool first = above(l0, l1);
        const A hi = first ? l0 : l1, lo = first ? l1 : l0;
        if (above(hi, a.m)) {
            if (!is_neg_inf(a.m)) {      // (the sums are 0 otherwise)
                const A sc = wexp<F>(a.m - hi);
                a.s = mul_rn(a.s, sc); a.sx = mul_rn(a.sx, sc); a.sy = mul_rn(a.sy, sc);
            }
            a.m = hi;
        }
        A eh = static_cast<A>(1), el = static_cast<A>(0);
        if (above(a.m, hi)) eh = wexp<F>(hi - a.m);
        if (v0 && v1) el = wexp<F>(lo - a.m);
        e0 = v0 ? (first ? eh : el) : static_cast<A>(0);
        e1 = v1 ? (first ? el : eh) : static_cast<A>(0);
    } else {
        const A mx = l0 > l1 ? l0 : l1;
        const A nm = mx > a.m ? mx : a.m;
        const A sc = (nm == neg_inf<A>()) ? static_cast<A>(1)
                                          : ((a.m == neg_inf<A>()) ? static_cast<A>(0) : wexp<F>(a.m - nm));
        a.s = mul_rn(a.s, sc); a.sx = mul_rn(a.sx, sc); a.sy = mul_rn(a.sy, sc);
        a.m = nm;
        e0 = v0 ? wexp<F>(l0 - a.m) : static_cast<A>(0);
        e1 = v1 ? wexp<F>(l1 - a.m) : static_cast<A>(0);
    }
    // (rounded step by step: an exponential's own last operation is a multiplication, which must
    // not be fused with these)
    a.s = add_rn(a.s, add_rn(e0, e1));
    a.sx = add_rn(a.sx, fma(e0, dx0, mul_rn(e1, dx1)));
    a.sy = add_rn(a.sy, fma(e0, dy0, mul_rn(e1, dy1)));
}

// Pixel of a position (reading C3): floor(v) + (v - floor(v) >= 0.5).  For |v| below
// 2^22 (float) or 2^51 (double) this equals floor(v + 0.5): adding 1/2 is exact unless
// it crosses into the next binade, which happens only when the fraction is >= 1/2 and
// then rounds to the same integer.  Positions are first clamped to +-2^20, far outside
// any frame (template pixels are clamped to the frame, reading C4).
__device__ __forceinline__ int pixel_of(float v) {
    return __float2int_rd(fminf(fmaxf(v, -1048576.0f), 1048576.0f) + 0.5f);
}
__device__ __forceinline__ int pixel_of(double v) {
    return __double2int_rd(fmin(fmax(v, -1048576.0), 1048576.0) + 0.5);
}

// Column (or row) of a position's pixel in a window: pixel_of(v) - origin as an unsigned value,
// and a value above any window's extent when the pixel lies outside [-2^20, 2^20] or v is not
// finite (the caller then takes pixel_of).  FP32: floor(v + 1/2) is formed by adding 1.5 * 2^23
// rounded downwards, which leaves the integer in the low mantissa bits: two additions and an
// integer subtraction instead of two clamps, an addition and a conversion (a quarter-rate
// unit).  For |v| >= 2^22 and any other large or special v the sum's bits differ from those of
// 1.5 * 2^23 by at least 2^22 in either direction, which stays outside the window after the
// subtraction (|origin| < 2^20).
__device__ __forceinline__ unsigned window_offset(float v, int origin) {
    return __float_as_uint(__fadd_rd(__fadd_rn(v, 0.5f), 12582912.0f)) - (0x4B400000u + static_cast<unsigned>(origin));
}
// FP64: floor(v + 1/2) = (floor(2 v) + 1) >> 1 from the words, in integer operations.
__device__ __forceinline__ unsigned window_offset(double v, int origin) {
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(v)), lo = static_cast<uint32_t>(__double2loint(v));
    const uint32_t m = (hi & 0xfffffu) | 0x100000u;
    const int sh = 1042 - static_cast<int>((hi >> 20) & 0x7ffu);   // 2 |v| = (m + lo 2^-32) 2^-sh
    const int s = sh < 31 ? sh : 31;                                // (m >> 31 = 0)
    const uint32_t ip = m >> (s & 31);
    const bool rest = (ip << (s & 31)) != m || lo != 0u;
    const int fl = static_cast<int>(hi) < 0 ? -static_cast<int>(ip) - (rest ? 1 : 0) : static_cast<int>(ip);
    return sh >= 0 ? static_cast<unsigned>((fl + 1) >> 1) - static_cast<unsigned>(origin) : 0xffffffffu;
}

// kItems consecutive elements between memory and registers as 16-byte vectors (kItems *
// sizeof(T) is a multiple of 16 for every element type here; the address is 16-byte
// aligned).  The elements are unpacked from (packed into) the vector words with bit
// operations on constant indices, so the register arrays never need an address (an
// array whose address is taken lives in local memory).
__device__ __forceinline__ uint32_t vword(const uint4 &v, int k) {
    return k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w));
}
__device__ __forceinline__ void set_vword(uint4 &v, int k, uint32_t w) {
    if (k == 0) v.x = w; else if (k == 1) v.y = w; else if (k == 2) v.z = w; else v.w = w;
}
template <typename T> struct Bits;
template <> struct Bits<double> {
    __device__ static __forceinline__ double get(const uint4 *v, int m) {
        return __hiloint2double(static_cast<int>(vword(v[m >> 1], 2 * (m & 1) + 1)),
                                static_cast<int>(vword(v[m >> 1], 2 * (m & 1))));
    }
    __device__ static __forceinline__ void put(uint4 *v, int m, double x) {
        set_vword(v[m >> 1], 2 * (m & 1), static_cast<uint32_t>(__double2loint(x)));
        set_vword(v[m >> 1], 2 * (m & 1) + 1, static_cast<uint32_t>(__double2hiint(x)));
    }
};
template <> struct Bits<float> {
    __device__ static __forceinline__ float get(const uint4 *v, int m) { return __uint_as_float(vword(v[m >> 2], m & 3)); }
    __device__ static __forceinline__ void put(uint4 *v, int m, float x) { set_vword(v[m >> 2], m & 3, __float_as_uint(x)); }
};
template <> struct Bits<int32_t> {
    __device__ static __forceinline__ int32_t get(const uint4 *v, int m) { return static_cast<int32_t>(vword(v[m >> 2], m & 3)); }
    __device__ static __forceinline__ void put(uint4 *v, int m, int32_t x) { set_vword(v[m >> 2], m & 3, static_cast<uint32_t>(x)); }
};
template <> struct Bits<__half> {
    __device__ static __forceinline__ __half get(const uint4 *v, int m) {
        const uint32_t w = vword(v[m >> 3], (m >> 1) & 3);
        return __ushort_as_half(static_cast<unsigned short>((m & 1) ? (w >> 16) : (w & 0xffffu)));
    }
    __device__ static __forceinline__ void put(uint4 *v, int m, __half x) {
        const uint32_t h = __half_as_ushort(x);
        uint32_t w = vword(v[m >> 3], (m >> 1) & 3);
        w = (m & 1) ? ((w & 0xffffu) | (h << 16)) : ((w & 0xffff0000u) | h);
        set_vword(v[m >> 3], (m >> 1) & 3, w);
    }
};
template <> struct Bits<__nv_bfloat16> {
    __device__ static __forceinline__ __nv_bfloat16 get(const uint4 *v, int m) {
        const uint32_t w = vword(v[m >> 3], (m >> 1) & 3);
        return __ushort_as_bfloat16(static_cast<unsigned short>((m & 1) ? (w >> 16) : (w & 0xffffu)));
    }
    __device__ static __forceinline__ void put(uint4 *v, int m, __nv_bfloat16 x) {
        const uint32_t h = __bfloat16_as_ushort(x);
        uint32_t w = vword(v[m >> 3], (m >> 1) & 3);
        w = (m & 1) ? ((w & 0xffffu) | (h << 16)) : ((w & 0xffff0000u) | h);
        set_vword(v[m >> 3], (m >> 1) & 3, w);
    }
};

template <typename T>
__device__ __forceinline__ void load_items(T (&dst)[kItems], const T *src) {
    constexpr int kVec = static_cast<int>(sizeof(T)) * kItems / 16;
    static_assert(kVec * 16 == static_cast<int>(sizeof(T)) * kItems, "kItems elements must fill 16-byte vectors");
    const uint4 *s = reinterpret_cast<const uint4 *>(src);
    uint4 v[kVec];
#pragma unroll
    for (int k = 0; k < kVec; ++k) v[k] = s[k];
#pragma unroll
    for (int m = 0; m < kItems; ++m) dst[m] = Bits<T>::get(v, m);
}
template <typename T>
__device__ __forceinline__ void store_items(T *dst, const T (&src)[kItems]) {
    constexpr int kVec = static_cast<int>(sizeof(T)) * kItems / 16;
    uint4 v[kVec];
#pragma unroll
    for (int k = 0; k < kVec; ++k) v[k] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int m = 0; m < kItems; ++m) Bits<T>::put(v, m, src[m]);
    uint4 *d = reinterpret_cast<uint4 *>(dst);
#pragma unroll
    for (int k = 0; k < kVec; ++k) d[k] = v[k];
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// t mod n for t >= 0 and 0 < n <= 2^16, in 32-bit divisions: a 64-bit one is a called routine, around
// which registers of the whole tile were spilled (F16 2^20 particles 20.0 -> 19.6 us a frame).
__device__ __forceinline__ int64_t mod_small(int64_t t, uint32_t n) {
    const uint32_t hi = static_cast<uint32_t>(static_cast<uint64_t>(t) >> 32), lo = static_cast<uint32_t>(t);
    uint32_t r = hi % n;
    r = ((r << 16) | (lo >> 16)) % n;
    return ((r << 16) | (lo & 0xffffu)) % n;
}

struct FrameView {
    const uint8_t *p;
    int64_t pitch;
    int W, H, r;
    __device__ __forceinline__ uint32_t at(int x, int y) const {
        return __ldg(p + static_cast<int64_t>(clampi(y, 0, H - 1)) * pitch + clampi(x, 0, W - 1));
    }
};

// Integer sum of the template pixels around (px, py) (the exact form of Eq. 3; reading
// C4 clamps template pixels to the frame).  w[i] = half-width of template row dy = i - r
// (TrackerDev::w).
__device__ uint32_t disk_sum(const FrameView &f, const int8_t *w, int px, int py) {
    uint32_t s = 0;
    const int r = f.r;
    if (px - r >= 0 && px + r < f.W && py - r >= 0 && py + r < f.H) {
        const uint8_t *row = f.p + static_cast<int64_t>(py - r) * f.pitch + px;
        for (int i = 0; i <= 2 * r; ++i, row += f.pitch) {
            const int hw = w[i];
            for (int dx = -hw; dx <= hw; ++dx) s += __ldg(row + dx);
        }
    } else {
        for (int dy = -r; dy <= r; ++dy) {
            const int hw = w[dy + r];
            for (int dx = -hw; dx <= hw; ++dx) s += f.at(px + dx, py + dy);
        }
    }
    return s;
}

// Eq. 3 from the integer disk sum: sum (I-bg)^2 - (I-fg)^2 = (fg-bg)(2 sum I - (bg+fg)|D|).
template <typename A>
__device__ __forceinline__ A lik_from_sum(uint32_t s, A c1, A c2D, A den) {
    return (c1 * (static_cast<A>(2) * static_cast<A>(s) - c2D)) / den;
}

// ----------------------------------------------------------------------------------
// Eq. 4 per-pixel scaled form in half precision: a = (I - bg) kappa, b = (I - fg) kappa,
// term = a*a - b*b, summed over the template row by row, left to right, in the lane type
// (F16, the paper's form) or in FP32 (BF16 and PF_FLAG_ACCUM32).
// ----------------------------------------------------------------------------------
template <typename H> struct HalfOps;

template <>
struct HalfOps<__half> {
    using h2 = __half2;
#ifndef PF_NAIVE_RESAMPLE
    // (1024 + I) has the bit pattern 0x6400 | I in binary16, so the pixel enters the
    // half arithmetic without a conversion instruction: h - (1024 + level) is exact.
    static constexpr float kLevelOffset = 1024.0f;
    __device__ static __forceinline__ __half pix(uint32_t i) { return __ushort_as_half(static_cast<unsigned short>(0x6400u | i)); }
#else
    // study build: an integer-to-half conversion per pixel (the same exact value of I - level)
    static constexpr float kLevelOffset = 0.0f;
    __device__ static __forceinline__ __half pix(uint32_t i) { return __uint2half_rn(i); }
#endif
    __device__ static __forceinline__ __half from_f(float v) { return __float2half_rn(v); }
    __device__ static __forceinline__ float to_f(__half v) { return __half2float(v); }
    __device__ static __forceinline__ h2 pack(__half a, __half b) { return __halves2half2(a, b); }
    __device__ static __forceinline__ h2 from_f2(float a, float b) { return __floats2half2_rn(a, b); }
    __device__ static __forceinline__ float lo(h2 v) { return __low2float(v); }
    __device__ static __forceinline__ float hi(h2 v) { return __high2float(v); }
    __device__ static __forceinline__ __half lo_h(h2 v) { return __low2half(v); }
    __device__ static __forceinline__ __half hi_h(h2 v) { return __high2half(v); }
};

template <>
struct HalfOps<__nv_bfloat16> {
    using h2 = __nv_bfloat162;
    static constexpr float kLevelOffset = 0.0f;
    __device__ static __forceinline__ __nv_bfloat16 pix(uint32_t i) { return __float2bfloat16_rn(static_cast<float>(i)); }
    __device__ static __forceinline__ __nv_bfloat16 from_f(float v) { return __float2bfloat16_rn(v); }
    __device__ static __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
    __device__ static __forceinline__ h2 pack(__nv_bfloat16 a, __nv_bfloat16 b) { return __halves2bfloat162(a, b); }
    __device__ static __forceinline__ h2 from_f2(float a, float b) { return __floats2bfloat162_rn(a, b); }
    __device__ static __forceinline__ float lo(h2 v) { return __low2float(v); }
    __device__ static __forceinline__ float hi(h2 v) { return __high2float(v); }
    __device__ static __forceinline__ __nv_bfloat16 lo_h(h2 v) { return __low2bfloat16(v); }
    __device__ static __forceinline__ __nv_bfloat16 hi_h(h2 v) { return __high2bfloat16(v); }
};

// The half-form sum (reading C10): each template row summed left to right, then the row
// sums added top to bottom, every addition in the lane type (F16, the paper's half
// accumulation) or in FP32 (BF16 and PF_FLAG_ACCUM32) and the result rounded to the lane
// type.  Every route below (a thread over the frame, a thread over staged terms, a warp
// over the frame) performs exactly these operations in this order.
template <typename H>
struct HalfLik {
    H kap, bgo, fgo;
    bool half_acc;
    __device__ __forceinline__ H term(uint32_t i) const {
        const H h = HalfOps<H>::pix(i);
        const H a = __hmul(__hsub(h, bgo), kap);
        const H b = __hmul(__hsub(h, fgo), kap);
        return __hfma(a, a, __hneg(__hmul(b, b)));
    }
    // direct evaluation from the frame by one thread
    __device__ H at(const FrameView &f, const int8_t *w, int px, int py) const {
        H hacc = HalfOps<H>::from_f(0.0f);
        float facc = 0.0f;
        for (int dy = -f.r; dy <= f.r; ++dy) {
            const int hw = w[dy + f.r];
            H hrow = HalfOps<H>::from_f(0.0f);
            float frow = 0.0f;
            for (int dx = -hw; dx <= hw; ++dx) {
                const H tm = term(f.at(px + dx, py + dy));
                if (half_acc) hrow = __hadd(hrow, tm); else frow += HalfOps<H>::to_f(tm);
            }
            if (half_acc) hacc = __hadd(hacc, hrow); else facc += frow;
        }
        return half_acc ? hacc : HalfOps<H>::from_f(facc);
    }
    // from per-pixel terms staged in shared memory (row pitch rw, template centred at
    // column cx + r, row cy + r)
    __device__ H from_terms(const H *tm, int rw, const int8_t *w, int r, int cx, int cy) const {
        if (half_acc) {
            H acc = HalfOps<H>::from_f(0.0f);
            for (int i = 0; i <= 2 * r; ++i) {
                const int hw = w[i];
                const H *row = tm + (cy + i) * rw + cx + r;
                H rs = HalfOps<H>::from_f(0.0f);
#pragma unroll 4
                for (int dx = -hw; dx <= hw; ++dx) rs = __hadd(rs, row[dx]);
                acc = __hadd(acc, rs);
            }
            return acc;
        }
        float acc = 0.0f;
        for (int i = 0; i <= 2 * r; ++i) {
            const int hw = w[i];
            const H *row = tm + (cy + i) * rw + cx + r;
            float rs = 0.0f;
#pragma unroll 4
            for (int dx = -hw; dx <= hw; ++dx) rs += HalfOps<H>::to_f(row[dx]);
            acc += rs;
        }
        return HalfOps<H>::from_f(acc);
    }
    // by one warp from the frame: lane l sums rows l, l + 32, ... (each left to right);
    // lane 0 adds the row sums top to bottom.  Valid in lane 0.
    __device__ H warp_at(const FrameView &f, const int8_t *w, int px, int py) const {
        const int lane = threadIdx.x & 31, nrow = 2 * f.r + 1;
        H hacc = HalfOps<H>::from_f(0.0f);
        float facc = 0.0f;
        for (int base = 0; base < nrow; base += 32) {
            const int i = base + lane;
            H hrow = HalfOps<H>::from_f(0.0f);
            float frow = 0.0f;
            if (i < nrow) {
                const int dy = i - f.r;
                const int hw = w[i];
                for (int dx = -hw; dx <= hw; ++dx) {
                    const H tm = term(f.at(px + dx, py + dy));
                    if (half_acc) hrow = __hadd(hrow, tm); else frow += HalfOps<H>::to_f(tm);
                }
            }
            const int n = nrow - base < 32 ? nrow - base : 32;
            for (int k = 0; k < n; ++k) {
                if (half_acc) {
                    const H v = __shfl_sync(0xffffffffu, hrow, k);
                    hacc = __hadd(hacc, v);
                } else {
                    facc += __shfl_sync(0xffffffffu, frow, k);
                }
            }
        }
        return half_acc ? hacc : HalfOps<H>::from_f(facc);
    }
};

// The half-form constants of a tracker: kappa, and the two levels offset so that a pixel
// enters half arithmetic without a conversion (HalfOps<H>::pix).
template <typename H>
__device__ __forceinline__ HalfLik<H> half_lik(const TrackerDev &T) {
    HalfLik<H> hk;
    const float lo = HalfOps<H>::kLevelOffset;
    hk.kap = HalfOps<H>::from_f(T.kappa);
    hk.bgo = HalfOps<H>::from_f(lo + T.bg_f);
    hk.fgo = HalfOps<H>::from_f(lo + T.fg_f);
    hk.half_acc = std::is_same<H, __half>::value && !(T.flags & 0x2u);
    return hk;
}

// Integer disk sum by one warp (lanes take template rows; exact, so the order is free).
__device__ __forceinline__ uint32_t warp_disk_sum(const FrameView &f, const int8_t *w, int px, int py) {
    const int lane = threadIdx.x & 31, nrow = 2 * f.r + 1;
    uint32_t s = 0;
    for (int i = lane; i < nrow; i += 32) {
        const int hw = w[i];
        for (int dx = -hw; dx <= hw; ++dx) s += f.at(px + dx, py + i - f.r);
    }
    return __reduce_add_sync(0xffffffffu, s);
}

// The likelihood of a pixel straight from the frame, by one lane.
template <int P, typename L>
__device__ __forceinline__ L direct_likelihood(const TrackerDev &T, const FrameView &f, const int8_t *w, int px, int py) {
    using acc_t = typename Prec<P>::acc_t;
    if constexpr (Prec<P>::kHalf) {
        return half_lik<L>(T).at(f, w, px, py);
    } else {
        constexpr bool kF64 = sizeof(acc_t) == 8;
        return lik_from_sum<acc_t>(disk_sum(f, w, px, py), kF64 ? static_cast<acc_t>(T.c1) : static_cast<acc_t>(T.c1f),
                                   kF64 ? static_cast<acc_t>(T.c2 * T.D) : static_cast<acc_t>(T.c2Df),
                                   kF64 ? static_cast<acc_t>(T.den) : static_cast<acc_t>(T.denf));
    }
}

// The direct route of the offspring loop: the likelihoods of pixels outside the tile's window,
// straight from the frame, for all the lanes of `act` that are in the loop's iteration together
// (miss: which of the lane's two particles need one, 1 and 2).
// Few of them (a draw beyond the window's 3.5 sigma): the lanes take the template's rows of one
// particle after another, so a particle costs one or two round trips of loads in flight
// together; its own lane alone read |D| pixels in a nearly serial chain, microseconds
// that the whole block waited for at the next barrier.  The sums are HalfLik::at's (rows left
// to right, row sums top to bottom) and disk_sum's, so the bits are.  F16, the paper's motion
// model at 65536 particles (about four such particles a tile): 20.1 -> 18.6 us a frame.
// Many (no window fits a table: every draw, from about 10 px of noise on): each lane its own, where
// none waits for another's and the chains of a warp run side by side.  Every particle of 65536,
// noise 10, radius 5, one after another -> each lane its own: F16 807 -> 108 us a frame, F32 367 ->
// 98, REF64 409 -> 99; 200003, radius 40: F16 15 930 -> 5390, F32 10 970 -> 4570.
// So a warp's 64 particles one after another cost 7.5 (F16) and 3.7 (F32) times as much as at once
// with 81 pixels, 3.0 and 2.4 with 5025: the line lies at an eighth of them in half and
// at a quarter otherwise.
template <int P> constexpr int kDirectShare = Prec<P>::kHalf ? 4 : 2;   // per lane in the iteration
template <int P, typename L>
__device__ __forceinline__ void direct_likelihoods(const TrackerDev &T, const FrameView &f, const int8_t *w, unsigned act,
                                                   int miss, int px0, int py0, int px1, int py1, L &l0, L &l1) {
    using acc_t = typename Prec<P>::acc_t;
    const int lane = threadIdx.x & 31, n = __popc(act), rank = __popc(act & ((1u << lane) - 1u));
    if (kDirectShare<P> * (__popc(__ballot_sync(act, miss != 0)) + __popc(__ballot_sync(act, miss == 3))) > n) {
        for (int side = 1; side <= 2; ++side) {
            if (!(miss & side)) continue;
            const L v = direct_likelihood<P, L>(T, f, w, side == 1 ? px0 : px1, side == 1 ? py0 : py1);
            if (side == 1) l0 = v; else l1 = v;
        }
        return;
    }
    const int nrow = 2 * f.r + 1;
    for (unsigned left; (left = __ballot_sync(act, miss != 0)) != 0u;) {
        const int src = __ffs(static_cast<int>(left)) - 1;
        const bool first = (miss & 1) != 0;
        const int px = __shfl_sync(act, first ? px0 : px1, src), py = __shfl_sync(act, first ? py0 : py1, src);
        L v;
        if constexpr (Prec<P>::kHalf) {
            const HalfLik<L> hk = half_lik<L>(T);
            L hacc = HalfOps<L>::from_f(0.0f);
            float facc = 0.0f;
            for (int base = 0; base < nrow; base += n) {
                const int i = base + rank;
                L hrow = HalfOps<L>::from_f(0.0f);
                float frow = 0.0f;
                if (i < nrow) {
                    const int hw = w[i];
#pragma unroll 4
                    for (int dx = -hw; dx <= hw; ++dx) {
                        const L tm = hk.term(f.at(px + dx, py + i - f.r));
                        if (hk.half_acc) hrow = __hadd(hrow, tm); else frow += HalfOps<L>::to_f(tm);
                    }
                }
                unsigned lanes = act;
                for (int k = base; k < base + n && k < nrow; ++k) {
                    const int from = __ffs(static_cast<int>(lanes)) - 1;
                    lanes &= lanes - 1u;
                    if (hk.half_acc) hacc = __hadd(hacc, __shfl_sync(act, hrow, from));
                    else facc += __shfl_sync(act, frow, from);
                }
            }
            v = hk.half_acc ? hacc : HalfOps<L>::from_f(facc);
        } else {
            constexpr bool kF64 = sizeof(acc_t) == 8;
            uint32_t s = 0;
            for (int i = rank; i < nrow; i += n) {
                const int hw = w[i];
#pragma unroll 4
                for (int dx = -hw; dx <= hw; ++dx) s += f.at(px + dx, py + i - f.r);
            }
            v = lik_from_sum<acc_t>(__reduce_add_sync(act, s), kF64 ? static_cast<acc_t>(T.c1) : static_cast<acc_t>(T.c1f),
                                    kF64 ? static_cast<acc_t>(T.c2 * T.D) : static_cast<acc_t>(T.c2Df),
                                    kF64 ? static_cast<acc_t>(T.den) : static_cast<acc_t>(T.denf));
        }
        if (lane == src) {
            if (first) l0 = v; else l1 = v;
            miss &= first ? 2 : 0;
        }
    }
}

// Shared memory of the step kernel (dynamic: sizeof(StepSmem<P>) bytes).
template <int P>
struct __align__(16) StepSmem {
    using Tr = Prec<P>;
    using pos_t = typename Tr::pos_t;
    using lik_t = typename Tr::lik_t;
    using acc_t = typename Tr::acc_t;
    // ancestor positions of the tile (previous frame): x then y, or, in F16 / BF16, one word a
    // particle (x in the low half), so that the offspring loop gathers both with one load
    alignas(16) pos_t a[2 * kTile];
    lik_t table[kTableMax];   // likelihood of each pixel of the tile's window
    union {
        uint16_t pre[kRoiMax];      // integer form: row prefix sums of the staged region
        lik_t term[Tr::kHalf ? kRoiMax : 1];   // half form: per-pixel Eq. 4 terms of the staged region
        // F16 half accumulation, staged regions of up to kRoiMax / 2 pixels: the terms of
        // pixels x and x + 1 of a row side by side, so one half2 addition advances the sums
        // of two neighbouring cells
        __half2 term2[P == 2 ? kRoiMax / 2 : 1];
    } u;
    alignas(16) int warp_imax[kWarps];
    alignas(16) acc_t warp_sum[kWarps];
    alignas(16) acc_t warp_max[kWarps];
    alignas(16) float box[kWarps][4];
    U128 red128[kWarps];
    alignas(16) int warp_incl[kWarps];
    Stats<acc_t> red[kWarps];
    U128 agg_x;               // the tile aggregate (fixed point)
    int jbeg, jend;           // the tile's offspring are j in [jbeg, jend)
    double u0d;               // resampling offset u0 of the previous frame
    float u0f;
    alignas(16) uint32_t rk[20];   // Philox round keys of the tracker
    uint32_t skeys[4];        // stratified resampling: key_lo, key_hi, frame t - 1, tracker id
    int win_x0, win_y0, win_w, win_h;   // likelihood table window (win_w = 0: none)
    int qmin;
    uint32_t ticket;
    uint32_t last;
    int cached;               // tracker whose descriptor / state / frame are loaded below
    TrackerDev trk;
    TrackerState st;
    FrameRef fr;
    // last: the strata counts and the ancestor map of the step mode, whose row sums lie over both;
    // the other modes allocate the first half, their map (see counts_array)
    alignas(16) int32_t tail[2 * kTile];
};

// Block-wide merge of per-thread stats, result valid in thread 0.  Each warp takes its
// max of m (butterfly), rescales every lane's sums to it (one exp a lane) and adds them
// (butterfly); warp 0 does the same over the warps' results.  Max, rescale and sums run
// in a fixed order, so the result is deterministic.  The caller synchronises before
// sm.red is written again.
// Warp max / min of floats by redux.sync on an order-preserving integer image (the sign bit
// kept, the other bits flipped for negative values); exact, -inf included (no NaN here).
__device__ __forceinline__ int float_key(float x) {
    const int b = __float_as_int(x);
    return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float key_float(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }
__device__ __forceinline__ float warp_max(float x) { return key_float(__reduce_max_sync(0xffffffffu, float_key(x))); }
__device__ __forceinline__ float warp_min(float x) { return key_float(__reduce_min_sync(0xffffffffu, float_key(x))); }
__device__ __forceinline__ double warp_max(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double y = __shfl_xor_sync(0xffffffffu, x, o);
        x = above(y, x) ? y : x;
    }
    return x;
}

template <int P, typename A>
__device__ __forceinline__ Stats<A> warp_stats(Stats<A> v) {
    constexpr bool F = Prec<P>::kHalf;
    const A m = warp_max(v.m);
    if (is_neg_inf(m)) return Stats<A>{m, 0, 0, 0};
    const A sc = is_neg_inf(v.m) ? static_cast<A>(0) : wexp<F>(v.m - m);
    A s = mul_rn(v.s, sc), sx = mul_rn(v.sx, sc), sy = mul_rn(v.sy, sc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s = add_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
        sx = add_rn(sx, __shfl_xor_sync(0xffffffffu, sx, o));
        sy = add_rn(sy, __shfl_xor_sync(0xffffffffu, sy, o));
    }
    return Stats<A>{m, s, sx, sy};
}

// Warp-level min / max of a bounding box (x0, x1, y0, y1), returned to every lane; lane 0
// also leaves it in sm.box for merge_warp_boxes after the next barrier.
template <int P>
__device__ __forceinline__ float4 warp_box(float4 b, StepSmem<P> &sm) {
    b = make_float4(warp_min(b.x), warp_max(b.y), warp_min(b.z), warp_max(b.w));
    if ((threadIdx.x & 31) == 0) *reinterpret_cast<float4 *>(sm.box[threadIdx.x >> 5]) = b;
    return b;
}
// The block's box from the warps' boxes in sm.box, by one whole warp (lane w reads warp w's),
// returned to every lane of that warp.
template <int P>
__device__ __forceinline__ float4 merge_warp_boxes(const StepSmem<P> &sm) {
    const int lane = threadIdx.x & 31;
    const float4 b = lane < kWarps ? *reinterpret_cast<const float4 *>(sm.box[lane])
                                   : make_float4(FLT_MAX, -FLT_MAX, FLT_MAX, -FLT_MAX);
    return make_float4(warp_min(b.x), warp_max(b.y), warp_min(b.z), warp_max(b.w));
}

template <int P, typename A>
__device__ Stats<A> block_stats(Stats<A> v, StepSmem<P> &sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_stats<P>(v);
    if (lane == 0) sm.red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = (lane < kWarps) ? sm.red[lane] : Stats<A>{neg_inf<A>(), 0, 0, 0};
        v = warp_stats<P>(v);
    }
    return v;
}

// Decoupled lookback over the tracker's earlier tiles, kThreads tiles per round (thread
// i inspects tile base - i).  Sums the fixed-point aggregates back to the nearest tile
// that has published its inclusive prefix.  Whole block, one barrier per round; the
// result is valid in every thread.
template <int P>
__device__ U128 lookback(const LookbackDesc *look, int lt, uint64_t tag, TrackerState *st, StepSmem<P> &sm) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    U128 total{0ull, 0ull};
    for (int base = lt - 1; base >= 0; base -= kThreads) {
        const int idx = base - tid;
        uint32_t f = 0u;
        U128 v{0ull, 0ull};
        if (idx >= 0) {
            f = wait_desc(&look[idx], tag, st, v);
            if (f == 0u) { f = 2u; v = U128{0ull, 0ull}; }   // timed out: an inclusive zero (step flagged invalid)
        }
        // the warp's nearest inclusive predecessor (lowest lane); lanes past it contribute 0
        const uint32_t incl = __ballot_sync(0xffffffffu, f == 2u);
        const int first = incl ? __ffs(static_cast<int>(incl)) - 1 : 32;
        if (lane > first) v = U128{0ull, 0ull};
        if (base - warp * 32 >= 0) {          // the warp has predecessors in this round
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v = add128(v, shfl_down128(v, o));
        }
        if (lane == 0) { sm.red128[warp] = v; sm.warp_incl[warp] = incl != 0u; }
        const int found = __syncthreads_or(incl != 0u);
        {   // every warp: the warp sums up to the first warp with an inclusive predecessor
            U128 x{0ull, 0ull};
            int inc = 0;
            if (lane < kWarps) { x = sm.red128[lane]; inc = sm.warp_incl[lane]; }
            const uint32_t im = __ballot_sync(0xffffffffu, inc != 0);
            const int fw = im ? __ffs(static_cast<int>(im)) - 1 : 32;
            if (lane > fw) x = U128{0ull, 0ull};
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) x = add128(x, shfl_xor128(x, o));
            total = add128(total, x);
        }
        if (found) break;
        __syncthreads();           // red128 is rewritten by the next round
    }
    return total;
}

// First index e in [0, n) with J[e] > j (J non-decreasing, J[n-1] > j).
__device__ __forceinline__ int upper_index(const int32_t *J, int n, int j) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (J[mid] > j) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// The new state from a tracker's merged statistics (in every lane of the first warp).
template <int P, typename A>
__device__ __forceinline__ void finish_tracker(const TrackerDev &T, TrackerState *st, StepSmem<P> &sm, Stats<A> v,
                                               float4 bb, double *est_out, bool track_box) {
    using acc_t = A;
    constexpr bool kF64 = sizeof(acc_t) == 8;
    if (threadIdx.x < 32) {
        // The new state, from the block's statistics (thread 0's, broadcast) and this launch's
        // starting state (the copy in shared memory, which no tile changes), written field by
        // field with stores only by four lanes in parallel: lane 0 the x estimate and
        // anchors, lane 1 the y ones, lane 2 the weight scalars, lane 3 the rest.  The status
        // word is not written (another tile may have raised it).
        const int lane = threadIdx.x;
        Stats<acc_t> r;
        r.m = __shfl_sync(0xffffffffu, v.m, 0);
        r.s = __shfl_sync(0xffffffffu, v.s, 0);
        r.sx = __shfl_sync(0xffffffffu, v.sx, 0);
        r.sy = __shfl_sync(0xffffffffu, v.sy, 0);
        const TrackerState &o = sm.st;
        const int64_t slot = (o.t >= 0 && o.t < 0x7fffffffll)
                                 ? static_cast<int64_t>(static_cast<uint32_t>(o.t) % static_cast<uint32_t>(T.est_cap))
                                 : o.t % T.est_cap;
        if (lane < 2) {
            const bool ly = lane == 1;
            const acc_t rs = ly ? r.sy : r.sx;
            const double on = ly ? o.ny : o.nx;        // the anchor the positions were written against
            const int32_t oni = ly ? o.nyi : o.nxi;
            double e, nn;
            int32_t ni;
            if constexpr (kF64) {
                e = on + rs / r.s;
                nn = on;
                if (isfinite(e) && fabs(e) < 1.0e6) nn = floor(e) + ((e - floor(e)) >= 0.5 ? 1.0 : 0.0);
                ni = static_cast<int32_t>(nn);
            } else {
                // FP32 quotient; the next anchor in FP32 / integers (FP64 only to widen the
                // results the host reads)
                const float q = rs / r.s;
                const float fq = static_cast<float>(oni) + q;
                ni = oni;
                if (isfinite(fq) && fabsf(fq) < 1.0e6f) ni = __float2int_rd(fq + 0.5f);
                nn = static_cast<double>(ni);
                e = on + static_cast<double>(q);
            }
            if (ly) { st->ay = on; st->ayi = oni; st->ny = nn; st->nyi = ni; st->est_y = e; }
            else { st->ax = on; st->axi = oni; st->nx = nn; st->nxi = ni; st->est_x = e; }
            T.est_ring[2 * slot + lane] = e;
            if (est_out) est_out[lane] = e;
        } else if (lane == 2) {
            const acc_t inv = static_cast<acc_t>(1) / r.s;
            st->M = static_cast<double>(r.m);
            st->S = static_cast<double>(r.s);
            st->invS = static_cast<double>(inv);
            st->M_f = static_cast<float>(r.m);
            st->invS_f = static_cast<float>(inv);
            T.stat_ring[2 * slot] = static_cast<double>(r.m);
            T.stat_ring[2 * slot + 1] = static_cast<double>(r.s);
        } else if (lane == 3) {
            // the box of the new positions sizes the next step's tracker table (unknown if
            // the launch did not track it, or empty)
            const bool box_ok = track_box && bb.x <= bb.y && bb.z <= bb.w;
            st->bb_x0 = box_ok ? bb.x : __int_as_float(0x7fc00000);
            st->bb_x1 = box_ok ? bb.y : __int_as_float(0x7fc00000);
            st->bb_y0 = box_ok ? bb.z : __int_as_float(0x7fc00000);
            st->bb_y1 = box_ok ? bb.w : __int_as_float(0x7fc00000);
            st->t = o.t + 1;
            st->epoch = o.epoch + 1u;
            // every tile of this launch has counted; the next launch sees the reset after the
            // kernel boundary
            *T.done = 0u;
        }
    }
}

// The tile that completed the tracker: all partials merged (one per thread, all loads in
// flight, then the block merge: deterministic), then the new state.
template <int P>
__device__ void finalize_tracker(const TrackerDev &T, TrackerState *st, StepSmem<P> &sm, double *est_out,
                                 bool track_box) {
    using acc_t = typename Prec<P>::acc_t;
    constexpr bool kF64 = sizeof(acc_t) == 8;
    constexpr bool F = Prec<P>::kHalf;
    Stats<acc_t> v{neg_inf<acc_t>(), 0, 0, 0};
    float4 bb = make_float4(FLT_MAX, -FLT_MAX, FLT_MAX, -FLT_MAX);
    const uint64_t tg = partial_tag(sm.st.epoch);
    for (int i = threadIdx.x; i < T.ntiles; i += kThreads) {
        Stats<acc_t> w;
        uint64_t q[8];
        if constexpr (kF64) {
            const double *p = T.part[i].d;
            w = Stats<acc_t>{__ldcg(p + 0), __ldcg(p + 1), __ldcg(p + 2), __ldcg(p + 3)};
            const unsigned long long *pb = reinterpret_cast<const unsigned long long *>(T.part[i].b);
#pragma unroll
            for (int k = 0; k < 4; ++k) q[4 + k] = track_box ? __ldcg(pb + k) : 0ull;
        } else {
            wait_partial(&T.part[i], tg, st, q, track_box);
            w = Stats<acc_t>{__uint_as_float(static_cast<uint32_t>(q[0])), __uint_as_float(static_cast<uint32_t>(q[1])),
                             __uint_as_float(static_cast<uint32_t>(q[2])), __uint_as_float(static_cast<uint32_t>(q[3]))};
        }
        v = stats_merge<F>(v, w);
        bb.x = fminf(bb.x, __uint_as_float(static_cast<uint32_t>(q[4])));
        bb.y = fmaxf(bb.y, __uint_as_float(static_cast<uint32_t>(q[5])));
        bb.z = fminf(bb.z, __uint_as_float(static_cast<uint32_t>(q[6])));
        bb.w = fmaxf(bb.w, __uint_as_float(static_cast<uint32_t>(q[7])));
    }
    __syncthreads();              // (sm.red and sm.box still hold the tile's own)
    if (track_box) warp_box(bb, sm);
    v = block_stats<P>(v, sm);
    if (track_box && threadIdx.x < 32) bb = merge_warp_boxes(sm);
    finish_tracker<P>(T, st, sm, v, bb, est_out, track_box);
}

// The tracker's likelihood table of this launch into the tile's shared-memory table: each
// cell's word if it carries this launch's tag, else the cell computed here (the builder
// has not reached it yet; the same operations give the same bits).
template <int P, typename A>
__device__ __forceinline__ void fetch_table(const TrackerDev &T, StepSmem<P> &sm, int gx0, int gy0, int gw, int cells,
                                            const FrameView &fv, A c1, A c2D, A den, TrackerState *st) {
    (void)st;
    using H = typename std::conditional<Prec<P>::kHalf, typename Prec<P>::pos_t, __half>::type;
    const uint64_t gtag = static_cast<uint64_t>(sm.st.epoch % 0x7fffffffu + 1u) << 32;
    for (int c = threadIdx.x; c < cells; c += kThreads) {
        const uint64_t v = __ldcg(reinterpret_cast<const unsigned long long *>(T.gtab) + PF_IDX(c, kTableMax));
        uint32_t payload;
        const bool built = (v & 0xffffffff00000000ull) == gtag;
        if constexpr (Prec<P>::kHalf) {
            if (built) {
                payload = static_cast<uint32_t>(v);
            } else {
                const H h = half_lik<H>(T).at(fv, sm.trk.w, gx0 + c % gw, gy0 + c / gw);
                payload = static_cast<uint32_t>(*reinterpret_cast<const unsigned short *>(&h));
            }
            const unsigned short bits = static_cast<unsigned short>(payload);
            sm.table[PF_IDX(c, kTableMax)] = *reinterpret_cast<const H *>(&bits);
        } else {
            payload = built ? static_cast<uint32_t>(v) : disk_sum(fv, sm.trk.w, gx0 + c % gw, gy0 + c / gw);
            sm.table[PF_IDX(c, kTableMax)] = lik_from_sum<A>(payload, c1, c2D, den);
        }
    }
}

// The strata counts of a thread's elements (phase 1d): C_k of each element from the tile's
// local prefix loc[m] pinned to the exact boundaries excl / pend, and J = the number of
// strata points at or below C_k (elements past the tile's last repeat its count).  nrm is
// the saved 1/S (the naive study build: S itself).  Force-inlined so that loc and Jr stay in
// registers.
// The element loop holds no branch (systematic points): the phase is bound by instruction
// latency, and the eight independent counts overlap.  The tile's last element, whose prefix
// is the tile's end, and the tracker's last, whose CDF is 1, are set after the loop by the
// one thread that owns them.
template <typename A, typename Str>
__device__ __forceinline__ void strata_counts(const Str &str, const A (&loc)[kItems], int (&Jr)[kItems], A excl,
                                              A pend, A nrm, int eb, int cnt, int k0, int N, A *dbg_cdf,
                                              TrackerState *st) {
    (void)st;
    if (eb >= cnt) {   // (whole warps, but for one)
#pragma unroll
        for (int m = 0; m < kItems; ++m) Jr[m] = N;
        return;
    }
#ifdef PF_NAIVE_RESAMPLE
    const A Sdiv = nrm;
#else
    const A invS = nrm;
#endif
    // the normalised CDF cannot exceed 1; the FP32 scan can round above it
    A cprev = static_cast<A>(-1);
    int jprev = 0;
#pragma unroll
    for (int m = 0; m < kItems; ++m) {
        const A C = prefix_min(PF_NORM(prefix_min(add_rn(excl, loc[m]), pend)), static_cast<A>(1));
        if constexpr (Str::kReuse) {   // a count costs Philox blocks: repeated values reuse it
            Jr[m] = C == cprev ? jprev : str.count_le(C);
            cprev = C;
            jprev = Jr[m];
        } else {
            Jr[m] = str.count_le(C);
        }
    }
    const int last = cnt - 1 - eb;   // the tile's last element, if this thread owns it
    if (last < kItems) {
        const int J = (k0 + cnt == N) ? N : str.count_le(prefix_min(PF_NORM(pend), static_cast<A>(1)));
#pragma unroll
        for (int m = 0; m < kItems; ++m)
            if (m >= last) Jr[m] = J;
    }
    if (dbg_cdf) {
#pragma unroll
        for (int m = 0; m < kItems; ++m) {
            const int e = eb + m;
            A C = prefix_min(PF_NORM(e == cnt - 1 ? pend : prefix_min(add_rn(excl, loc[m]), pend)), static_cast<A>(1));
            if (k0 + e == N - 1) C = static_cast<A>(1);
            if (e < cnt) dbg_cdf[PF_IDX(k0 + e, N)] = C;
        }
    }
}

// The descriptor, state and frame reference of launch position ti (slot `slot`) into shared
// memory, by the whole block (the caller synchronises).  what & 1: the descriptor and the
// frame reference; what & 2: the state.
template <int P>
__device__ __forceinline__ void load_descriptor(const StepLaunch &Lp, int slot, int ti, StepSmem<P> &sm, int what) {
    const uint32_t *src_t = reinterpret_cast<const uint32_t *>(Lp.trk + slot);
    const uint32_t *src_s = reinterpret_cast<const uint32_t *>(Lp.states + slot);
    const uint32_t *src_f = reinterpret_cast<const uint32_t *>(Lp.frames + ti);
    uint32_t *dt = reinterpret_cast<uint32_t *>(&sm.trk);
    uint32_t *ds = reinterpret_cast<uint32_t *>(&sm.st);
    uint32_t *df = reinterpret_cast<uint32_t *>(&sm.fr);
    constexpr int nt = sizeof(TrackerDev) / 4, ns = sizeof(TrackerState) / 4, nf = sizeof(FrameRef) / 4;
    // state first: one pass of the block loads any of the three sets
    const int lo = (what & 2) ? 0 : ns, hi = (what & 1) ? ns + nt + nf : ns;
    for (int i = lo + threadIdx.x; i < hi; i += kThreads) {
        if (i < ns) ds[i] = __ldcg(src_s + i);
        else if (i < ns + nt) dt[i - ns] = __ldcg(src_t + i - ns);
        else df[i - ns - nt] = __ldcg(src_f + i - ns - nt);
    }
}

// Kernel modes: the step kernel (systematic and stratified trackers, every phase), and for
// multinomial trackers the CDF kernel (phase 1 up to the CDF, written to T.cdf) and the
// pull kernel (resampling from T.cdf, phases 2-5), launched in that order; the pull kernel
// also takes the Gumbel-max, Metropolis and rejection trackers (ancestors from T.anc).
constexpr int kModeStep = 0, kModeCdf = 1, kModePull = 2;
// The step kernel with the tracker table (phase 0) and the bounding box that sizes it: a
// separate instantiation, launched for a tracker of at least two waves of tiles, so that the
// common launch carries none of its code or registers.
constexpr int kModeStepBig = 3;

// Where a mode keeps J[e], the strata assigned to particles k0 .. k0 + e (cumulative), searched
// when a tile has more offspring than the map holds.  The step mode stores it always, in its
// own array: kept in registers until the tile's last count is known, it spills (2^20 F16
// 21.9 us a frame against 21.6, 65536 20.9 against 20.4).  The tracker-table mode keeps it and
// stores it over the map when it must (2^24 F16 259 us against 265).  The pull kernel keeps
// its ancestors' indices there; without the array its CTAs leave 16 KB more to the L1 that its
// searches run in (2^19 F16 50.8 us against 51.4).
template <int P, int kMode>
__device__ __forceinline__ int32_t *counts_array(StepSmem<P> &sm) {
    return sm.tail;
}
// Ancestor (tile element + 1) of each offspring.
template <int P, int kMode>
__device__ __forceinline__ uint16_t *map_array(StepSmem<P> &sm) {
    return reinterpret_cast<uint16_t *>(kMode == kModeStep ? sm.tail + kTile : sm.tail);
}
// Where the table's row sums lie while it is built: in the step mode in the counts' memory, not
// written before the table is read, and, if there are more, in the map's first half, which is
// cleared again behind them.  (An array of their own, 24 KB more a CTA, left the L1 28 KB an SM of
// 92: F16, noise 40, 65536 particles, radius 5, all scored from the frame, 297 us a frame against
// 202; 2^20 722 against 456; the same at noise 1.  A place that starts where the number of words says
// costs an address a load: BF16 300007 particles, radius 10, 17.0 against 16.6.)  In the pull
// mode the map, which has no use there but for the ancestors' indices when debug arrays are on.
template <int P>
__device__ __forceinline__ uint32_t *row_words(StepSmem<P> &sm) {
    return reinterpret_cast<uint32_t *>(sm.tail);
}
template <int P, int kMode> constexpr size_t smem_bytes() {
    return kMode == kModeStep ? sizeof(StepSmem<P>) : offsetof(StepSmem<P>, tail) + sizeof(int32_t) * kTile;
}
static_assert(sizeof(uint16_t) * kMapMax == sizeof(int32_t) * kTile, "the map and the counts are of one size");

// The half-form table of a window from the staged terms, by row sums.  A cell is the sum of its
// template rows top to bottom, each summed left to right (HalfLik); a row's sum depends only on
// its half-width, its place and its frame row, so rows of equal half-width (a class) are the
// same sum for every cell that has the row at some dy.  Phase A sums every (class, frame row,
// cell column) once, four classes at a time from one pass over the row's terms; phase B adds
// each cell's 2 r + 1 row sums.  Every cell performs the additions of HalfLik::from_terms in the
// same order (kPair: two neighbouring cells in the lanes of a half2, accumulated in half; else
// one cell a word, accumulated in FP32).  A disk of radius 5 has 4 classes for 11 rows (28
// additions instead of 81 a cell and row phase), radius 10 has 7 for 21 (95 instead of 317),
// and the row sums spread over every thread of the block where one thread a cell left most
// idle in a chain of |D| dependent additions.  Windows whose row sums do not fit are done in
// bands of `band` cell rows.  Measured us a
// frame, cells one by one -> row sums: BF16 300007 particles r = 10 20.9 -> 19.0, F16 4096
// particles r = 12 18.8 -> 16.1; r = 5, F16 2^20 particles 19.4 -> 18.9, 450001 15.8 -> 15.0.
template <int P, int kMode, bool kPair>
__device__ __forceinline__ void table_by_rows(StepSmem<P> &sm, int rw, int pw, int ww, int wh, int band,
                                              TrackerState *st) {
    (void)st;
    using H = typename Prec<P>::pos_t;
    using R = typename std::conditional<kPair, __half2, float>::type;
    const TrackerDev &T = sm.trk;
    const int r = T.r, ncls = T.ncls, tid = threadIdx.x;
    R *rows = reinterpret_cast<R *>(row_words(sm));
    constexpr int cap = kMode == kModeStep ? kRowWords : kMapMax / 2;   // words there
    const auto zero = [] { if constexpr (kPair) return __float2half2_rn(0.0f); else return 0.0f; };
    const auto add = [](R a, R b) { if constexpr (kPair) return __hadd2(a, b); else return a + b; };
    const auto term = [&](int i) {
        if constexpr (kPair) return sm.u.term2[PF_IDX(i, kRoiMax / 2)];
        else return HalfOps<H>::to_f(sm.u.term[PF_IDX(i, kRoiMax)]);
    };
    for (int y0 = 0; y0 < wh; y0 += band) {
        const int nb = wh - y0 < band ? wh - y0 : band, nr = nb + 2 * r;
        for (int i = tid; i < nr * pw; i += kThreads) {
            const int yy = i / pw, hp = i - yy * pw;
            const int base = (y0 + yy) * rw + (kPair ? 2 * hp : hp) + r;
            for (int c = 0; c < ncls; c += 4) {
                const int h0 = T.chw[c], h1 = T.chw[c + 1], h2 = T.chw[c + 2], h3 = T.chw[c + 3];
                R a0 = zero(), a1 = a0, a2 = a0, a3 = a0;
#pragma unroll 4
                for (int dx = -h0; dx <= h0; ++dx) {
                    const R t = term(base + dx);
                    const int ad = dx < 0 ? -dx : dx;
                    a0 = add(a0, t);
                    if (ad <= h1) a1 = add(a1, t);
                    if (ad <= h2) a2 = add(a2, t);
                    if (ad <= h3) a3 = add(a3, t);
                }
                const int o = (c * nr + yy) * pw + hp;
                rows[PF_IDX(o, cap)] = a0;
                if (h1 >= 0) rows[PF_IDX(o + nr * pw, cap)] = a1;
                if (h2 >= 0) rows[PF_IDX(o + 2 * nr * pw, cap)] = a2;
                if (h3 >= 0) rows[PF_IDX(o + 3 * nr * pw, cap)] = a3;
            }
        }
        __syncthreads();
        for (int i = tid; i < nb * pw; i += kThreads) {
            const int cy = i / pw, hp = i - cy * pw;
            R acc = zero();
#pragma unroll 4
            for (int k = 0; k <= 2 * r; ++k) acc = add(acc, rows[PF_IDX((T.rc[k] * nr + cy + k) * pw + hp, cap)]);
            if constexpr (kPair) {
                const int cx = 2 * hp, c = (y0 + cy) * ww + cx;
                sm.table[PF_IDX(c, kTableMax)] = __low2half(acc);
                if (cx + 1 < ww) sm.table[PF_IDX(c + 1, kTableMax)] = __high2half(acc);
            } else {
                sm.table[PF_IDX((y0 + cy) * ww + hp, kTableMax)] = HalfOps<H>::from_f(acc);
            }
        }
        if (y0 + band < wh) __syncthreads();   // (the next band rewrites the row sums)
    }
}

// Multinomial draws: for each of a thread's values u the first k with C_k >= u, eight searches in
// step (live: the thread has draws; a tile below kTile particles leaves whole warps without).  Three
// levels: the CDF at the end of every 64 entries, staged in shared memory (every
// 64 << lb beyond 2^20 particles; the memory of the positions, the table and the staging, not in
// use yet), searched by bisection without branches; the eight ends of 8 entries below the one
// found, read as whole sectors and counted; the eight entries below that, likewise.  The chain
// of dependent reads from L2 is two long, where a bisection below a coarse table took seven or
// eight, most of them a sector each.  C is non-decreasing and its last value is 1, so the index
// is that of a search of the whole CDF.  Measured us a frame: F16 2^19 particles 47.3 -> 41.1.
// (With the warps past a tile's end searching too, F16 1500001, of whose 4096 places a tile fills 2472,
// took 118 us against 103 before the levels; 94 without.)
template <int P>
__device__ __forceinline__ void cdf_search(const TrackerDev &T, const typename Prec<P>::acc_t (&u)[kItems], int (&k)[kItems],
                                           bool live, StepSmem<P> &sm, TrackerState *st) {
    using A = typename Prec<P>::acc_t;
    (void)st;
    constexpr int kCoarse = static_cast<int>(offsetof(StepSmem<P>, warp_imax) / sizeof(A));
    constexpr int kVec = 16 / static_cast<int>(sizeof(A));   // elements a 16-byte load
    const int N = static_cast<int>(T.N), n8 = static_cast<int>((T.N + 7) >> 3), n64 = static_cast<int>((T.N + 63) >> 6);
    const A *c64 = static_cast<const A *>(T.cdf64), *c8 = static_cast<const A *>(T.cdf8), *c1 = static_cast<const A *>(T.cdf);
    int lb = 0;
    while (((n64 - 1) >> lb) + 1 > kCoarse) ++lb;
    const int nb = ((n64 - 1) >> lb) + 1;
    A *cs = reinterpret_cast<A *>(&sm);
    for (int i = threadIdx.x; i < nb; i += kThreads) {
        const int64_t last = ((static_cast<int64_t>(i) + 1) << lb) - 1;
        cs[PF_IDX(i, kCoarse)] = __ldg(c64 + (last < n64 ? last : n64 - 1));
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < kItems; ++m) k[m] = 0;
    for (int w = live ? 1 << (31 - __clz(nb)) : 0; w > 0; w >>= 1) {   // k = coarse entries below u
#pragma unroll
        for (int m = 0; m < kItems; ++m) {
            const int q = k[m] + w;
            if (q <= nb && !(cs[PF_IDX(q - 1, kCoarse)] >= u[m])) k[m] = q;
        }
    }
    __syncthreads();                      // (the memory of cs is the tile's again)
    if (!live) return;
#pragma unroll
    for (int m = 0; m < kItems; ++m) k[m] <<= lb + 3;
    for (int w = 4 << lb; w >= 8; w >>= 1) {                // beyond 2^20 particles: down to 8 ends of 8
#pragma unroll
        for (int m = 0; m < kItems; ++m) {
            const int q = k[m] + w;
            if (q <= n8 && !(__ldg(c8 + PF_IDX(q - 1, n8)) >= u[m])) k[m] = q;
        }
    }
    // entries below u among c[k .. k + 8), n of them in all and room for a whole number of eights
    const auto count8 = [&](const A *c, int n) {
        const int starts = ((n + 7) & ~7) - 7;
        (void)starts;
#pragma unroll
        for (int g = 0; g < kItems; g += 4) {
            uint4 v[4][8 / kVec];
#pragma unroll
            for (int m = 0; m < 4; ++m)
#pragma unroll
                for (int i = 0; i < 8 / kVec; ++i) v[m][i] = __ldg(reinterpret_cast<const uint4 *>(c + PF_IDX(k[g + m], starts)) + i);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                int below = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    below += (k[g + m] + i < n && !(Bits<A>::get(v[m], i) >= u[g + m])) ? 1 : 0;
                k[g + m] += below;
            }
        }
    };
    count8(c8, n8);
#pragma unroll
    for (int m = 0; m < kItems; ++m) k[m] = (k[m] < n8 ? k[m] : n8 - 1) << 3;
    count8(c1, N);
#pragma unroll
    for (int m = 0; m < kItems; ++m) k[m] = k[m] < N ? k[m] : N - 1;
}

// One tile of a launch in mode kMode (trackers of the other modes are skipped).
template <int P, int kMode>
__device__ void run_tile(const StepLaunch &Lp, int g, StepSmem<P> &sm) {
    constexpr bool kPull = kMode == kModePull;
    using Tr = Prec<P>;
    using pos_t = typename Tr::pos_t;
    using lik_t = typename Tr::lik_t;
    using acc_t = typename Tr::acc_t;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // launch position of the tile, its first tile and its slot
    int ti = 0;
    if (Lp.ntrk > 1) {
        if (Lp.tile_trk) {
            ti = __ldg(&Lp.tile_trk[g]);
        } else {   // last position whose first tile is <= g
            int lo = 0, hi = Lp.ntrk - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (__ldg(&Lp.tile_prefix[mid]) <= g) lo = mid; else hi = mid - 1;
            }
            ti = lo;
        }
    }
    const int slot = Lp.slot_of ? __ldg(&Lp.slot_of[ti]) : ti;
    TrackerState *const st = Lp.states + slot;

    // ---- the tracker's descriptor, state and frame reference, loaded in one round trip
    // and kept for the CTA's later tiles of the same tracker (none of them changes
    // before the tracker's last tile of this launch has finished)
    if (ti != sm.cached) {
        load_descriptor(Lp, slot, ti, sm, 3);
        __syncthreads();
        if (tid == 0) sm.cached = ti;
    }
    const TrackerDev &T = sm.trk;
    if (!sm.fr.active) return;
    if (sm.st.status & kStatusTimeout) return;   // a failed step: results are invalid
    // (the host gives each launch only its own family's tiles; the CDF and pull kernels
    // check as well)
    if constexpr (kMode == kModeCdf) {
        if (T.resampler != kResampleMultinomial && T.resampler != kResampleShard) return;
    } else if constexpr (kMode == kModePull) {
        if (T.resampler != kResampleMultinomial && !ancestors_given(T.resampler)) return;
    }

    const int N = static_cast<int>(T.N);
    const int lt = g - (Lp.tile_prefix ? __ldg(&Lp.tile_prefix[ti]) : T.tile_begin);
    const int k0 = lt * T.tile;
    const int cnt = (N - k0) < T.tile ? (N - k0) : T.tile;
    const int64_t t = sm.st.t;
    if constexpr (kMode == kModeCdf) {
        if (t == 0) return;                        // frame 0 resamples nothing
    }
    const uint64_t dtag = desc_tag(sm.st.epoch);    // this launch's lookback tag
    constexpr bool kF64 = sizeof(acc_t) == 8;    // REF64; the other kernels use no FP64
    const int nxi = sm.st.nxi, nyi = sm.st.nyi;     // anchor of the offspring
    const int axi_anc = sm.st.axi, ayi_anc = sm.st.ayi;   // anchor of the ancestors
    const int in = static_cast<int>((t + 1) & 1), out = static_cast<int>(t & 1);
    acc_t *const dbg_cdf = static_cast<acc_t *>(T.dbg_cdf);
    LookbackDesc *const look = T.look;

    FrameView fv;
    fv.W = T.W; fv.H = T.H; fv.r = T.r;
    if (Lp.frame_override) { fv.p = Lp.frame_override; fv.pitch = Lp.pitch_override; }
    else {
        // a ring of staged frames, or a resident video
        const int64_t ft = sm.fr.ring ? mod_small(t, static_cast<uint32_t>(sm.fr.ring)) : t;
        fv.p = sm.fr.base + (sm.fr.stride ? ft * sm.fr.stride : 0);
        fv.pitch = sm.fr.pitch;
    }
    const int r = fv.r;

    using H = typename std::conditional<Tr::kHalf, pos_t, __half>::type;

    // ------------------------------------------------------------ 0. the tracker's table
    // A step launch of a tracker of at least two waves of tiles (twice as many tiles as the
    // launch has CTAs) whose previous positions' bounding box is known shares one likelihood
    // table per frame: the window every offspring can reach (the box widened by the drift
    // and the largest draw, kDrawMax sigma, plus one pixel of rounding), tabulated once in
    // device memory instead of once per tile.  (With a single wave the per-tile tables are
    // built while the tiles wait for their predecessors' aggregates, at no cost; so are the
    // builders' cells here, after the aggregate is published.)  The tracker's first
    // min(ntiles, grid) tiles build it, one cell per warp; every cell carries this launch's
    // tag, and a tile that finds a cell not yet built computes it itself (same operations,
    // same bits), so no tile waits for another.
    const bool track_box = kMode == kModeStepBig && T.gtab != nullptr &&
                           T.ntiles >= 2 * static_cast<int>(gridDim.x);
    bool gt = false;
    int gx0 = 0, gy0 = 0, gw = 0, gh = 0;
    if constexpr (kMode == kModeStepBig) {
        const float b0 = sm.st.bb_x0, b1 = sm.st.bb_x1, c0 = sm.st.bb_y0, c1b = sm.st.bb_y1;
        if (track_box && b0 <= b1 && c0 <= c1b && fabsf(b0) < 1.0e6f && fabsf(b1) < 1.0e6f &&
            fabsf(c0) < 1.0e6f && fabsf(c1b) < 1.0e6f) {
            const float mxr = fabsf(T.drift_xf) + kDrawMax * T.sigma_xf + 1.0f;
            const float myr = fabsf(T.drift_yf) + kDrawMax * T.sigma_yf + 1.0f;
            if (mxr < 4096.0f && myr < 4096.0f && b1 - b0 < 4096.0f && c1b - c0 < 4096.0f) {
                gx0 = static_cast<int>(floorf(b0 - mxr));
                gy0 = static_cast<int>(floorf(c0 - myr));
                gw = static_cast<int>(ceilf(b1 + mxr)) - gx0 + 1;
                gh = static_cast<int>(ceilf(c1b + myr)) - gy0 + 1;
                gt = static_cast<int64_t>(gw) * gh <= kTableMax;
            }
        }
        // the window for the rest of the tile (ordered by the barrier of phase 1b)
        if (gt && tid == 0) { sm.win_x0 = gx0; sm.win_y0 = gy0; sm.win_w = gw; sm.win_h = gh; }
    }

    // ------------------------------------------------------------ 1a. local scan of e
    acc_t loc[kItems];
    acc_t mex = static_cast<acc_t>(0);   // running max of the preceding lanes of the warp
    // bounding box of the ancestors with non-negligible weight (absolute pixel units)
    float bx0 = FLT_MAX, bx1 = -FLT_MAX, by0 = FLT_MAX, by1 = -FLT_MAX;
    const int eb = tid * kItems;  // blocked arrangement: thread tid owns elements eb .. eb+kItems-1
    if (!kPull && t > 0) {
        const lik_t *__restrict__ Lin = static_cast<const lik_t *>(T.pl[in]);
        const pos_t *__restrict__ Xin = static_cast<const pos_t *>(T.px[in]);
        const pos_t *__restrict__ Yin = static_cast<const pos_t *>(T.py[in]);
        const acc_t M = Lp.shard ? static_cast<acc_t>(Lp.g_M)
                                 : (kF64 ? static_cast<acc_t>(sm.st.M) : static_cast<acc_t>(sm.st.M_f));
        lik_t lv[kItems];
        // the thread's kItems positions as raw 16-byte vectors: copied to shared memory as
        // they are (the offspring loop reads its ancestors there), unpacked only where the
        // window's bounding box needs a value
        constexpr int kVp = static_cast<int>(sizeof(pos_t)) * kItems / 16;
        uint4 xr[kVp], yr[kVp];
        if (eb + kItems <= cnt) {
            // kItems consecutive values of each array, 16-byte aligned (k0 and eb are
            // multiples of kItems = 8 and the buffers are 16-byte aligned)
            load_items(lv, Lin + k0 + eb);
#pragma unroll
            for (int k = 0; k < kVp; ++k) {
                xr[k] = reinterpret_cast<const uint4 *>(Xin + k0 + eb)[k];
                yr[k] = reinterpret_cast<const uint4 *>(Yin + k0 + eb)[k];
            }
        } else {
            pos_t xv[kItems], yv[kItems];
#pragma unroll
            for (int m = 0; m < kItems; ++m) {
                const int e = eb + m;
                lv[m] = (e < cnt) ? Lin[k0 + e] : no_weight<lik_t>();
                xv[m] = (e < cnt) ? Xin[k0 + e] : pos_t{};
                yv[m] = (e < cnt) ? Yin[k0 + e] : pos_t{};
            }
#pragma unroll
            for (int k = 0; k < kVp; ++k) { xr[k] = make_uint4(0u, 0u, 0u, 0u); yr[k] = xr[k]; }
#pragma unroll
            for (int m = 0; m < kItems; ++m) { Bits<pos_t>::put(xr, m, xv[m]); Bits<pos_t>::put(yr, m, yv[m]); }
        }
        if constexpr (Tr::kHalf) {
            // eight words (x, y) from the four of x and the four of y
            uint4 *d = reinterpret_cast<uint4 *>(reinterpret_cast<uint32_t *>(sm.a) + eb);
            d[0] = make_uint4(__byte_perm(xr[0].x, yr[0].x, 0x5410), __byte_perm(xr[0].x, yr[0].x, 0x7632),
                              __byte_perm(xr[0].y, yr[0].y, 0x5410), __byte_perm(xr[0].y, yr[0].y, 0x7632));
            d[1] = make_uint4(__byte_perm(xr[0].z, yr[0].z, 0x5410), __byte_perm(xr[0].z, yr[0].z, 0x7632),
                              __byte_perm(xr[0].w, yr[0].w, 0x5410), __byte_perm(xr[0].w, yr[0].w, 0x7632));
        } else {
#pragma unroll
            for (int k = 0; k < kVp; ++k) {
                reinterpret_cast<uint4 *>(sm.a + eb)[k] = xr[k];
                reinterpret_cast<uint4 *>(sm.a + kTile + eb)[k] = yr[k];
            }
        }
        // clear the ancestor map (its heads are written after the strata are counted)
#pragma unroll
        for (int i = 0; i < kMapMax / 8 / kThreads; ++i)
            reinterpret_cast<uint4 *>(map_array<P, kMode>(sm))[tid + i * kThreads] = make_uint4(0u, 0u, 0u, 0u);
        const float sx = Tr::kHalf ? static_cast<float>(axi_anc) : 0.0f;
        const float sy = Tr::kHalf ? static_cast<float>(ayi_anc) : 0.0f;
        // FP64: a warp wholly past the tile's end (a REF64 tile may hold a quarter of kTile)
        // issues none of the arithmetic; its sums are 0, and no one reads its prefixes
        const bool live = !kF64 || warp * 32 * kItems < cnt;
        acc_t run = static_cast<acc_t>(0);
        if (!live) {
#pragma unroll
            for (int m = 0; m < kItems; ++m) loc[m] = static_cast<acc_t>(0);
        } else {
#pragma unroll
            for (int m = 0; m < kItems; ++m) {
                const acc_t v = wexp<Tr::kHalf>(to_acc(lv[m]) - M);   // 0 past the tile's end
                if (!gt && counts_in_box(v)) {
                    const float xa = to_f32(to_acc(Bits<pos_t>::get(xr, m))) + sx;
                    const float ya = to_f32(to_acc(Bits<pos_t>::get(yr, m))) + sy;
                    bx0 = fminf(bx0, xa); bx1 = fmaxf(bx1, xa);
                    by0 = fminf(by0, ya); by1 = fmaxf(by1, ya);
                }
                run = (m == 0) ? v : add_rn(run, v);
                loc[m] = run;
            }
        }
        // block exclusive scan of the thread totals
        acc_t x = run;
        if (live) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const acc_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
        }
        if (lane == 31) sm.warp_sum[warp] = x;
        if (kMode != kModeCdf && !gt) warp_box(make_float4(bx0, bx1, by0, by1), sm);   // (merged after the barrier)
        acc_t xex = __shfl_up_sync(0xffffffffu, x, 1);
        if (lane == 0) xex = static_cast<acc_t>(0);
        __syncthreads();
        acc_t wpre = static_cast<acc_t>(0);
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            if (kF64 && (w >= warp || !live)) break;   // (an FP64 addition not needed is not issued either)
            const acc_t v = sm.warp_sum[w];
            if (w < warp) wpre += v;
        }
        const acc_t off = wpre + xex;
        if (tid != 0 && live) {
#pragma unroll
            for (int m = 0; m < kItems; ++m) loc[m] = off + loc[m];
        }
        // The tile aggregate is the prefix at its last particle; the thread that holds it
        // publishes it at once (tile 0: as the inclusive prefix) and leaves it for thread 0,
        // which reads it after the next barrier.  (Every prefix of the tile is later clamped
        // to the exact boundary excl + aggregate.)
        {
            const int el = cnt - 1;
            if (el / kItems == tid) {
                acc_t a = loc[0];
#pragma unroll
                for (int m = 1; m < kItems; ++m)
                    if (m == el % kItems) a = loc[m];
                const U128 ax = to_fixed(a);
                desc_publish(&look[lt], lt == 0 ? 1 : 0, ax, dtag);
                sm.agg_x = ax;
            }
        }
        // running max across threads, which makes the tile-local prefix non-decreasing: the
        // warp part here, the block part after the next barrier (phase 1d)
        acc_t mx = loc[kItems - 1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const acc_t y = __shfl_up_sync(0xffffffffu, mx, o);
            if (lane >= o) mx = prefix_max(mx, y);
        }
        if (lane == 31) sm.warp_max[warp] = mx;
        mex = __shfl_up_sync(0xffffffffu, mx, 1);
    } else if (kPull && t > 0) {
        // The pull kernel's gather: offspring j = k0 + e takes the first particle a whose
        // CDF value reaches v_j (word j mod 4 of Philox(j / 4, t - 1, 1, tracker)); the
        // eight searches of a thread advance together.  a goes to J[e], the ancestor's
        // position (previous frame) to ax/ay[e], and the box of the gathered positions
        // sizes the likelihood window as in the step kernel.
        const pos_t *__restrict__ Xin = static_cast<const pos_t *>(T.px[in]);
        const pos_t *__restrict__ Yin = static_cast<const pos_t *>(T.py[in]);
        int lo[kItems];
        if (ancestors_given(T.resampler)) {
            // Gumbel-max, Metropolis, rejection: the ancestor kernel wrote every offspring's ancestor
#pragma unroll
            for (int m = 0; m < kItems; ++m) {
                const int a = (eb + m < cnt) ? __ldg(T.anc + PF_IDX(k0 + eb + m, N)) : 0;
                lo[m] = a > 0 ? a : 0;
            }
        } else {
            acc_t uq[kItems];
            const bool live = eb < cnt;
#pragma unroll
            for (int h = 0; h < kItems; h += 4) {
                const uint32_t blk = static_cast<uint32_t>(k0 + eb + h) >> 2;   // k0 + eb is a multiple of 8
                const uint4 wv = philox4x32_10(make_uint4(blk, static_cast<uint32_t>(t - 1), 1u, T.tracker_id),
                                               T.key_lo, T.key_hi);
                const uint32_t ws[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if constexpr (kF64) uq[h + i] = uniform_f64(ws[i]); else uq[h + i] = uniform_f32(ws[i]);
            }
            cdf_search<P>(T, uq, lo, live, sm, st);
        }
        const float sx = Tr::kHalf ? static_cast<float>(axi_anc) : 0.0f;
        const float sy = Tr::kHalf ? static_cast<float>(ayi_anc) : 0.0f;
#pragma unroll
        for (int m = 0; m < kItems; ++m) {
            const int e = eb + m;
            if (e < cnt) {
                const int a = lo[m] < N ? lo[m] : N - 1;
                const pos_t xa = Xin[PF_IDX(a, N)], ya = Yin[PF_IDX(a, N)];
                counts_array<P, kMode>(sm)[PF_IDX(e, kTile)] = a;
                sm.a[Tr::kHalf ? 2 * PF_IDX(e, kTile) : PF_IDX(e, kTile)] = xa;
                sm.a[Tr::kHalf ? 2 * PF_IDX(e, kTile) + 1 : kTile + PF_IDX(e, kTile)] = ya;
                const float xf = static_cast<float>(to_acc(xa)) + sx, yf = static_cast<float>(to_acc(ya)) + sy;
                bx0 = fminf(bx0, xf); bx1 = fmaxf(bx1, xf);
                by0 = fminf(by0, yf); by1 = fmaxf(by1, yf);
            }
        }
    } else {
        bx0 = bx1 = T.init_xf;
        by0 = by1 = T.init_yf;
    }

    // ------------------------------------------------------------ 1b. likelihood window
    // The bounding box of the heavy ancestors, widened by the drift and 3.5 sigma of the
    // draw: almost all of their offspring's pixels fall inside it.  Computed before the
    // lookback, so that the predecessors publish meanwhile.  (The pull kernel sizes it by
    // the gathered ancestors; the CDF kernel has none.)
    if constexpr (kMode != kModeCdf) {
        if (!gt && (kPull || t == 0)) {   // (else the scan's barrier ordered the warps' boxes)
            warp_box(make_float4(bx0, bx1, by0, by1), sm);
            __syncthreads();
        }
        // the tracker table's share of this tile (after the aggregate is out)
        if (gt) {
            const uint64_t gtag = static_cast<uint64_t>(sm.st.epoch % 0x7fffffffu + 1u) << 32;
            const int K = T.ntiles < static_cast<int>(gridDim.x) ? T.ntiles : static_cast<int>(gridDim.x);
            const int gcells = gw * gh;
            for (int c = lt + K * warp; lt < K && c < gcells; c += K * kWarps) {
                const int px = gx0 + c % gw, py = gy0 + c / gw;
                uint32_t payload;
                if constexpr (Tr::kHalf) {
                    const H v = half_lik<H>(T).warp_at(fv, T.w, px, py);
                    payload = static_cast<uint32_t>(*reinterpret_cast<const unsigned short *>(&v));
                } else {
                    payload = warp_disk_sum(fv, T.w, px, py);
                }
                if (lane == 0) st_relaxed_u64(&T.gtab[PF_IDX(c, kTableMax)], gtag | payload);
            }
        }
        if (tid >= 64 && tid < 84)   // the round keys of the propagation draws (ordered by the barrier below)
            sm.rk[tid - 64] = philox_round_key(tid - 64, T.key_lo, T.key_hi);
        // the resampling offset u0 of frame t - 1 (Philox tag 1, index 0), once per tile
        if (t > 0 && tid == 32) {
            const uint32_t w0 =
                philox4x32_10(make_uint4(0u, static_cast<uint32_t>(t - 1), 1u, T.tracker_id), T.key_lo, T.key_hi).x;
            if constexpr (kF64) sm.u0d = uniform_f64(w0); else sm.u0f = uniform_f32(w0);
            sm.skeys[0] = T.key_lo; sm.skeys[1] = T.key_hi;
            sm.skeys[2] = static_cast<uint32_t>(t - 1); sm.skeys[3] = T.tracker_id;
        }
        if (!gt && warp == 0) {   // the block's box, in every lane of warp 0
            const float4 b = merge_warp_boxes(sm);
            bx0 = b.x; bx1 = b.y; by0 = b.z; by1 = b.w;
        }
        if (!gt && tid == 0) {
            // Every draw lies within kDrawMax sigma: if that window takes a single pass of
            // the block, no offspring needs the direct route; otherwise kWindowSigmas
            // (the tracker's window policy may force either).
            float mxr = fabsf(T.drift_xf) + kDrawMax * T.sigma_xf + 1.0f;
            float myr = fabsf(T.drift_yf) + kDrawMax * T.sigma_yf + 1.0f;
            if (T.window == 1 ||
                (T.window == 0 && (ceilf(bx1 + mxr) - floorf(bx0 - mxr) + 1.0f) * (ceilf(by1 + myr) - floorf(by0 - myr) + 1.0f) >
                                      static_cast<float>(kThreads))) {
                mxr = fabsf(T.drift_xf) + kWindowSigmas * T.sigma_xf + 1.0f;
                myr = fabsf(T.drift_yf) + kWindowSigmas * T.sigma_yf + 1.0f;
            }
            int ww = 0, wh = 0, x0 = 0, y0 = 0;
            if (bx0 <= bx1 && by0 <= by1 && bx1 - bx0 < 4096.0f && by1 - by0 < 4096.0f &&
                fabsf(bx0) < 1.0e6f && fabsf(by0) < 1.0e6f && mxr < 4096.0f && myr < 4096.0f) {
                x0 = static_cast<int>(floorf(bx0 - mxr));
                y0 = static_cast<int>(floorf(by0 - myr));
                ww = static_cast<int>(ceilf(bx1 + mxr)) - x0 + 1;
                wh = static_cast<int>(ceilf(by1 + myr)) - y0 + 1;
                const int64_t cells = static_cast<int64_t>(ww) * wh;
                const int64_t roi = static_cast<int64_t>(ww + 2 * r + 1) * (wh + 2 * r);
                // (a table is built even for fewer particles than cells: 81-odd global loads
                // in a dependent chain per particle cost more than the table's shared loads)
                if (cells > kTableMax || roi > kRoiMax) { ww = 0; wh = 0; }
            }
            sm.win_x0 = x0; sm.win_y0 = y0; sm.win_w = ww; sm.win_h = wh;
        }
        __syncthreads();
    }
    const bool no_table = kMode == kModeCdf;
    const int wx0 = no_table ? 0 : sm.win_x0, wy0 = no_table ? 0 : sm.win_y0;
    const int ww = no_table ? 0 : sm.win_w, wh = no_table ? 0 : sm.win_h;
    const int cells = ww * wh;
    if (kMode != kModeCdf && T.dbg_win && tid == 0) {   // test hook: the tile's window
        int32_t *dw = T.dbg_win + PF_IDX(4 * lt, 4 * T.ntiles);
        dw[0] = wx0; dw[1] = wy0; dw[2] = ww; dw[3] = wh;
    }
    HalfLik<H> hk;
    if constexpr (Tr::kHalf) hk = half_lik<H>(T);

    const acc_t c1 = kF64 ? static_cast<acc_t>(T.c1) : static_cast<acc_t>(T.c1f);
    const acc_t c2D = kF64 ? static_cast<acc_t>(T.c2 * T.D) : static_cast<acc_t>(T.c2Df);
    const acc_t den = kF64 ? static_cast<acc_t>(T.den) : static_cast<acc_t>(T.denf);

    // ------------------------------------------------------------ 1c. likelihood table
    if constexpr (kMode != kModeCdf) if (cells > 0 && !gt) {
        // stage the frame region the window's templates cover (clamped to the frame);
        // warp w takes rows w, w + kWarps, ...; its lanes walk the row
        const int rx0 = wx0 - r, ry0 = wy0 - r, rw = ww + 2 * r, rh = wh + 2 * r;
        bool paired = false;
        if constexpr (P == 2) paired = hk.half_acc && rw * rh <= kRoiMax / 2;
        for (int yy = warp; yy < rh; yy += kWarps) {
            const uint8_t *row = fv.p + static_cast<int64_t>(clampi(ry0 + yy, 0, fv.H - 1)) * fv.pitch;
            if constexpr (P == 2) {
                if (paired) {
                    // term2[x] = (term x, term x + 1): the right neighbour from the next lane
                    // (lane 31 loads it; x + 1 = rw reads the clamped pixel after the row)
                    for (int x0 = 0; x0 < rw; x0 += 32) {
                        const int xx = x0 + lane;
                        const H tx = hk.term(__ldg(row + clampi(rx0 + xx, 0, fv.W - 1)));
                        H tn = __shfl_down_sync(0xffffffffu, tx, 1);
                        if (lane == 31) tn = hk.term(__ldg(row + clampi(rx0 + xx + 1, 0, fv.W - 1)));
                        if (xx < rw) sm.u.term2[PF_IDX(yy * rw + xx, kRoiMax / 2)] = __halves2half2(tx, tn);
                    }
                    continue;
                }
            }
            if constexpr (Tr::kHalf) {
                for (int xx = lane; xx < rw; xx += 32)
                    sm.u.term[PF_IDX(yy * rw + xx, kRoiMax)] = hk.term(__ldg(row + clampi(rx0 + xx, 0, fv.W - 1)));
            } else {
                // integer form: exclusive row prefix sums pre[y * (rw + 1) + x] = sum of the
                // row's pixels 0 .. x-1 (uint16, modular), by a warp scan per 32 columns
                const int last = yy * (rw + 1) + rw;      // the row's last prefix entry
                uint16_t *pre = sm.u.pre + (PF_IDX(last, kRoiMax) == last ? last - rw : 0);
                if (lane == 0) pre[0] = 0;
                uint32_t carry = 0;
                for (int x0 = 0; x0 < rw; x0 += 32) {
                    const int xx = x0 + lane;
                    uint32_t v = (xx < rw) ? static_cast<uint32_t>(__ldg(row + clampi(rx0 + xx, 0, fv.W - 1))) : 0u;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
                        if (lane >= o) v += y;
                    }
                    if (xx < rw) pre[xx + 1] = static_cast<uint16_t>(carry + v);
                    carry += __shfl_sync(0xffffffffu, v, 31);
                }
            }
        }
        __syncthreads();
        bool by_rows = false;
        if constexpr (Tr::kHalf) {
            const int pw = paired ? (ww + 1) >> 1 : (ww > 0 ? ww : 1);   // words a row
            // (the tracker-table mode has no memory for them: its map is in use; a tile of its
            // own is the exception there)
            int band = (kMode == kModeStep ? kRowWords : kMapMax / 2) / (T.ncls * pw) - 2 * r;
            if (band > wh) band = wh;
            // Row sums where they are the shorter way, block passes counted: about 10 issue slots
            // a term of a row (four classes at once) and 5 a row of a cell, against 4 a template
            // pixel (a dependent load and addition) and 10 a row, every cell by itself.  So by
            // rows except where the cells fill one pass and their rows several
            const int by_row = ((rh * pw - 1) / kThreads + 1) * (10 * T.row_terms + 30) +
                               ((wh * pw - 1) / kThreads + 1) * 5 * (2 * r + 1);
            const int by_cell = ((wh * pw - 1) / kThreads + 1) * (4 * T.D + 10 * (2 * r + 1));
            by_rows = (paired || !hk.half_acc) && (band == wh || band >= 4) && by_row < by_cell &&
                      (kMode == kModeStep || (kMode == kModePull && !T.dbg_anc));
            if (by_rows) {
                if constexpr (P == 2) {
                    if (paired) table_by_rows<P, kMode, true>(sm, rw, pw, ww, wh, band, st);
                }
                if (!paired) table_by_rows<P, kMode, false>(sm, rw, pw, ww, wh, band, st);
                if constexpr (kMode == kModeStep) {
                    if (T.ncls * pw * (band + 2 * r) > kTile) {   // the map's first half was in use
                        __syncthreads();
                        reinterpret_cast<uint4 *>(map_array<P, kMode>(sm))[tid] = make_uint4(0u, 0u, 0u, 0u);
                    }
                    if (lt == 0) __syncthreads();   // (before counts and map are written; else the lookback's)
                }
            }
        }
        if (paired && !by_rows) {
            // two neighbouring cells (cx, cx + 1) a thread, one in each half2 lane: each lane
            // performs its cell's additions of from_terms in the same order (an odd row's
            // last pair computes a cell past the row and drops it)
            const int hpr = (ww + 1) >> 1;
            for (int pi = tid; pi < hpr * wh; pi += kThreads) {
                const int cy = pi / hpr, cx = 2 * (pi - cy * hpr);
                __half2 acc = __float2half2_rn(0.0f);
                for (int i = 0; i <= 2 * r; ++i) {
                    const int hw = sm.trk.w[i];
                    const int b = (cy + i) * rw + cx + r;
                    __half2 rs = __float2half2_rn(0.0f);
#pragma unroll 4
                    for (int dx = -hw; dx <= hw; ++dx) rs = __hadd2(rs, sm.u.term2[PF_IDX(b + dx, kRoiMax / 2)]);
                    acc = __hadd2(acc, rs);
                }
                const int c = cy * ww + cx;
                const __half2 a2 = acc;
                lik_t *tab = sm.table;
                tab[PF_IDX(c, kTableMax)] = *reinterpret_cast<const lik_t *>(&a2);
                if (cx + 1 < ww) tab[PF_IDX(c + 1, kTableMax)] = reinterpret_cast<const lik_t *>(&a2)[1];
            }
        }
        const int wdiv = kMode != kModeCdf ? ww : 1;    // (no table in the CDF kernel)
        for (int c = paired || by_rows ? cells : tid, cy = tid / wdiv, cx = tid - (tid / wdiv) * wdiv; c < cells; c += kThreads) {
            if constexpr (Tr::kHalf) {
                sm.table[PF_IDX(c, kTableMax)] = hk.from_terms(sm.u.term, rw, sm.trk.w, r, cx, cy);
            } else {
                uint32_t ssum = 0;
#pragma unroll 4
                for (int i = 0; i <= 2 * r; ++i) {
                    const uint16_t *p = sm.u.pre + (cy + i) * (rw + 1) + cx + r;
                    const int hw = sm.trk.w[i];
                    ssum += static_cast<uint32_t>(static_cast<uint16_t>(p[hw + 1] - p[-hw]));
                }
                sm.table[PF_IDX(c, kTableMax)] = lik_from_sum<acc_t>(ssum, c1, c2D, den);
            }
            cx += kThreads;               // next cell: kThreads further in row-major order
            while (cx >= ww) { cx -= ww; ++cy; }
        }
        // (no barrier: the next one, before the offspring, orders the table's writes)
    }

    // ------------------------------------------------------------ 1d. lookback, CDF, strata
    int Jr[kItems];           // J of the thread's elements (frames t > 0)
    int jb, je;               // the tile's offspring are j in [jb, je)
    if (!kPull && t > 0) {
        // the step kernel's window phase ordered the tile aggregate (sm.agg_x) and the warps'
        // running maxima before this point; the CDF kernel has no window phase
        if constexpr (kMode == kModeCdf) __syncthreads();
        {   // the block part of the running max
            acc_t wmax = static_cast<acc_t>(0);
            if constexpr (kF64) {
#pragma unroll
                for (int w = 0; w < kWarps; ++w) {
                    const acc_t v = sm.warp_max[w];
                    if (w < warp) wmax = prefix_max(wmax, v);
                }
            } else {   // lane w < warp holds warp w's maximum (prefixes are >= 0): one redux
                wmax = warp_max(lane < warp ? sm.warp_max[lane] : static_cast<acc_t>(0));
            }
            if (lane == 0) mex = wmax; else mex = prefix_max(mex, wmax);
#pragma unroll
            for (int m = 0; m < kItems; ++m) loc[m] = prefix_max(loc[m], mex);
        }
        const acc_t invS = Lp.shard ? static_cast<acc_t>(Lp.g_invS)
                                    : (kF64 ? static_cast<acc_t>(sm.st.invS) : static_cast<acc_t>(sm.st.invS_f));
#ifdef PF_NAIVE_RESAMPLE
        const acc_t Sdiv = static_cast<acc_t>(sm.st.S);   // study build: a division per element
#endif
        const acc_t u0 = kF64 ? static_cast<acc_t>(sm.u0d) : static_cast<acc_t>(sm.u0f);
#ifdef PF_NAIVE_RESAMPLE
        const acc_t inv_n = static_cast<acc_t>(N);     // the study build divides by N per point
#else
        const acc_t inv_n = sizeof(acc_t) == 8 ? static_cast<acc_t>(T.inv_n) : static_cast<acc_t>(T.inv_n_f);
#endif
        // exact prefix before the tile (every thread) and after it (published as inclusive)
        const U128 exclx = (lt > 0) ? lookback<P>(look, lt, dtag, st, sm) : U128{0ull, 0ull};
        const U128 endx = add128(exclx, sm.agg_x);
        if (tid == 0 && lt > 0) desc_publish(&look[lt], 1, endx, dtag);
        // Prefix of the tile's elements: FP inside the tile, pinned to the exact fixed-point
        // values at both tile boundaries, so neighbouring tiles see the same boundary.
        acc_t excl, pend;
        if constexpr (kF64) { excl = from_fixed(exclx); pend = from_fixed(endx); }
        else { excl = from_fixed_f(exclx); pend = from_fixed_f(endx); }
        if constexpr (kMode == kModeCdf) {
            acc_t *const cdf = static_cast<acc_t *>(T.cdf);
            // a shard: its prefix starts at the other ranks' total before it and ends pinned
            // at shard_hi, the value its successor starts from
            const acc_t slo = static_cast<acc_t>(Lp.shard_lo), shi = static_cast<acc_t>(Lp.shard_hi);
            if (Lp.shard) { excl = add_rn(excl, slo); pend = add_rn(pend, slo); }
#pragma unroll
            for (int m = 0; m < kItems; ++m) {
                const int e = eb + m;
                if (e < cnt) {
                    const int k = k0 + e;
                    acc_t Pk = (e == cnt - 1) ? pend : prefix_min(add_rn(excl, loc[m]), pend);
                    if (Lp.shard) Pk = (k == N - 1) ? shi : prefix_min(Pk, shi);
                    acc_t C = prefix_min(PF_NORM(Pk), static_cast<acc_t>(1));
                    if (k == N - 1 && (!Lp.shard || Lp.shard_last)) C = static_cast<acc_t>(1);
                    cdf[PF_IDX(k, N)] = C;
                    // the pull kernel's coarser levels: the value at the end of every 8 and 64
                    if ((m == kItems - 1 || k == N - 1) && T.cdf8) {
                        static_cast<acc_t *>(T.cdf8)[PF_IDX(k >> 3, (N + 7) >> 3)] = C;
                        if ((k & 63) == 63 || k == N - 1) static_cast<acc_t *>(T.cdf64)[PF_IDX(k >> 6, (N + 63) >> 6)] = C;
                    }
                }
            }
            return;                       // the pull kernel takes the offspring
        }
        // J of the tile's first element and of each element, for either resampling scheme
#ifdef PF_NAIVE_RESAMPLE
        const acc_t nrm = Sdiv;
#else
        const acc_t nrm = invS;
#endif
        int jbl = 0, jprev0 = 0;   // the tile's first count; the count before the thread's first element
        // The count before a warp's first element: that element's predecessor is the previous
        // warp's last, whose clamped prefix is the running max of all preceding warps (the
        // running max at lane 0 of this warp, mex), so the count is taken here from the same
        // value, with the same arithmetic, as its owner takes it.
        const acc_t c_beg = prefix_min(PF_NORM(excl), static_cast<acc_t>(1));
        const acc_t c_prev = prefix_min(PF_NORM(prefix_min(add_rn(excl, mex), pend)), static_cast<acc_t>(1));
        const auto counts = [&](const auto &str) {
            strata_counts(str, loc, Jr, excl, pend, nrm, eb, cnt, k0, N, dbg_cdf, st);
            if (!kF64 || warp * 32 * kItems < cnt) jbl = (lt == 0) ? 0 : str.count_le(c_beg);
            if (lane == 0 && tid != 0 && eb < cnt) jprev0 = str.count_le(c_prev);
            if (tid == 0) jprev0 = jbl;
        };
        if (T.resampler == kResampleStratified) {
            // (key_lo, key_hi, frame t - 1, tracker id) of the stratum offsets
            Stratified<acc_t> str;
            str.init(N, inv_n, sm.skeys);
            counts(str);
        } else if (kF64 || (kMode != kModeStepBig && N <= (1 << 20))) {
            Systematic<acc_t, true> str;
            str.init(N, u0, inv_n);
            counts(str);
        } else if constexpr (!kF64) {
            Systematic<acc_t, false> str;
            str.init(N, u0, inv_n);
            counts(str);
        }
        // Every thread knows the tile's first count and the count before its first element,
        // so the ancestor map's heads go in now (phase 1e fills the gaps): map[jp - mb] =
        // 1 + element, jp the first offspring of each element that has offspring, mb the
        // tile's first offspring rounded down to even (a pair is one aligned word of the map).
        {
            const int mbl = jbl & ~1;
            int jp = __shfl_up_sync(0xffffffffu, Jr[kItems - 1], 1);
            if (lane == 0) jp = jprev0;
            if (eb < cnt) {
#pragma unroll
                for (int m = 0; m < kItems; ++m) {
                    if (Jr[m] > jp && jp - mbl < kMapMax)
                        map_array<P, kMode>(sm)[PF_IDX(jp - mbl, kMapMax)] = static_cast<uint16_t>(eb + m + 1);
                    jp = Jr[m];
                }
                if constexpr (kMode == kModeStep) store_items(counts_array<P, kMode>(sm) + eb, Jr);
                if (eb + kItems >= cnt) sm.jend = Jr[kItems - 1];   // the tile's last element's owner
            }
        }
        if (tid == 0) sm.jbeg = jbl;
        if (gt) fetch_table<P>(T, sm, wx0, wy0, ww, cells, fv, c1, c2D, den, st);
        __syncthreads();          // the heads, jbeg, jend and the likelihood table are complete
        jb = sm.jbeg;
        je = sm.jend;
    } else {
        jb = k0;
        je = k0 + cnt;
        if (gt) fetch_table<P>(T, sm, wx0, wy0, ww, cells, fv, c1, c2D, den, st);
        __syncthreads();          // the likelihood table is complete
    }

    // ------------------------------------------------------------ 1e. ancestor map
    // map[j - mb] = 1 + tile element that is the ancestor of offspring j: the heads (phase
    // 1d; the map was cleared at the start of the tile), then a block-wide running max fills
    // the gaps, two entries of a word at a time.
    const int mb = jb & ~1;
    const bool use_map = !kPull && (t > 0) && je - mb <= kMapMax;
    if (use_map) {
        // thread tid fills entries [tid*ch, tid*ch + ch), ch = 8 or 16 (16-byte vectors)
        const int nv = (je - mb > kThreads * 8) ? 2 : 1;
        uint4 *mv = reinterpret_cast<uint4 *>(map_array<P, kMode>(sm)) + tid * nv;
        uint4 c0 = mv[0], c1 = make_uint4(0u, 0u, 0u, 0u);
        if (nv == 2) c1 = mv[1];
        uint32_t m2 = __vmaxu2(__vmaxu2(__vmaxu2(c0.x, c0.y), __vmaxu2(c0.z, c0.w)),
                               __vmaxu2(__vmaxu2(c1.x, c1.y), __vmaxu2(c1.z, c1.w)));
        int xm = static_cast<int>(max(m2 & 0xffffu, m2 >> 16));
        // (a lane without a lane o below gets its own value: no change to a maximum)
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) xm = max(xm, __shfl_up_sync(0xffffffffu, xm, o));
        if (lane == 31) sm.warp_imax[warp] = xm;
        int run = __shfl_up_sync(0xffffffffu, xm, 1);
        if (lane == 0) run = 0;
        __syncthreads();
        // the maxima of the preceding warps: lane w < warp holds warp w's (entries are >= 0)
        run = max(run, __reduce_max_sync(0xffffffffu, lane < warp ? sm.warp_imax[lane] : 0));
        uint32_t r2 = __byte_perm(static_cast<uint32_t>(run), 0u, 0x1010);   // in both halves
        uint32_t w4[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (i < 4 * nv) {
                w4[i] = __vmaxu2(__vmaxu2(w4[i], w4[i] << 16), r2);
                r2 = __byte_perm(w4[i], 0u, 0x3232);
            }
        }
        mv[0] = make_uint4(w4[0], w4[1], w4[2], w4[3]);
        if (nv == 2) mv[1] = make_uint4(w4[4], w4[5], w4[6], w4[7]);
        __syncthreads();
    } else if (kMode == kModeStepBig && t > 0) {   // (the barrier above ordered the map's heads)
        store_items(counts_array<P, kMode>(sm) + eb, Jr);
        __syncthreads();
    }

    // ------------------------------------------------------------ 2-4. offspring
    pos_t *__restrict__ Xout = static_cast<pos_t *>(T.px[out]);
    pos_t *__restrict__ Yout = static_cast<pos_t *>(T.py[out]);
    lik_t *__restrict__ Lout = static_cast<lik_t *>(T.pl[out]);
    int32_t *__restrict__ dbg_anc = T.dbg_anc;
    const uint32_t tctr = static_cast<uint32_t>(t);
    const uint32_t trk_id = T.tracker_id;
    const int jpair0 = static_cast<int>(T.j_base >> 1);   // global pair index of local pair 0
    Stats<acc_t> stats{neg_inf<acc_t>(), 0, 0, 0};
    const acc_t nxa_a = static_cast<acc_t>(nxi), nya_a = static_cast<acc_t>(nyi);
    const int axi = nxi, ayi = nyi;
    const acc_t dxm = kF64 ? static_cast<acc_t>(T.drift_x) : static_cast<acc_t>(T.drift_xf);
    const acc_t dym = kF64 ? static_cast<acc_t>(T.drift_y) : static_cast<acc_t>(T.drift_yf);
    const acc_t sgx = kF64 ? static_cast<acc_t>(T.sigma_x) : static_cast<acc_t>(T.sigma_xf);
    const acc_t sgy = kF64 ? static_cast<acc_t>(T.sigma_y) : static_cast<acc_t>(T.sigma_yf);
    // offsets: the ancestors' anchor minus the offspring's anchor (integers)
    const float shx = static_cast<float>(axi_anc - nxi), shy = static_cast<float>(ayi_anc - nyi);
    const float ix0 = T.init_xf - static_cast<float>(nxi), iy0 = T.init_yf - static_cast<float>(nyi);

    // bounding box of the thread's new positions (for the next step's tracker table, when
    // the tracker is large enough to use one): absolute in REF64 / F32, anchor offsets in
    // half2 lanes in F16 / BF16
    acc_t pbx0 = static_cast<acc_t>(FLT_MAX), pbx1 = static_cast<acc_t>(-FLT_MAX);
    acc_t pby0 = static_cast<acc_t>(FLT_MAX), pby1 = static_cast<acc_t>(-FLT_MAX);
    using HB2 = typename HalfOps<H>::h2;
    HB2 hbx0 = HalfOps<H>::from_f2(65504.0f, 65504.0f), hbx1 = HalfOps<H>::from_f2(-65504.0f, -65504.0f);
    HB2 hby0 = hbx0, hby1 = hbx1;

    // (What bounds the loop is instruction issue, about 95 a particle.  An aligned map word a pair,
    // one gathered word an ancestor in F16 / BF16, uniforms by a funnel shift and window_offset
    // took F32 at 2^20 from 26.1 to 24.0 us a frame, F16 22.1 -> 21.6, REF64 at 200k 262 -> 231.)
    // One pair of offspring (j0, j1) = (2q, 2q + 1).  Compile-time flags: V0 / V1, the
    // particle lies in [jb, je); FAST, frame t > 0 with the ancestor map and no debug
    // arrays (the interior pairs of a tile in production take the FAST copy).
    auto pair = [&](const int q, auto V0c, auto V1c, auto FASTc) {
        constexpr bool v0 = decltype(V0c)::value, v1 = decltype(V1c)::value;
        constexpr bool kFast = decltype(FASTc)::value;
        const int j0 = 2 * q, j1 = j0 + 1;
        int e0 = 0, e1 = 0;
        if (kFast) {
            const uint32_t mw = reinterpret_cast<const uint32_t *>(map_array<P, kMode>(sm))[PF_IDX(q - (mb >> 1), kMapMax / 2)];
            e0 = static_cast<int>(mw & 0xffffu) - 1;
            e1 = static_cast<int>(mw >> 16) - 1;
        } else if (t > 0) {
            if constexpr (kPull) {
                // multinomial: the ancestors were gathered into ax/ay at the tile's own
                // output positions (J holds their indices)
                e0 = j0 - k0;
                e1 = j1 - k0;
            } else if (use_map) {
                e0 = v0 ? static_cast<int>(map_array<P, kMode>(sm)[PF_IDX(j0 - mb, kMapMax)]) - 1 : 0;
                e1 = v1 ? static_cast<int>(map_array<P, kMode>(sm)[PF_IDX(j1 - mb, kMapMax)]) - 1 : 0;
            } else {
                if (v0) e0 = upper_index(counts_array<P, kMode>(sm), cnt, j0);
                if (v1) e1 = (v0 && counts_array<P, kMode>(sm)[e0] > j1) ? e0 : upper_index(counts_array<P, kMode>(sm), cnt, j1);
            }
            if (!v0) e0 = e1;
            if (!v1) e1 = e0;
            if (dbg_anc) {
                if constexpr (kPull) {
                    if (v0) dbg_anc[PF_IDX(j0, N)] = counts_array<P, kMode>(sm)[e0];
                    if (v1) dbg_anc[PF_IDX(j1, N)] = counts_array<P, kMode>(sm)[e1];
                } else {
                    if (v0) dbg_anc[PF_IDX(j0, N)] = k0 + e0;
                    if (v1) dbg_anc[PF_IDX(j1, N)] = k0 + e1;
                }
            }
        }
        // one Philox block per particle pair: words (x, y) for j0, (z, w) for j1 (a shard's
        // pairs are numbered globally)
        const uint4 wd = philox4x32_10_keys(make_uint4(static_cast<uint32_t>(q + jpair0), tctr, 0u, trk_id),
                                            reinterpret_cast<const uint4 *>(sm.rk));

        if constexpr (!Tr::kHalf) {
            // ---------------- REF64 / F32: absolute positions, exact-integer likelihood
            acc_t xa0, ya0, xa1, ya1;
            if (t > 0) {
                xa0 = sm.a[PF_IDX(e0, kTile)]; ya0 = sm.a[kTile + PF_IDX(e0, kTile)];
                xa1 = sm.a[PF_IDX(e1, kTile)]; ya1 = sm.a[kTile + PF_IDX(e1, kTile)];
            }
            else {
                xa0 = xa1 = kF64 ? static_cast<acc_t>(T.init_x) : static_cast<acc_t>(T.init_xf);
                ya0 = ya1 = kF64 ? static_cast<acc_t>(T.init_y) : static_cast<acc_t>(T.init_yf);
            }
            acc_t n0x, n0y, n1x, n1y;
            if constexpr (sizeof(acc_t) == 8) {
                box_muller_table(wd.x, wd.y, n0x, n0y);
                box_muller_table(wd.z, wd.w, n1x, n1y);
            } else {
                box_muller(uniform_f32(wd.x), uniform_f32(wd.y), n0x, n0y);
                box_muller(uniform_f32(wd.z), uniform_f32(wd.w), n1x, n1y);
            }
            const acc_t x0 = add_rn(add_rn(xa0, dxm), mul_rn(sgx, n0x));
            const acc_t y0 = add_rn(add_rn(ya0, dym), mul_rn(sgy, n0y));
            const acc_t x1 = add_rn(add_rn(xa1, dxm), mul_rn(sgx, n1x));
            const acc_t y1 = add_rn(add_rn(ya1, dym), mul_rn(sgy, n1y));
            const unsigned cx0 = window_offset(x0, wx0), cy0 = window_offset(y0, wy0);
            const unsigned cx1 = window_offset(x1, wx0), cy1 = window_offset(y1, wy0);
            const bool in0 = cx0 < static_cast<unsigned>(ww) && cy0 < static_cast<unsigned>(wh);
            const bool in1 = cx1 < static_cast<unsigned>(ww) && cy1 < static_cast<unsigned>(wh);
            acc_t L0 = v0 && in0 ? sm.table[cy0 * ww + cx0] : static_cast<acc_t>(0);
            acc_t L1 = v1 && in1 ? sm.table[cy1 * ww + cx1] : static_cast<acc_t>(0);
            if constexpr (kMode == kModeStepBig) {   // (with the tracker's table none misses; without, see direct_likelihoods)
                if (v0 && !in0) L0 = lik_from_sum<acc_t>(disk_sum(fv, sm.trk.w, pixel_of(x0), pixel_of(y0)), c1, c2D, den);
                if (v1 && !in1) L1 = lik_from_sum<acc_t>(disk_sum(fv, sm.trk.w, pixel_of(x1), pixel_of(y1)), c1, c2D, den);
            } else {
                const int miss = (v0 && !in0 ? 1 : 0) | (v1 && !in1 ? 2 : 0);
                const unsigned act = __activemask();
                if (__any_sync(act, miss != 0))
                    direct_likelihoods<P>(T, fv, sm.trk.w, act, miss, pixel_of(x0), pixel_of(y0), pixel_of(x1), pixel_of(y1), L0, L1);
            }
            if (v0 && v1) {
                if constexpr (sizeof(acc_t) == 8) {
                    reinterpret_cast<double2 *>(Xout)[PF_IDX(q, N / 2)] = make_double2(x0, x1);
                    reinterpret_cast<double2 *>(Yout)[q] = make_double2(y0, y1);
                    reinterpret_cast<double2 *>(Lout)[q] = make_double2(L0, L1);
                } else {
                    reinterpret_cast<float2 *>(Xout)[PF_IDX(q, N / 2)] = make_float2(x0, x1);
                    reinterpret_cast<float2 *>(Yout)[q] = make_float2(y0, y1);
                    reinterpret_cast<float2 *>(Lout)[q] = make_float2(L0, L1);
                }
            } else if (v0) {
                Xout[PF_IDX(j0, N)] = x0; Yout[j0] = y0; Lout[j0] = L0;
            } else if (v1) {
                Xout[PF_IDX(j1, N)] = x1; Yout[j1] = y1; Lout[j1] = L1;
            }
            stats_add2<false>(stats, v0, L0, x0 - nxa_a, y0 - nya_a, v1, L1, x1 - nxa_a, y1 - nya_a);
            if (track_box) {
                if (v0) { pbx0 = fmin(pbx0, x0); pbx1 = fmax(pbx1, x0); pby0 = fmin(pby0, y0); pby1 = fmax(pby1, y0); }
                if (v1) { pbx0 = fmin(pbx0, x1); pbx1 = fmax(pbx1, x1); pby0 = fmin(pby0, y1); pby1 = fmax(pby1, y1); }
            }
        } else {
            // ---------------- F16 / BF16: half2 lanes = particles (j0, j1), offsets from the anchor
            using OPS = HalfOps<H>;
            using h2 = typename OPS::h2;
            h2 ox, oy;
            if (t > 0) {
                const uint32_t a0 = reinterpret_cast<const uint32_t *>(sm.a)[PF_IDX(e0, kTile)];
                const uint32_t a1 = reinterpret_cast<const uint32_t *>(sm.a)[PF_IDX(e1, kTile)];
                const uint32_t xw = __byte_perm(a0, a1, 0x5410), yw = __byte_perm(a0, a1, 0x7632);
                ox = *reinterpret_cast<const h2 *>(&xw);
                oy = *reinterpret_cast<const h2 *>(&yw);
                if (shx != 0.0f || shy != 0.0f) {
                    ox = __hadd2(ox, OPS::from_f2(shx, shx));
                    oy = __hadd2(oy, OPS::from_f2(shy, shy));
                }
            } else {
                ox = OPS::from_f2(ix0, ix0);
                oy = OPS::from_f2(iy0, iy0);
            }
            float a, b, c, d;
            box_muller_fast(uniform_f32(wd.x), uniform_f32(wd.y), a, b);
            box_muller_fast(uniform_f32(wd.z), uniform_f32(wd.w), c, d);
            ox = __hadd2(ox, OPS::from_f2(dxm + sgx * a, dxm + sgx * c));
            oy = __hadd2(oy, OPS::from_f2(dym + sgy * b, dym + sgy * d));
            const unsigned cx0 = window_offset(OPS::lo(ox), wx0 - axi), cy0 = window_offset(OPS::lo(oy), wy0 - ayi);
            const unsigned cx1 = window_offset(OPS::hi(ox), wx0 - axi), cy1 = window_offset(OPS::hi(oy), wy0 - ayi);
            const bool in0 = cx0 < static_cast<unsigned>(ww) && cy0 < static_cast<unsigned>(wh);
            const bool in1 = cx1 < static_cast<unsigned>(ww) && cy1 < static_cast<unsigned>(wh);
            H l0 = in0 ? sm.table[cy0 * ww + cx0] : OPS::from_f(0.0f);
            H l1 = in1 ? sm.table[cy1 * ww + cx1] : OPS::from_f(0.0f);
            if constexpr (kMode == kModeStepBig) {   // (with the tracker's table none misses; without, see direct_likelihoods)
                if (v0 && !in0) l0 = hk.at(fv, sm.trk.w, axi + pixel_of(OPS::lo(ox)), ayi + pixel_of(OPS::lo(oy)));
                if (v1 && !in1) l1 = hk.at(fv, sm.trk.w, axi + pixel_of(OPS::hi(ox)), ayi + pixel_of(OPS::hi(oy)));
            } else {
                const int miss = (v0 && !in0 ? 1 : 0) | (v1 && !in1 ? 2 : 0);
                const unsigned act = __activemask();
                if (__any_sync(act, miss != 0))
                    direct_likelihoods<P>(T, fv, sm.trk.w, act, miss, axi + pixel_of(OPS::lo(ox)), ayi + pixel_of(OPS::lo(oy)),
                                          axi + pixel_of(OPS::hi(ox)), ayi + pixel_of(OPS::hi(oy)), l0, l1);
            }
            if (v0 && v1) {
                reinterpret_cast<h2 *>(Xout)[PF_IDX(q, N / 2)] = ox;
                reinterpret_cast<h2 *>(Yout)[q] = oy;
                reinterpret_cast<h2 *>(Lout)[q] = OPS::pack(l0, l1);
            } else if (v0) {
                Xout[PF_IDX(j0, N)] = OPS::lo_h(ox); Yout[j0] = OPS::lo_h(oy); Lout[j0] = l0;
            } else if (v1) {
                Xout[PF_IDX(j1, N)] = OPS::hi_h(ox); Yout[j1] = OPS::hi_h(oy); Lout[j1] = l1;
            }
            stats_add2<true>(stats, v0, OPS::to_f(l0), OPS::lo(ox), OPS::lo(oy), v1, OPS::to_f(l1), OPS::hi(ox), OPS::hi(oy));
            // (a lane outside [jb, je) holds a draw around a valid ancestor: inside the reach
            // of the next step's table all the same)
            if (track_box) {
                hbx0 = __hmin2(hbx0, ox); hbx1 = __hmax2(hbx1, ox);
                hby0 = __hmin2(hby0, oy); hby1 = __hmax2(hby1, oy);
            }
        }
    };
    {
        using TT = std::true_type;
        using FF = std::false_type;
        const int qi0 = (jb + 1) >> 1, qi1 = je >> 1;   // pairs with both particles in [jb, je)
        if (t > 0 && use_map && !dbg_anc) {
            for (int q = qi0 + tid; q < qi1; q += kThreads) pair(q, TT{}, TT{}, TT{});
        } else {
            for (int q = qi0 + tid; q < qi1; q += kThreads) pair(q, TT{}, TT{}, FF{});
        }
        // the pairs that straddle the ends of [jb, je)
        if (tid == 0 && (jb & 1) && jb < je) pair(jb >> 1, FF{}, TT{}, FF{});
        if (tid == kThreads - 1 && (je & 1) && je > jb) pair(je >> 1, TT{}, FF{}, FF{});
    }

    // ------------------------------------------------------------ 5. tile partial + finalise
    float4 bb;
    if constexpr (Tr::kHalf) {
        const float ax = static_cast<float>(nxi), ay = static_cast<float>(nyi);
        bb = make_float4(fminf(HalfOps<H>::lo(hbx0), HalfOps<H>::hi(hbx0)) + ax,
                         fmaxf(HalfOps<H>::lo(hbx1), HalfOps<H>::hi(hbx1)) + ax,
                         fminf(HalfOps<H>::lo(hby0), HalfOps<H>::hi(hby0)) + ay,
                         fmaxf(HalfOps<H>::lo(hby1), HalfOps<H>::hi(hby1)) + ay);
    } else {
        // widened to whole pixels outwards, so the float box still contains every position
        bb = make_float4(static_cast<float>(floor(pbx0)), static_cast<float>(ceil(pbx1)),
                         static_cast<float>(floor(pby0)), static_cast<float>(ceil(pby1)));
    }
    if (track_box) warp_box(bb, sm);
    const Stats<acc_t> tot = block_stats<P>(stats, sm);
    if (track_box && warp == 0) bb = merge_warp_boxes(sm);
    double *const est_out = Lp.est_out ? Lp.est_out + 2 * ti : nullptr;
    if (T.ntiles == 1) {   // its statistics are the tracker's: no partial, no wait
        finish_tracker<P>(T, st, sm, tot, bb, est_out, track_box);
        return;
    }
    if (tid == 0) {
        TilePartial *p = &T.part[PF_IDX(lt, T.ntiles)];
        if (track_box) {
            const uint64_t btg = partial_tag(sm.st.epoch);
            st_relaxed_v2(&p->b[0], btg | __float_as_uint(bb.x), btg | __float_as_uint(bb.y));
            st_relaxed_v2(&p->b[2], btg | __float_as_uint(bb.z), btg | __float_as_uint(bb.w));
        }
        if constexpr (kF64) {
            p->d[0] = tot.m;
            p->d[1] = tot.s;
            p->d[2] = tot.sx;
            p->d[3] = tot.sy;
            // release: the partial is visible before the count; acquire: the last tile sees all
            sm.last = atom_add_acq_rel(T.done, 1u) == static_cast<uint32_t>(T.ntiles - 1) ? 1u : 0u;
        } else {
            const uint64_t tg = partial_tag(sm.st.epoch);
            st_relaxed_v2(&p->w[0], tg | __float_as_uint(tot.m), tg | __float_as_uint(tot.s));
            st_relaxed_v2(&p->w[2], tg | __float_as_uint(tot.sx), tg | __float_as_uint(tot.sy));
        }
    }
    // The tracker's last tile finalises, waiting for every partial's tag: no tile waits for a
    // counter's round trip (the tiles before it hold lower tickets, so they are running or
    // done).  REF64, whose partials carry no tags: the last tile to arrive.
    bool last = lt == T.ntiles - 1;
    if constexpr (kF64) {
        __syncthreads();
        last = sm.last != 0u;
    }
    if (last) finalize_tracker<P>(T, st, sm, est_out, track_box);
}

// CTAs per SM the register allocation must allow: 1024 threads per SM (64 registers a
// thread) for the FP32/FP16/BF16 kernels, 512 for REF64 (its FP64 Box-Muller needs ~128);
// measured best on GB300 for the latency-bound step.
template <int P> struct MinBlocks {
    static constexpr int value = (P == 0 ? 512 : 1024) / kThreads > 0 ? (P == 0 ? 512 : 1024) / kThreads : 1;
};

// kWaves: the launch may have more tiles than CTAs.  (Without the loop over tiles the kernels hold
// their registers better: F16 2^20 particles 19.66 -> 19.10 us a frame, F32 600001 17.1 -> 16.8,
// multinomial F16 2^20 65.0 -> 63.9, 2^19 40.4 -> 39.8.)
template <int P, int kMode, bool kWaves>
__global__ void __launch_bounds__(kThreads, MinBlocks<P>::value) step_kernel(const StepLaunch Lp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StepSmem<P> &sm = *reinterpret_cast<StepSmem<P> *>(smem_raw);
    // One tracker whose descriptor and frame reference no kernel writes (Lp.preload): they load
    // while the previous launch drains.
    if (Lp.ntrk == 1 && Lp.preload) load_descriptor(Lp, 0, 0, sm, 1);
    // Programmatic dependent launch: a launch that follows another step on the same stream
    // may be scheduled while that one drains; everything else it reads (ticket, state,
    // particles) is written by its predecessor, so it waits for the predecessor grid to
    // complete, then lets its own successor be scheduled.  (Both are no-ops for a launch
    // without the programmatic-serialization attribute.)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // Tiles in ticket order, every ticket drawn: a tile waits for its predecessors (the lookback; the
    // last tile's wait for all partials), and a drawn ticket says that the CTAs of all lower ones are
    // running.  A CTA's index does not: CUDA promises no order of dispatch, and where fewer
    // than gridDim.x CTAs are resident (a partition of the SMs, other kernels on them) the CTAs
    // of a launch of several waves came back for tiles whose predecessors were first tiles of CTAs
    // without an SM, and waited out their limit.  A launch of one wave draws once a CTA, while the
    // state loads, and the last draw sets the word back (against CTA indices and no draw: F16 2^20
    // particles 18.9 -> 19.1 us a frame, F32 21.6 -> 21.2, 600001 16.65 -> 16.8); a single tile waits
    // for no other and draws none.  In a longer launch a ticket is drawn when the CTA is ready for
    // it: drawn a tile ahead, its aggregate reaches the tiles that look back to it a tile later
    // (2^24 F16 265 -> 329 us).
    const auto total = [&] { return static_cast<uint32_t>(Lp.total_tiles); };
    if (threadIdx.x == 0) {
        uint32_t g = 0u;
        if (total() > 1u) {
            g = atomicAdd(Lp.ticket, 1u);
            if (total() <= gridDim.x && g == total() - 1u) atomicExch(Lp.ticket, 0u);
        }
        sm.ticket = g;
        sm.cached = Lp.ntrk == 1 ? 0 : -1;
    }
    if (Lp.ntrk == 1) load_descriptor(Lp, Lp.slot_of ? __ldg(&Lp.slot_of[0]) : 0, 0, sm, Lp.preload ? 2 : 3);
    __syncthreads();
    if constexpr (kWaves) {
        for (uint32_t g = sm.ticket; g < total();) {
            run_tile<P, kMode>(Lp, static_cast<int>(g), sm);
            if (total() <= gridDim.x) return;
            __syncthreads();
            if (threadIdx.x == 0) sm.ticket = atomicAdd(Lp.ticket, 1u);
            __syncthreads();
            g = sm.ticket;
        }
        // (several waves: total_tiles + gridDim.x draws in all)
        if (threadIdx.x == 0 && sm.ticket == total() + gridDim.x - 1u) atomicExch(Lp.ticket, 0u);
    } else {
        run_tile<P, kMode>(Lp, static_cast<int>(sm.ticket), sm);
    }
}

// Test hook: the lookback wait on a descriptor that nobody publishes, with a short limit;
// it must give up, raise the timeout bit and return.
__global__ void wait_probe_kernel(const LookbackDesc *d, TrackerState *st, uint32_t limit) {
    U128 v;
    wait_desc(d, desc_tag(1u), st, v, limit);
}

__global__ void philox_kernel(const uint4 *ctrs, int64_t n, uint32_t k0, uint32_t k1, uint4 *out) {
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i < n) out[i] = philox4x32_10(ctrs[i], k0, k1);
}

template <int P>
int configure_and_grid(int total_tiles) {
    // MinBlocks CTAs must fit in an SM's 228 KB of shared memory (1 KB reserved per CTA)
    // (the 1024-thread study build has no REF64 kernel: its tile does not fit)
    static_assert((sizeof(StepSmem<P>) + 1024) * MinBlocks<P>::value <= 228 * 1024 || kThreads > 512,
                  "shared memory of the step kernel exceeds its CTAs per SM");
    if (sizeof(StepSmem<P>) + 1024 > 228 * 1024) return -1;
    const int bytes = static_cast<int>(sizeof(StepSmem<P>));
    const auto allow = [&](auto *k) {
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    };
    if (!allow(step_kernel<P, kModeStep, false>) || !allow(step_kernel<P, kModeStep, true>) ||
        !allow(step_kernel<P, kModeStepBig, true>) || !allow(step_kernel<P, kModeCdf, false>) ||
        !allow(step_kernel<P, kModeCdf, true>) || !allow(step_kernel<P, kModePull, false>) ||
        !allow(step_kernel<P, kModePull, true>))
        return -1;
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, step_kernel<P, kModeStep, false>, kThreads, bytes);
    if (per_sm < 1) per_sm = 1;
    const int g = sms * per_sm;
    return total_tiles < g ? total_tiles : g;
}

}  // namespace

namespace {
// resident CTAs of the step kernel on the current device (cached per device and precision)
int slots_of(int precision) {
    static std::atomic<int> cache[64][4];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return -1; }
    if (precision < 0 || precision > 3) return -1;
    if (dev >= 0 && dev < 64) {
        const int c = cache[dev][precision].load(std::memory_order_relaxed);
        if (c > 0) return c;
    }
    int g = -1;
    switch (precision) {
        case 0: g = configure_and_grid<0>(0x7fffffff); break;
        case 1: g = configure_and_grid<1>(0x7fffffff); break;
        case 2: g = configure_and_grid<2>(0x7fffffff); break;
        case 3: g = configure_and_grid<3>(0x7fffffff); break;
    }
    if (g > 0 && dev >= 0 && dev < 64) cache[dev][precision].store(g, std::memory_order_relaxed);
    return g;
}
}  // namespace

int step_tile_size(int precision, int64_t n) {
    const int64_t slots = slots_of(precision);
    // a tracker that cannot fill half the device with full tiles keeps full tiles (in a
    // batch, other trackers fill the device)
    if (slots < 1) return kTile;
    if (n < slots * (kTile / 2)) {
        // REF64 is bound by the FP64 pipes of the SMs that have a tile, so a tracker of four
        // full tiles or more is spread over all of them, down to tiles of 1024 (below, a tile's
        // chain of phases costs as much as its arithmetic).  us a frame, full tiles -> these: 16384
        // particles 108 -> 51, 32768 110 -> 54, 200003 110 -> 64.  A batch that fills the device
        // loses by it (64 trackers of 20003 272 -> 327, 16 of 200003 548 -> 691), but a tracker's sums,
        // and so its bits, follow its tiles, and those are the same alone and in a batch.
        // Smaller trackers keep the tiles of 4096 that the window hook reports for them: 16383
        // particles 109, 4097 98.
        constexpr int64_t kLeast = kTile < 1024 ? kTile : 1024;
        if (precision == 0 && n >= 4 * kTile)
            return static_cast<int>(std::max(kLeast, ((n + slots - 1) / slots + 7) & ~int64_t(7)));
        return kTile;
    }
    const int64_t waves = (n + slots * kTile - 1) / (slots * kTile);
    int64_t tile = (n + slots * waves - 1) / (slots * waves);   // >= kTile / 2 here
    tile = (tile + 7) & ~int64_t(7);
    if (tile > kTile) tile = kTile;
    return static_cast<int>(tile);
}

int step_grid_size(int precision, int total_tiles) {
    switch (precision) {
        case 0: return configure_and_grid<0>(total_tiles);
        case 1: return configure_and_grid<1>(total_tiles);
        case 2: return configure_and_grid<2>(total_tiles);
        case 3: return configure_and_grid<3>(total_tiles);
    }
    return -1;
}

// A step-family launch with programmatic stream serialization: when the previous work on
// the stream is a step kernel (the previous frame), this launch is scheduled while that one
// drains and waits for it on the device (griddepcontrol.wait) instead of the stream
// serialising the two; captured into a CUDA graph as a programmatic dependency.
template <int P, int kMode>
int launch_one(int grid, const StepLaunch &L, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem_bytes<P, kMode>();
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if constexpr (kMode != kModeStepBig) {
        if (L.total_tiles <= grid) return static_cast<int>(cudaLaunchKernelEx(&cfg, step_kernel<P, kMode, false>, L));
    }
    return static_cast<int>(cudaLaunchKernelEx(&cfg, step_kernel<P, kMode, true>, L));
}

template <int kMode>
int launch_mode(int precision, const StepLaunch &L, int grid, void *stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (L.total_tiles < 1) return 0;
    grid = std::max(1, std::min(grid, static_cast<int>(L.total_tiles)));   // (one wave: a CTA a tile)
    int rc = -1;
    switch (precision) {
        case 0: rc = launch_one<0, kMode>(grid, L, s); break;
        case 1: rc = launch_one<1, kMode>(grid, L, s); break;
        case 2: rc = launch_one<2, kMode>(grid, L, s); break;
        case 3: rc = launch_one<3, kMode>(grid, L, s); break;
        default: return -1;
    }
    if (rc != 0) return rc;
    return static_cast<int>(cudaGetLastError());
}

int launch_step(int precision, const StepLaunch &L, int grid, void *stream) {
    // a single tracker of at least two waves of tiles takes the instantiation with the
    // tracker table (the kernel checks the condition again per tile)
    if (L.ntrk == 1 && L.total_tiles >= 2 * grid) return launch_mode<kModeStepBig>(precision, L, grid, stream);
    return launch_mode<kModeStep>(precision, L, grid, stream);
}

int launch_pull(int precision, const StepLaunch &L, int grid, bool with_cdf, void *stream) {
    const int rc = with_cdf ? launch_mode<kModeCdf>(precision, L, grid, stream) : 0;
    return rc != 0 ? rc : launch_mode<kModePull>(precision, L, grid, stream);
}

int launch_cdf(int precision, const StepLaunch &L, int grid, void *stream) {
    return launch_mode<kModeCdf>(precision, L, grid, stream);
}

// A shard's offspring run (see pf_internal.h): one thread per element of the shard's CDF,
// the count at its predecessor (J(c_lo) before the first) and at itself over the global
// strata, and the element's position copied to every offspring slot in between.
template <typename A>
__global__ void shard_expand_kernel(const A *C, const A *x, const A *y, int64_t n, int64_t n_global, int64_t t,
                                    uint32_t key_lo, uint32_t key_hi, uint32_t tracker, A c_lo, A *sx, A *sy,
                                    int64_t cap, int64_t *run, uint32_t *status) {
    const uint32_t w0 = philox4x32_10(make_uint4(0u, static_cast<uint32_t>(t - 1), 1u, tracker), key_lo, key_hi).x;
    const A u0 = sizeof(A) == 8 ? static_cast<A>(uniform_f64(w0)) : static_cast<A>(uniform_f32(w0));
    const A inv_n = sizeof(A) == 8 ? static_cast<A>(1.0 / static_cast<double>(n_global))
                                   : static_cast<A>(1.0f / static_cast<float>(n_global));
    Systematic<A, sizeof(A) == 8> str;
    str.init(static_cast<int>(n_global), u0, inv_n);
    const int64_t jb = str.count_le(c_lo);
    for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < n;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t j0 = k == 0 ? jb : str.count_le(C[k - 1]);
        const int64_t j1 = str.count_le(C[k]);
        const A xa = x[k], ya = y[k];
        for (int64_t j = j0; j < j1; ++j) {
            const int64_t i = j - jb;
            if (i >= 0 && i < cap) { sx[i] = xa; sy[i] = ya; }
            else atomicOr(status, 1u);
        }
        if (k == 0) run[0] = jb;
        if (k == n - 1) run[1] = j1;
    }
}

int launch_shard_expand(int precision, const void *cdf, const void *x, const void *y, int64_t n, int64_t n_global,
                        int64_t t, uint32_t key_lo, uint32_t key_hi, uint32_t tracker, double c_lo, void *sx,
                        void *sy, int64_t cap, int64_t *run, uint32_t *status, void *stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const unsigned blocks = static_cast<unsigned>(std::min<int64_t>((n + 255) / 256, 4096));
    if (precision == 0)
        shard_expand_kernel<double><<<blocks, 256, 0, s>>>(
            static_cast<const double *>(cdf), static_cast<const double *>(x), static_cast<const double *>(y), n, n_global,
            t, key_lo, key_hi, tracker, c_lo, static_cast<double *>(sx), static_cast<double *>(sy), cap, run, status);
    else if (precision == 1)
        shard_expand_kernel<float><<<blocks, 256, 0, s>>>(
            static_cast<const float *>(cdf), static_cast<const float *>(x), static_cast<const float *>(y), n, n_global,
            t, key_lo, key_hi, tracker, static_cast<float>(c_lo), static_cast<float *>(sx), static_cast<float *>(sy),
            cap, run, status);
    else
        return -1;
    return static_cast<int>(cudaGetLastError());
}

int launch_wait_probe(void *d_desc, void *d_state, uint32_t limit, void *stream) {
    wait_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const LookbackDesc *>(d_desc), static_cast<TrackerState *>(d_state), limit);
    return static_cast<int>(cudaGetLastError());
}

int launch_debug_philox(const uint32_t *d_ctrs, int64_t n, uint64_t seed, uint32_t *d_out, void *stream) {
    if (n <= 0) return 0;
    const int64_t blocks = (n + 255) / 256;
    philox_kernel<<<static_cast<unsigned>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        reinterpret_cast<const uint4 *>(d_ctrs), n, static_cast<uint32_t>(seed & 0xffffffffu),
        static_cast<uint32_t>(seed >> 32), reinterpret_cast<uint4 *>(d_out));
    return static_cast<int>(cudaGetLastError());
}

}  // namespace pfk
