// pf_gumbel.cu -- Gumbel-max resampling (sm_103a, CUDA cores only).
//
// Multinomial resampling in the log domain, the alternative to log-sum-exp that Sec. IV
// ("Numerical Stability Optimization") weighs: with g_jk = -ln(-ln u_jk) independent
// standard Gumbel variates, argmax_k (L_k + g_jk) follows the categorical law
// exp(L_k) / sum_i exp(L_i), so offspring j needs no maximum, no sum and no CDF of the
// weights -- only N draws of its own, hence N^2 draws a frame (trackers of at most
// kGumbelMaxN particles).
//
// u_jk is the uniform of word (k mod 4) of Philox(k / 4, t - 1, 4 + 256 j, tracker), and
// the sum is taken in the filter's weight precision: FP64 for REF64, FP32 for the others
// (L widened from its stored type).  Ties go to the smallest k.
//
// Most of the N^2 variates cannot win, and are refused without their two logarithms:
//   - g_jk lies in [-2.82, 16.64] (u has 24 bits), and the particle of the largest L enters
//     every offspring's argmax with at least max L - 2.82, so a particle below max L - 19.5
//     never wins: the CTA lists the quads with a particle above that line and draws for those
//     alone.  (max L is taken over the CTA's own pass over L, whatever state was loaded.)
//   - -ln u >= 1 - u gives g <= -ln(1 - u), so a variate beats the CTA's best b_j so far only
//     if (1 - u) exp(b_j - max L) <= exp(L_k - max L): one product in FP32 against two
//     logarithms, with a margin (1e-3 and 4e-6 max |L| relative) above the rounding of both sides.
// Whoever passes is evaluated as before, so the argmax and its ties are the same.
//
// Layout: CTA b takes kGumbelOffspring consecutive offspring of one tracker, thread i its
// offspring i mod 8 over every 32nd listed particle quad q (particles 4q .. 4q+3), from quad i / 8
// on: one Philox block per (quad, offspring) gives four draws, tested against the quad's four
// exp(L_k - max L) in shared memory (computed once for the CTA's offspring, kGumbelChunk quads at
// a time).  The best of an offspring's threads, as exp(b_j - max L), is shared through shared
// memory for the test above; it starts at the bound that the particle of the largest L gives.
// The CTA then reduces each offspring's (value, index) pairs, ties to the smaller index: two
// shuffles, then one thread per offspring over the warps' results.  The pull kernel gathers the
// ancestors written here.
// (A thread that draws for all eight offspring of its quad meets the shared best only in its
// second pass, after 1024 particles, leaves most threads idle on a short list, and holds 80
// registers to this one's 46.)
// Measured us a frame on the tracker's peaked weights, every variate in full -> these tests, a
// thread for all eight offspring of a quad -> this layout: F32 8191 particles 170 -> 86 -> 53, F16
// 1000 18.8 -> 21.4 -> 12.8, 2^16 10 040 -> 1144 -> 727, REF64 2047 603 -> 246 -> 103.
#include <math.h>

#include <type_traits>

#include "pf_ancestor.cuh"
#include "pf_device.cuh"
#include "pf_internal.h"

namespace pfk {
namespace {

__device__ __forceinline__ double gumbel_of(uint32_t w, double) { return -log(-log(uniform_f64(w))); }
__device__ __forceinline__ float gumbel_of(uint32_t w, float) { return -logf(-logf(uniform_f32(w))); }

// (v, k) <- (v2, k2) when v2 is larger, or equal with the smaller index
template <typename A>
__device__ __forceinline__ void take_best(A &v, int &k, A v2, int k2) {
    if (v2 > v || (v2 == v && k2 < k)) {
        v = v2;
        k = k2;
    }
}

constexpr int kGumbelChunk = 512;   // quads whose exp(L_k - max L) are in shared memory at a time
static_assert(kGumbelOffspring <= 32 && 32 % kGumbelOffspring == 0, "a warp holds whole groups of the CTA's offspring");

// The four L of particles k .. k + 3 (k a multiple of 4, L aligned to 16 bytes), -inf past the last.
template <typename L_t, typename A>
__device__ __forceinline__ void load_quad(const L_t *__restrict__ L, int k, int N, A (&l)[4]) {
    if (k + 3 < N) {
        using V = typename std::conditional<sizeof(L_t) == 2, uint2, uint4>::type;
        union {
            V v[4 * sizeof(L_t) / sizeof(V)];
            L_t e[4];
        } u;
#pragma unroll
        for (int i = 0; i < static_cast<int>(4 * sizeof(L_t) / sizeof(V)); ++i) u.v[i] = __ldg(reinterpret_cast<const V *>(L + k) + i);
#pragma unroll
        for (int i = 0; i < 4; ++i) l[i] = to_acc(u.e[i]);
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) l[i] = k + i < N ? static_cast<A>(to_acc(L[k + i])) : static_cast<A>(-INFINITY);
    }
}

template <int P>
__global__ void __launch_bounds__(kGumbelThreads) gumbel_kernel(const AncestorLaunch G) {
    using lik_t = typename Prec<P>::lik_t;
    using acc_t = typename Prec<P>::acc_t;
    constexpr int kJ = kGumbelOffspring;
    constexpr int kWarps = kGumbelThreads / 32;
    __shared__ acc_t s_v[kWarps][kJ];
    __shared__ int s_k[kWarps][kJ];
    __shared__ uint16_t s_list[kGumbelMaxN / 4];   // quads with a particle that can win
    __shared__ float4 s_el[kGumbelChunk];          // margin * exp(L_k - max L) of a chunk of listed quads
    __shared__ unsigned int s_n;
    __shared__ alignas(16) uint32_t s_rk[20];      // Philox round keys
    __shared__ acc_t s_max[kWarps];
    __shared__ unsigned int s_eb[kJ];              // exp(best - max L) of the CTA, float bits (>= 0)

    const int b = static_cast<int>(blockIdx.x);
    const int g = ancestor_tracker(G, b);
    const int slot = __ldg(G.slots + g);
    const TrackerDev &T = G.trk[slot];
    const TrackerState *st = T.state;
    const int64_t t = st->t;
    if (t <= 0 || (st->status & kStatusTimeout) || !G.frames[slot].active) return;
    const int N = static_cast<int>(T.N);
    const int j0 = (b - __ldg(G.cta_prefix + g)) * kJ;
    const lik_t *__restrict__ L = static_cast<const lik_t *>(T.pl[static_cast<int>((t + 1) & 1)]);
    const uint32_t tctr = static_cast<uint32_t>(t - 1);
    const uint32_t trk_id = T.tracker_id;

    const int nq = (N + 3) >> 2;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // the largest L (NaN aside) and the list of quads that can win
    acc_t mx = -INFINITY;
    for (int q = threadIdx.x; q < nq; q += kGumbelThreads) {
        acc_t l[4];
        load_quad(L, 4 * q, N, l);
#pragma unroll
        for (int i = 0; i < 4; ++i) mx = l[i] > mx ? l[i] : mx;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const acc_t y = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = y > mx ? y : mx;
    }
    if (lane == 0) s_max[wid] = mx;
    if (threadIdx.x == 0) s_n = 0u;
    if (threadIdx.x < 20) s_rk[threadIdx.x] = philox_round_key(threadIdx.x, T.key_lo, T.key_hi);
    const uint4 *rk = reinterpret_cast<const uint4 *>(s_rk);
    // exp(-2.82), rounded down: what the particle of the largest L is sure of
    if (threadIdx.x < kJ) s_eb[threadIdx.x] = __float_as_uint(0.0595f);
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kWarps; ++w) mx = s_max[w] > mx ? s_max[w] : mx;
    const bool finite = mx - mx == static_cast<acc_t>(0);   // else every quad is evaluated in full
    const acc_t line = mx - static_cast<acc_t>(19.5) - static_cast<acc_t>(1e-5) * (mx < 0 ? -mx : mx);
    for (int q0 = 0; q0 < nq; q0 += kGumbelThreads) {
        const int q = q0 + static_cast<int>(threadIdx.x);
        bool keep = false;
        if (q < nq) {
            acc_t l[4];
            load_quad(L, 4 * q, N, l);
            keep = !finite;
#pragma unroll
            for (int i = 0; i < 4; ++i) keep = keep || l[i] >= line;
        }
        const uint32_t mask = __ballot_sync(0xffffffffu, keep);
        unsigned int at = 0;
        if (lane == 0 && mask) at = atomicAdd(&s_n, static_cast<unsigned int>(__popc(mask)));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (keep) s_list[at + __popc(mask & ((1u << lane) - 1u))] = static_cast<uint16_t>(q);
    }
    __syncthreads();
    const int nl = static_cast<int>(s_n);
    const float mxf = static_cast<float>(mx);
    const float margin = 1.001f + 4e-6f * fabsf(mxf);
    const int jj = threadIdx.x % kJ, j = j0 + jj;
    acc_t best = -INFINITY;
    int arg = N;
    for (int c0 = 0; c0 < nl; c0 += kGumbelChunk) {
        const int nc = nl - c0 < kGumbelChunk ? nl - c0 : kGumbelChunk;
        if (c0 > 0) __syncthreads();
        for (int p = threadIdx.x; p < nc; p += kGumbelThreads) {
            acc_t l[4];
            load_quad(L, 4 * static_cast<int>(s_list[c0 + p]), N, l);
            float el[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) el[i] = margin * __expf(static_cast<float>(l[i] - mx));
            s_el[p] = make_float4(el[0], el[1], el[2], el[3]);
        }
        __syncthreads();
        if (j >= N) continue;
        for (int p = threadIdx.x / kJ; p < nc; p += kGumbelThreads / kJ) {
            const int q = s_list[c0 + p], k = 4 * q;
            const float4 e4 = s_el[p];
            const float el[4] = {e4.x, e4.y, e4.z, e4.w};
            const uint4 w = philox4x32_10_keys(make_uint4(static_cast<uint32_t>(q), tctr, 4u + (static_cast<uint32_t>(j) << 8),
                                                     trk_id),
                                          rk);
            const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
            const float eb = __uint_as_float(*reinterpret_cast<volatile unsigned int *>(&s_eb[jj]));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                // (not taken when either side is NaN: evaluated in full)
                if (finite && (1.0f - uniform_f32(ws[i])) * eb > el[i]) continue;
                if (k + i < N) {
                    const acc_t v = to_acc(L[k + i]) + gumbel_of(ws[i], acc_t{});
                    if (v > best || (v == best && k + i < arg && arg < N)) {
                        best = v;
                        arg = k + i;
                        if (finite) atomicMax(&s_eb[jj], __float_as_uint(__expf(static_cast<float>(v - mx))));
                    }
                }
            }
        }
    }
#pragma unroll
    for (int o = 16; o >= kJ; o >>= 1) {
        const acc_t v2 = __shfl_xor_sync(0xffffffffu, best, o);
        const int k2 = __shfl_xor_sync(0xffffffffu, arg, o);
        take_best(best, arg, v2, k2);
    }
    if (lane < kJ) {
        s_v[wid][lane] = best;
        s_k[wid][lane] = arg;
    }
    __syncthreads();
    if (threadIdx.x < kJ) {
        acc_t v = s_v[0][jj];
        int k = s_k[0][jj];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) take_best(v, k, s_v[w][jj], s_k[w][jj]);
        // k = N only if no value compared larger than -inf (a NaN likelihood)
        if (j < N) T.anc[j] = k < N ? k : N - 1;
    }
}

template <int P>
int launch_p(const AncestorLaunch &G, cudaStream_t s) {
    gumbel_kernel<P><<<G.total_ctas, kGumbelThreads, 0, s>>>(G);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace

int launch_gumbel(int precision, const AncestorLaunch &G, void *stream) {
    if (G.total_ctas <= 0 || G.ntrk <= 0) return 0;
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    switch (precision) {
        case 0: return launch_p<0>(G, s);
        case 1: return launch_p<1>(G, s);
        case 2: return launch_p<2>(G, s);
        case 3: return launch_p<3>(G, s);
        default: return 1;
    }
}

}  // namespace pfk
