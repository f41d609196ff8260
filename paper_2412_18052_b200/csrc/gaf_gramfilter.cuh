// Gram-first schedule of Algorithm 1.
//
// The test of step t needs <g_i, g>, |g|^2 and |g_i|^2 where g is the sum of the
// gradients accepted so far.  Dot products are bilinear, so all of them follow from
// the K x K Gram matrix G_ij = <g_i, g_j> of the raw micro-gradients:
//     <g_i, sum_A g_j> = sum_{j in A} G_ji,     |sum_A g_j|^2 = sum_{j,l in A} G_jl.
// The schedule therefore reads every gradient ONCE to build G (binary64 sums), walks
// the K-1 sequential decisions of Algorithm 1 on K^2 scalars in one warp, and
// then reads only the accepted gradients once more to write g/c (Eq. 5):
// ((K + c) b + 4) D bytes instead of one pass over the running sum per step, and no
// grid-wide serialisation per step.  (Up to 8 gradients gaf_fused.cuh writes g/c in the
// first pass, under a predicted accept pattern.)  The accepted gradients are added in processing
// order in binary32, so the macro-gradient is bit-identical to the streaming
// schedules'; the distances differ from theirs only by rounding (the running sum is
// never rounded to binary32 here).
#pragma once

#include "gaf_device.cuh"

namespace gaf {

constexpr int kGsMaxK = 8;                  // gradients the one-pass kernel (gaf_fused.cuh) and the bucketed form handle
constexpr int kGsFlushEvery = 16;           // iterations between binary64 flushes
constexpr int kMsThreads = 512;
constexpr int kMsLongRun = 8;                // chunks per run of the masked-mean pass on long vectors

struct ReplayArgs {
    int K;
    double tau;
    int idx[GAF_MAX_K];                     // original index of the gradient processed at step t
    uint8_t *mask_out;
    float *dist_out;                        // may be null
    int32_t *count_out;
    Control *ctl;
};

// Order-indifferent variant (end of Section 3.1): Algorithm 1 from every seed s with the others following in ring
// order s, s+1, ..., K-1, 0, ..., s-1; the seed with the largest accepted count wins, ties to the smallest s.
struct RingArgs {
    int K;
    double tau;
    uint8_t *mask_out;
    float *dist_out;                        // may be null
    int32_t *count_out;
    int32_t *seed_out;
    Control *ctl;
};

// ---- Algorithm 1 on a K x K Gram matrix in shared memory, by one warp ----
// The order is the ring order from `seed` (seed 0: 0, 1, ..., K-1).  Lane l carries <g_j, running sum> for j = l, l + 32, ...
// (JW values), each summed in processing order; every lane takes every decision.  A step's distance needs a square
// root and a division, 350 cycles when the steps wait for one another; but the decision alone needs the cosine to the
// accuracy of its distance from 1 - tau, so it is taken on a binary32 estimate (error below 1e-6) where that is 1e-5 or more away
// and on Eq. 4 itself otherwise.  The distances are Eq. 4 for all steps at once, afterwards.  (One thread that walked the
// matrix in global memory took 17 us with 16 gradients, 60 with 32 and 150 with 64; this takes 1, 2 and 4.)
template <int JW> struct WalkSteps {        // what lane l knows of the steps of its gradients j
    double p[JW], na[JW], norm_sq[JW];      // <g_j, g>, |g|^2 before the step, sum of |g_i|^2 with g_j
    int count[JW];                          // c if g_j is accepted
};
struct WalkResult {
    unsigned long long bits;                // bit j = gradient j accepted
    int count;
};
template <int JW>
__device__ __forceinline__ WalkResult warp_walk(const double *gram, int K, int seed, double tau, WalkSteps<JW> &st) {
    const int lane = threadIdx.x & 31;
    double pj[JW];
#pragma unroll
    for (int w = 0; w < JW; ++w) {
        pj[w] = lane + 32 * w < K ? gram[seed * K + lane + 32 * w] : 0.0;
        st.p[w] = st.na[w] = st.norm_sq[w] = 0.0;
        st.count[w] = 1;
    }
    double na = gram[seed * K + seed], norm_sq = na;
    const float bound = (float)(1.0 - tau);
    WalkResult r = {1ull << seed, 1};
#pragma unroll 1
    for (int t = 1; t < K; ++t) {
        const int i = seed + t < K ? seed + t : seed + t - K;
        double mine = pj[0];
#pragma unroll
        for (int w = 1; w < JW; ++w) mine = i >= 32 * w ? pj[w] : mine;
        const double p = __shfl_sync(0xFFFFFFFFu, mine, i & 31), ng = gram[i * K + i];
        double row[JW];                     // (loaded before the decision is known)
#pragma unroll
        for (int w = 0; w < JW; ++w) row[w] = lane + 32 * w < K ? gram[i * K + lane + 32 * w] : 0.0;
        const float fp = (float)p, fa = (float)na, fg = (float)ng;
        // (clamped like Eq. 4's cosine: where accepted gradients have nearly cancelled, the sums' rounding can put it outside)
        const float margin = fminf(fmaxf(fp * (rsqrtf(fa) * rsqrtf(fg)), -1.0f), 1.0f) - bound;
        bool accept = margin >= 0.0f;
        const bool safe = fa > 1e-30f && fa < 1e30f && fg > 1e-30f && fg < 1e30f && fabsf(fp) < 1e30f && fabsf(margin) > 1e-5f;
        if (!safe) {
            int ignored = 0;
            accept = cosine_distance(p, na, ng, &ignored) <= tau;
        }
#pragma unroll
        for (int w = 0; w < JW; ++w)
            if (lane + 32 * w == i) { st.p[w] = p; st.na[w] = na; st.norm_sq[w] = norm_sq + ng; st.count[w] = r.count + 1; }
        if (accept) {
            r.bits |= 1ull << i;
            ++r.count;
            na = na + 2.0 * p + ng;         // |g + g_i|^2
            norm_sq += ng;
#pragma unroll
            for (int w = 0; w < JW; ++w) pj[w] += row[w];
        }
    }
    return r;
}
// Mask, distances and count of a walk to their places, by the warp that walked.  Gradient j of the matrix is gradient
// idx[j] of the caller (idx null: the same).
template <int JW>
__device__ __forceinline__ void walk_outputs(const double *gram, int K, int seed, const WalkResult &r, const WalkSteps<JW> &st,
                                             const int *idx, uint8_t *mask_out, float *dist_out, int32_t *count_out,
                                             Control *ctl) {
    const int lane = threadIdx.x & 31;
    int status = 0;
#pragma unroll
    for (int w = 0; w < JW; ++w) {
        const int j = lane + 32 * w;
        if (j >= K) continue;
        const bool accepted = (r.bits >> j) & 1ull;
        double d = 0.0;
        if (j != seed) {
            const double ng = gram[j * K + j];
            d = cosine_distance(st.p[w], st.na[w], ng, &status);
            // the conditioning of the sum that an accept leaves behind
            if (accepted) status |= ill_conditioned(st.count[w], st.norm_sq[w], st.na[w] + 2.0 * st.p[w] + ng);
        }
        const int o = idx ? idx[j] : j;
        mask_out[o] = accepted ? 1 : 0;
        if (dist_out) dist_out[o] = (float)d;
    }
    status = __reduce_or_sync(0xFFFFFFFFu, status);
    if (lane == 0) {
        *count_out = r.count;
        ctl->accept_bits = r.bits;
        ctl->count = r.count;
        // (OR, not store: an earlier kernel of the operation may have raised a bit; the first kernel cleared the word)
        if (status) atomicOr(&ctl->status, status);
    }
}
// The seed with the largest accepted count; the warps of `Sync` share the walks.  `counts`: K ints in shared memory.
template <int JW, typename Sync>
__device__ __forceinline__ int best_seed(const double *gram, int K, double tau, int *counts) {
    const int lane = threadIdx.x & 31;
    for (int s = threadIdx.x >> 5; s < K; s += Sync::threads() / 32) {
        WalkSteps<JW> st;
        const WalkResult r = warp_walk<JW>(gram, K, s, tau, st);
        if (lane == 0) counts[s] = r.count;
    }
    Sync::sync();
    unsigned int key = 0;
#pragma unroll
    for (int w = 0; w < JW; ++w) {
        const int s = lane + 32 * w;
        if (s < K) key = max(key, ((unsigned int)counts[s] << 8) | (unsigned int)(GAF_MAX_K - 1 - s));
    }
    return GAF_MAX_K - 1 - (int)(__reduce_max_sync(0xFFFFFFFFu, key) & 0xFFu);
}

// 16-byte read-only load with an explicit L2 eviction policy.
__device__ __forceinline__ uint4 ld16_policy(const void *p, uint64_t policy) {
    uint4 r;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "l"(p), "l"(policy));
    return r;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_normal() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

template <typename T> struct GsVec;         // one 16-byte load per gradient and iteration
template <> struct GsVec<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ void load(const float *base, int64_t e, uint64_t policy, float (&v)[4]) {
        uint4 r = ld16_policy(base + e, policy);
        v[0] = __uint_as_float(r.x); v[1] = __uint_as_float(r.y);
        v[2] = __uint_as_float(r.z); v[3] = __uint_as_float(r.w);
    }
};
template <> struct GsVec<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ void load(const __nv_bfloat16 *base, int64_t e, uint64_t policy,
                                                float (&v)[8]) {
        uint4 r = ld16_policy(base + e, policy);
        unsigned int w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[2 * k] = bf16_bits_to_float(w[k] & 0xFFFFu);
            v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
        }
    }
};

// Accumulator of the Gram sums of up to 8 gradients on CUDA cores (gaf_fused.cuh, gaf_bucketed.cuh).
// binary32 inputs, up to 4 gradients: binary64.  A product of two binary32 values is exact in binary64, so
// the Gram sums are exact up to binary64 rounding and need no periodic flush; binary64 FMAs (half the
// binary32 rate on this GPU) keep up with HBM here (measured: the same pass time, and a shorter call because
// the flushes are gone).  With 5 to 8 gradients there are up to 1.4 binary64 operations per byte read and
// the long passes, which run under the power cap, lost 8 %: binary32 chains there.
// bfloat16 inputs: binary32 chains (a product of two bfloat16 values is exact in binary32; there are twice
// as many products per byte), widened to binary64 every kGsFlushEvery rounds like the binary32 chains above.
template <typename T, int KT> struct GsAcc {
    using type = float;
    static constexpr bool kPeriodicFlush = true;
};
template <> struct GsAcc<float, 1> { using type = double; static constexpr bool kPeriodicFlush = false; };
template <> struct GsAcc<float, 2> { using type = double; static constexpr bool kPeriodicFlush = false; };
template <> struct GsAcc<float, 3> { using type = double; static constexpr bool kPeriodicFlush = false; };
template <> struct GsAcc<float, 4> { using type = double; static constexpr bool kPeriodicFlush = false; };
__device__ __forceinline__ float gs_fma(float a, float b, float s) { return fmaf(a, b, s); }
__device__ __forceinline__ double gs_fma(float a, float b, double s) { return fma((double)a, (double)b, s); }

// ------------------------------------------------------- masked mean (Eq. 5) --

// Eight consecutive elements as loaded (streaming, evict-first), widened on use.
template <typename T> struct RawOct;
template <> struct RawOct<float> {
    float4 a, b;
    static __device__ __forceinline__ RawOct load(const float *base, int64_t e) {
        const float4 *p = reinterpret_cast<const float4 *>(base + e);
        return {__ldcs(p), __ldcs(p + 1)};
    }
    __device__ __forceinline__ void widen(float (&v)[8]) const {
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
};
template <> struct RawOct<__nv_bfloat16> {
    uint4 r;
    static __device__ __forceinline__ RawOct load(const __nv_bfloat16 *base, int64_t e) {
        return {__ldcs(reinterpret_cast<const uint4 *>(base + e))};
    }
    __device__ __forceinline__ void widen(float (&v)[8]) const {
        const unsigned int w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[2 * k] = bf16_bits_to_float(w[k] & 0xFFFFu);
            v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
        }
    }
};

struct MaskedMeanArgs {
    const void *g[GAF_MAX_K];               // processing order; original order in any-seed mode, where
                                            // the order starts at the winning seed and wraps around
    int K;
    int64_t D;
    float *out;
    const Control *ctl;
    int run;                                // chunks (of one CTA's 512 groups of 8 elements) a CTA takes in a row
    int may_be_done;                        // the Gram pass may have written the mean already (ctl->mean_done)
};

// out = (((g_0 + g_a) + g_b) + ...) / c over the accepted steps a < b < ..., binary32,
// in processing order: the same association as the streaming schedule.  The vector is
// walked from its END: the Gram pass that ran just before walked it from the start, so
// its last-read lines are the ones still in L2.  A CTA takes `run` consecutive chunks, then
// jumps ahead by the whole grid's share: with run = U the grid works on one compact window of
// every vector at any moment (short vectors: every CTA has work); on long vectors longer runs
// keep an SM inside the same pages for several trips, which the address translation needs
// (12 GB through this pass: 5.5 TB/s with run = U, measured, against the 6.5 TB/s it reaches
// on shorter vectors).
template <typename T>
struct MeanVec;
template <> struct MeanVec<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ void widen(const uint4 &r, float (&v)[4]) {
        v[0] = __uint_as_float(r.x); v[1] = __uint_as_float(r.y); v[2] = __uint_as_float(r.z); v[3] = __uint_as_float(r.w);
    }
};
template <> struct MeanVec<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ void widen(const uint4 &r, float (&v)[8]) {
        const unsigned int w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[2 * k] = bf16_bits_to_float(w[k] & 0xFFFFu);
            v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
        }
    }
};

// masked_mean_kernel for short vectors of many gradients, where a call waits for memory latencies and not for bytes: one
// 16-byte vector per thread and sixteen gradients in flight instead of three, the list made by 128 threads instead of one.
// Whole filter calls: 64 bf16 gradients of 20 k / 500 k elements 55.1 -> 40.8 / 68.1 -> 53.5 us, 32 bf16 of 100 k
// 34.5 -> 26.7, 16 fp32 of 100 k 17.7 -> 15.5.
constexpr int kMsShortThreads = 128;
constexpr int kMsShortGrads = 16;
template <typename T>
__global__ void __launch_bounds__(kMsShortThreads) masked_mean_short_kernel(const __grid_constant__ MaskedMeanArgs a) {
    constexpr int N = MeanVec<T>::N;
    __shared__ const T *list[GAF_MAX_K + kMsShortGrads];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const unsigned long long bits = __ldcg(&a.ctl->accept_bits);
    const int seed = __ldcg(&a.ctl->ring_seed), start = seed < 0 ? 0 : seed;
    const int n = __popcll(bits);
    // accepted gradients in processing order: the ring order from `start`
    for (int i = threadIdx.x; i < a.K; i += kMsShortThreads)
        if ((bits >> i) & 1ull) {
            const unsigned long long below = bits & ((1ull << i) - 1ull), from = bits & ~((1ull << start) - 1ull);
            const int rank = i >= start ? __popcll(below & from) : __popcll(from) + __popcll(below);
            list[rank] = static_cast<const T *>(a.g[i]);
        }
    __syncthreads();
    const float cdiv = (float)n;
    const int64_t n_vec = a.D / N, q = (int64_t)blockIdx.x * kMsShortThreads + threadIdx.x;
    if (q < n_vec) {
        const int64_t e = q * N;
        float v[N];
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] = -0.0f;                       // (-0 + x = x for every x)
        for (int i = 0; i < n; i += kMsShortGrads) {
            uint4 w[kMsShortGrads];
#pragma unroll
            for (int g = 0; g < kMsShortGrads; ++g)
                if (i + g < n) w[g] = __ldcs(reinterpret_cast<const uint4 *>(list[i + g] + e));
#pragma unroll
            for (int g = 0; g < kMsShortGrads; ++g)
                if (i + g < n) {
                    float x[N];
                    MeanVec<T>::widen(w[g], x);
#pragma unroll
                    for (int k = 0; k < N; ++k) v[k] += x[k];
                }
        }
#pragma unroll
        for (int h = 0; h < N / 4; ++h)
            *(reinterpret_cast<float4 *>(a.out + e) + h) =
                make_float4(v[4 * h] / cdiv, v[4 * h + 1] / cdiv, v[4 * h + 2] / cdiv, v[4 * h + 3] / cdiv);
    }
    const int64_t tail0 = n_vec * N;
    if (blockIdx.x == 0 && tail0 + threadIdx.x < a.D) {
        const int64_t e = tail0 + threadIdx.x;
        float v = -0.0f;
        for (int i = 0; i < n; ++i) v += load1<T>(list[i], e);
        a.out[e] = v / cdiv;
    }
}

template <typename T>
__global__ void __launch_bounds__(kMsThreads, 2) masked_mean_kernel(const __grid_constant__ MaskedMeanArgs a) {
    __shared__ const T *list[GAF_MAX_K];
    __shared__ int n_list;
    __shared__ float cdiv_s;
    // when launched as a programmatic dependent of the Gram pass: wait until that grid has
    // completed and its writes (the accept bits) are visible; otherwise a no-op
    asm volatile("griddepcontrol.wait;" ::: "memory");
    unsigned long long bits = 0;
    int seed = -1, done = 0;
    if (threadIdx.x == 0) {
        bits = __ldcg(&a.ctl->accept_bits);                      // (independent L2 loads)
        seed = __ldcg(&a.ctl->ring_seed);
        if (a.may_be_done) done = __ldcg(&a.ctl->mean_done);
    }
    if (threadIdx.x == 0) {
        const int start = seed < 0 ? 0 : seed;
        int n = 0;
        for (int t = 0; t < a.K && !done; ++t) {
            const int i = (start + t) % a.K;
            if ((bits >> i) & 1ull) list[n++] = static_cast<const T *>(a.g[i]);
        }
        n_list = n;
        cdiv_s = (float)n;
    }
    __syncthreads();
    const int n = n_list;
    if (n == 0) return;                             // written by the Gram pass
    const float cdiv = cdiv_s;
    const int64_t n_oct = a.D / kOct;
    // U groups of 8 elements per thread and round (two for 2-byte inputs, so that as many bytes
    // are in flight as with 4-byte inputs); loads stay packed until they are added
    constexpr int U = sizeof(T) == 2 ? 2 : 1;
    constexpr int kChunk = 3;                       // further gradients fetched together
    const int64_t n_chunks = (n_oct + kMsThreads - 1) / kMsThreads;
    const int64_t run = a.run;
    for (int64_t base = (int64_t)blockIdx.x * run; base < n_chunks; base += (int64_t)gridDim.x * run)
    for (int64_t rr = 0; rr < run && base + rr < n_chunks; rr += U) {
        int64_t e[U];
        bool ok[U];
        RawOct<T> first[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t o = (base + rr + u) * kMsThreads + threadIdx.x;
            ok[u] = rr + u < run && o < n_oct;
            e[u] = (n_oct - 1 - (ok[u] ? o : 0)) * kOct;
            if (ok[u]) first[u] = RawOct<T>::load(list[0], e[u]);
        }
        float v[U][8];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (ok[u]) first[u].widen(v[u]);
        for (int i = 1; i < n; i += kChunk) {
            RawOct<T> w[U][kChunk];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int j = 0; j < kChunk; ++j)
                    if (ok[u] && i + j < n) w[u][j] = RawOct<T>::load(list[i + j], e[u]);
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int j = 0; j < kChunk; ++j)
                    if (ok[u] && i + j < n) {
                        float x[8];
                        w[u][j].widen(x);
#pragma unroll
                        for (int k = 0; k < 8; ++k) v[u][k] += x[k];
                    }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (ok[u]) {
#pragma unroll
                for (int k = 0; k < 8; ++k) v[u][k] = v[u][k] / cdiv;
                store8(a.out, e[u], v[u], true);
            }
    }
    const int64_t tail0 = n_oct * kOct;
    if (blockIdx.x == 0 && tail0 + threadIdx.x < a.D) {
        const int64_t e = tail0 + threadIdx.x;
        float v = load1<T>(list[0], e);
        for (int i = 1; i < n; ++i) v += load1<T>(list[i], e);
        a.out[e] = v / cdiv;
    }
}

}  // namespace gaf
