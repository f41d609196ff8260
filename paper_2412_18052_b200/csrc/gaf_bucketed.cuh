// Bucketed variant: the parameter vector is cut into S consecutive buckets (for example the
// tensors of a network, or the buckets of a ring all-reduce) and Algorithm 1 + Eq. 5 run on every
// bucket independently.  Gram-first, as for the whole vector: one pass builds a K x K Gram matrix
// PER BUCKET, a small kernel walks Algorithm 1 per bucket, one pass writes every bucket's g/c.
//
// Work split: every CTA owns one contiguous range of the D elements, and inside it handles the part of every bucket
// that intersects the range.  A (CTA c, bucket b) intersection writes its partial Gram sums to slot c + b, which is
// unique because both indices only grow along the vector.  The per-bucket totals are taken over the CTAs in
// ascending order (fixed order).  Every further bucket costs a CTA a reduction and a memory latency, and two thirds of a network's
// tensors have a few hundred elements, so a bucket counts as kBkBucketCost elements when the ranges are cut (62 tensors of
// ResNet18, 4 fp32 gradients, whole call: 75.0 us with equal shares, 74.0 / 72.3 / 71.6 with a bucket counted as 1024 / 2048 / 5000
// elements; 200 buckets of 3 M: 34.9, 30.0, 28.6, 29.2.  Before, with a walk that recomputed every range in every thread and a
// mean pass with two barriers a bucket: 78.6 and 47.4 us; 20 buckets of 100 k: 28.1, now 12.8).  Eight 16-byte vectors in flight per
// thread of the mean pass, whatever the number of gradients, and no eviction hint beyond L2: 71.6 -> 63.7.
#pragma once

#include "gaf_device.cuh"
#include "gaf_gramfilter.cuh"

namespace gaf {

constexpr int kBkThreads = 512;
constexpr int kBkMaxBuckets = GAF_MAX_BUCKETS;
constexpr int kBkMaxCtas = 296;

struct BucketTable {
    int S;
    int64_t off[kBkMaxBuckets + 1];         // element offsets, off[0] = 0, off[S] = D
};

// Largest b with off[b] <= e (e < D).
__device__ __forceinline__ int bucket_of(const BucketTable &bt, int64_t e) {
    int lo = 0, hi = bt.S;                  // off[lo] <= e < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (bt.off[mid] <= e) lo = mid; else hi = mid;
    }
    return lo;
}

// Where CTA c's range starts, out of G equal shares of (elements + kBkBucketCost per bucket): a multiple of 8.
constexpr int kBkBucketCost = 3072;
__device__ __forceinline__ int64_t cta_start(const BucketTable &bt, int64_t D, int c, int G) {
    if (c <= 0) return 0;
    if (c >= G) return D;
    const int64_t x = (D + (int64_t)kBkBucketCost * bt.S) * c / G;
    int lo = 0, hi = bt.S;                  // largest b with off[b] + cost b <= x
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (bt.off[mid] + (int64_t)kBkBucketCost * mid <= x) lo = mid; else hi = mid;
    }
    const int64_t into = x - (bt.off[lo] + (int64_t)kBkBucketCost * (lo + 1));
    const int64_t e = bt.off[lo] + (into > 0 ? into : 0), end = bt.off[lo + 1];
    return (e < end ? e : end) / kOct * kOct;
}
__device__ __forceinline__ void cta_range(const BucketTable &bt, int64_t D, int c, int G, int64_t &lo, int64_t &hi) {
    lo = cta_start(bt, D, c, G);
    hi = cta_start(bt, D, c + 1, G);
}

struct BucketGramArgs {
    const void *g[kGsMaxK];                 // processing order
    int64_t D;
    int64_t keep_elems;                     // the last so many elements of every CTA's range are loaded "keep in L2"
    int evict_first;                        // the others are the first to leave it
    double *partials;                       // [slot][64], slot = cta + bucket
    Control *ctl;
};

template <typename T, int KT>
__global__ void __launch_bounds__(kBkThreads, (KT <= 4 ? 2 : 1))
bucket_gram_kernel(const __grid_constant__ BucketGramArgs a, const __grid_constant__ BucketTable bt) {
    constexpr int NP = KT * (KT + 1) / 2;
    constexpr int N = GsVec<T>::N;
    constexpr int U = KT <= 2 ? 4 / KT : 1; // vectors of a gradient a thread has in flight
    static_assert(kGsFlushEvery % U == 0, "the sums are flushed between rounds");
    __shared__ double sacc[kBkThreads / 32][NP];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const T *row[KT];
#pragma unroll
    for (int r = 0; r < KT; ++r) row[r] = static_cast<const T *>(a.g[r]);
    // the mean pass walks every CTA's range from its end: the end of the range is asked to stay in L2
    const uint64_t pol_first = a.evict_first ? l2_policy_evict_first() : l2_policy_evict_normal(), pol_last = l2_policy_evict_last();
    int64_t lo, hi;
    cta_range(bt, a.D, blockIdx.x, gridDim.x, lo, hi);
    // a programmatic dependent of what precedes it on the stream (a no-op after an ordinary launch)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (blockIdx.x == 0 && threadIdx.x == 0) a.ctl->status = 0;     // first kernel of the operation
    if (lo >= hi) return;
    int b = bucket_of(bt, lo);
    while (true) {
        const int64_t s0 = lo > bt.off[b] ? lo : bt.off[b];
        const int64_t s1 = hi < bt.off[b + 1] ? hi : bt.off[b + 1];
        if (s1 > s0) {
            for (int p = lane; p < NP; p += 32) sacc[warp][p] = 0.0;
            __syncwarp();
            using Acc = typename GsAcc<T, KT>::type;
            Acc acc[NP];
#pragma unroll
            for (int p = 0; p < NP; ++p) acc[p] = Acc(0);
            auto flush = [&]() {
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    Acc v = acc[p];
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, d);
                    if (lane == 0) sacc[warp][p] += (double)v;
                    acc[p] = Acc(0);
                }
            };
            // s0 is a multiple of 8 elements (bucket offsets and CTA ranges are), so vector loads are aligned
            const int64_t n_vec = (s1 - s0) / N;
            int since_flush = 0;
            // warp-uniform trip count: the flush shuffles across the whole warp
            for (int64_t qw = threadIdx.x & ~31; qw < n_vec; qw += U * kBkThreads) {
                float x[U][KT][N];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t q = qw + u * kBkThreads + lane;
                    const uint64_t pol = (s0 + q * N >= hi - a.keep_elems) ? pol_last : pol_first;
                    if (q < n_vec) {
#pragma unroll
                        for (int r = 0; r < KT; ++r) GsVec<T>::load(row[r], s0 + q * N, pol, x[u][r]);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (qw + u * kBkThreads + lane >= n_vec) break;
                    int p = 0;
#pragma unroll
                    for (int r = 0; r < KT; ++r)
#pragma unroll
                        for (int c = r; c < KT; ++c, ++p) {
                            Acc s = acc[p];
#pragma unroll
                            for (int k = 0; k < N; ++k) s = gs_fma(x[u][r][k], x[u][c][k], s);
                            acc[p] = s;
                        }
                }
                if (GsAcc<T, KT>::kPeriodicFlush && (since_flush += U) == kGsFlushEvery) { flush(); since_flush = 0; }
            }
            const int64_t t0 = s0 + n_vec * N;          // fewer than N leftover elements
            if (t0 + threadIdx.x < s1) {
                float x[KT];
#pragma unroll
                for (int r = 0; r < KT; ++r) x[r] = load1<T>(row[r], t0 + threadIdx.x);
                int p = 0;
#pragma unroll
                for (int r = 0; r < KT; ++r)
#pragma unroll
                    for (int c = r; c < KT; ++c, ++p) acc[p] = gs_fma(x[r], x[c], acc[p]);
            }
            flush();
            __syncthreads();
            if (threadIdx.x < NP) {
                double s = 0.0;
                for (int w = 0; w < kBkThreads / 32; ++w) s += sacc[w][threadIdx.x];
                a.partials[(size_t)(blockIdx.x + b) * 64 + threadIdx.x] = s;
            }
            __syncthreads();
        }
        if (bt.off[b + 1] >= hi || b + 1 >= bt.S) break;
        ++b;
    }
    // the per-bucket walk is launched as a programmatic dependent: its blocks may be placed now
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

struct BucketWalkArgs {
    int K;
    int64_t D;
    int ctas;                               // grid of the Gram pass
    double tau;
    const double *partials;
    uint8_t *mask_out;                      // [S][K], by original index
    float *dist_out;                        // [S][K] or null
    int32_t *count_out;                     // [S]
    unsigned long long *bits;               // [S], bit t = step t accepted (workspace)
    int idx[kGsMaxK];                       // original index of step t
    Control *ctl;
};

// One CTA per bucket (64 pairs x 16 chains of threads): totals over the intersecting CTAs in
// ascending order, then the walk by one warp.
constexpr int kWalkChains = 16;
__global__ void __launch_bounds__(64 * kWalkChains)
bucket_walk_kernel(const __grid_constant__ BucketWalkArgs a, const __grid_constant__ BucketTable bt) {
    __shared__ double sgram[kGsMaxK * kGsMaxK];
    __shared__ double part[kWalkChains][64];
    __shared__ int first, last;
    __shared__ unsigned char meets[kBkMaxCtas];
    const int b = blockIdx.x, K = a.K, NP = K * (K + 1) / 2;
    const int64_t b0 = bt.off[b], b1 = bt.off[b + 1];
    if (threadIdx.x == 0) { first = a.ctas; last = -1; }
    __syncthreads();
    // CTAs of the Gram pass whose range meets [b0, b1): one thread per CTA looks
    if ((int)threadIdx.x < a.ctas) {
        int64_t lo, hi;
        cta_range(bt, a.D, threadIdx.x, a.ctas, lo, hi);
        const bool m = (lo > b0 ? lo : b0) < (hi < b1 ? hi : b1);
        meets[threadIdx.x] = m ? 1 : 0;
        if (m) { atomicMin(&first, (int)threadIdx.x); atomicMax(&last, (int)threadIdx.x); }
    }
    static_assert(kBkMaxCtas <= 64 * kWalkChains, "one thread per CTA");
    __syncthreads();
    const int p = threadIdx.x & 63, chain = threadIdx.x >> 6;
    // programmatic dependent of the Gram pass: wait for that grid and its partial sums; the mean pass
    // behind this kernel may be placed at once (it waits for this grid in turn)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    {
        const int n = last - first + 1;
        const int per = (n + kWalkChains - 1) / kWalkChains;
        const int c0 = first + chain * per, c1 = min(last + 1, c0 + per);
        double s = 0.0;
        if (p < NP) {
#pragma unroll 4
            for (int c = c0; c < c1; ++c)
                if (meets[c]) s += __ldcg(a.partials + (size_t)(c + b) * 64 + p);
        }
        part[chain][p] = s;
    }
    __syncthreads();
    if ((int)threadIdx.x < NP) {
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < kWalkChains; ++c) s += part[c][threadIdx.x];
        int r = 0, rem = threadIdx.x;
        while (rem >= K - r) { rem -= K - r; ++r; }
        const int cc = r + rem;
        sgram[r * K + cc] = s;
        sgram[cc * K + r] = s;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        WalkSteps<1> st;
        const WalkResult r = warp_walk<1>(sgram, K, 0, a.tau, st);
        if (threadIdx.x == 0) a.bits[b] = r.bits;
        walk_outputs<1>(sgram, K, 0, r, st, a.idx, a.mask_out + (size_t)b * K, a.dist_out ? a.dist_out + (size_t)b * K : nullptr,
                        a.count_out + b, a.ctl);
    }
}

struct BucketMeanArgs {
    const void *g[kGsMaxK];                 // processing order
    int K;
    int64_t D;
    float *out;
    int evict_first;                        // what is read leaves L2 first
    const unsigned long long *bits;         // [S]
};

template <typename T, int KM>               // KM: at most so many gradients
__global__ void __launch_bounds__(kBkThreads, 2)
bucket_mean_kernel(const __grid_constant__ BucketMeanArgs a, const __grid_constant__ BucketTable bt) {
    constexpr int N = MeanVec<T>::N;        // elements of a 16-byte load
    constexpr int U = 8 / KM;               // vectors of a gradient a thread has in flight
    const uint64_t policy = a.evict_first ? l2_policy_evict_first() : l2_policy_evict_normal();
    int64_t lo, hi;
    cta_range(bt, a.D, blockIdx.x, gridDim.x, lo, hi);
    // programmatic dependent of the per-bucket walk: wait for its accept bits
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (lo >= hi) return;
    // The range is walked from its END (buckets last to first, each from its end): the Gram pass walked it from the start,
    // so its last-read lines are the ones still in L2.  Every thread looks at the bucket's bits itself: no barriers.
    int b = bucket_of(bt, hi - 1);
    while (true) {
        const int64_t s0 = lo > bt.off[b] ? lo : bt.off[b];
        const int64_t s1 = hi < bt.off[b + 1] ? hi : bt.off[b + 1];
        if (s1 > s0) {
            const unsigned int bits = (unsigned int)__ldcg(a.bits + b);
            const float cdiv = (float)__popc(bits);
            const int64_t n_vec = (s1 - s0) / N;
            for (int64_t o = threadIdx.x; o < n_vec; o += U * kBkThreads) {
                uint4 w[U][KM];
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int t = 0; t < KM; ++t)
                        if (((bits >> t) & 1u) && o + u * kBkThreads < n_vec)
                            w[u][t] = ld16_policy(static_cast<const T *>(a.g[t]) + s0 + (n_vec - 1 - o - u * kBkThreads) * N, policy);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (o + u * kBkThreads >= n_vec) break;
                    const int64_t e = s0 + (n_vec - 1 - o - u * kBkThreads) * N;
                    float v[N];
#pragma unroll
                    for (int k = 0; k < N; ++k) v[k] = -0.0f;       // (-0 + x = x for every x)
#pragma unroll
                    for (int t = 0; t < KM; ++t)
                        if ((bits >> t) & 1u) {
                            float x[N];
                            MeanVec<T>::widen(w[u][t], x);
#pragma unroll
                            for (int k = 0; k < N; ++k) v[k] += x[k];
                        }
#pragma unroll
                    for (int h = 0; h < N / 4; ++h)
                        __stcs(reinterpret_cast<float4 *>(a.out + e) + h,
                               make_float4(v[4 * h] / cdiv, v[4 * h + 1] / cdiv, v[4 * h + 2] / cdiv, v[4 * h + 3] / cdiv));
                }
            }
            const int64_t t0 = s0 + n_vec * N;
            if (t0 + threadIdx.x < s1) {
                const int64_t e = t0 + threadIdx.x;
                float v = -0.0f;
                for (int t = 0; t < a.K; ++t)
                    if ((bits >> t) & 1u) v += load1<T>(static_cast<const T *>(a.g[t]), e);
                a.out[e] = v / cdiv;
            }
        }
        if (bt.off[b] <= lo || b == 0) break;
        --b;
    }
}

}  // namespace gaf
