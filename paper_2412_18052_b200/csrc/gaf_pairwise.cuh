// Pairwise cosine-distance matrix (Eq. 4 for every pair of K micro-gradients):
// Gram matrix G = X X^T over D, then dist_ij = 1 - G_ij / (sqrt(G_ii) sqrt(G_jj)).
//
// What the Gram kernels for more than 8 gradients share (gaf_gram_digits.cuh and gaf_gram_tc.cuh on tensor cores,
// gaf_gram_mma.cuh, gaf_gram_panel.cuh on CUDA cores): the K x K matrix cut into 8 x 8 tiles of pairs, per-CTA
// binary64 partial sums in a [tile pair][slice][64] layout, and the finishing kernel that totals
// the slices in a fixed order and derives the distances, or whose last CTA walks Algorithm 1 on the matrix.
#pragma once

#include "gaf_device.cuh"
#include "gaf_gramfilter.cuh"

namespace gaf {

constexpr int kGramTile = 8;
constexpr int kGramMaxSlices = 296;     // most D-slices (CTAs along x)

struct GramArgs {
    const void *g[GAF_MAX_K];
    int K;
    int64_t D;
    int tiles;              // ceil(K / 8)
    double *partials;       // [tile_pair][slice][64]
    double *gram;           // [K][K]
    float *dist_out;        // [K][K]
    double *gram_out;       // [K][K] or null
    Control *ctl;
    int slices;
    ReplayArgs replay;      // replay.K > 0: Algorithm 1 on the matrix instead of the distances of all pairs
    RingArgs ring;          // ring.K > 0: its order-indifferent variant
};

// Decode the linear upper-triangle tile index into (ti, tj), ti <= tj.
__device__ __forceinline__ void tile_pair(int idx, int tiles, int &ti, int &tj) {
    ti = 0;
    while (idx >= tiles - ti) { idx -= tiles - ti; ++ti; }
    tj = ti + idx;
}

// One CTA per tile pair: sums the slices in a fixed order.  For the distances of all pairs it sums the diagonal entries of its
// gradients as well, in the same order, and is done; for the filter it writes its entries, both triangles, and the last CTA to finish
// takes the decisions on the matrix.
constexpr int kFinishParts = 16;        // each entry's slices are summed in 16 independent chains
// (10 loads of a chain in flight together are what 148 slices have; with 4, and the distances by a last CTA, 2 us more)
constexpr int kFinishLoads = 10;
struct FinishBlock {
    static __device__ __forceinline__ void sync() { __syncthreads(); }
    static __device__ __forceinline__ constexpr int threads() { return 64 * kFinishParts; }
};
__device__ __forceinline__ double finish_chain(const double *src, int chain, int slices) {
    const int per = (slices + kFinishParts - 1) / kFinishParts, lo = chain * per, hi = min(slices, lo + per);
    double s = 0.0;
    for (int base = lo; base < hi; base += kFinishLoads) {
        double v[kFinishLoads];
#pragma unroll
        for (int k = 0; k < kFinishLoads; ++k) v[k] = base + k < hi ? __ldcg(src + (size_t)(base + k) * 64) : 0.0;
#pragma unroll
        for (int k = 0; k < kFinishLoads; ++k) s += v[k];
    }
    return s;
}
__global__ void __launch_bounds__(64 * kFinishParts) gram_finish_kernel(const __grid_constant__ GramArgs a) {
    __shared__ double part[kFinishParts][64];
    __shared__ double diag[kFinishParts][16];
    __shared__ double sgram[GAF_MAX_K * GAF_MAX_K];
    __shared__ bool is_last;
    int ti, tj;
    tile_pair(blockIdx.x, a.tiles, ti, tj);
    const int p = threadIdx.x & 63, chain = threadIdx.x >> 6;
    const bool pairs = a.replay.K == 0 && a.ring.K == 0;
    // launched as a programmatic dependent of the Gram kernel: wait until that grid has completed
    // and its partial sums are visible (a no-op in an ordinary launch)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // a dependent of this launch may be placed now (it waits for this grid before it touches global memory)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    part[chain][p] = finish_chain(a.partials + (size_t)blockIdx.x * a.slices * 64 + p, chain, a.slices);
    if (pairs && p < 16) {
        // |g|^2 of the eight gradients of the rows and the eight of the columns
        const int t = p < 8 ? ti : tj, tp = t * a.tiles - t * (t - 1) / 2;
        diag[chain][p] = finish_chain(a.partials + (size_t)tp * a.slices * 64 + (p & 7) * 9, chain, a.slices);
    }
    __syncthreads();
    if (threadIdx.x < 64) {
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < kFinishParts; ++c) s += part[c][p];
        int r = p / kGramTile, c = p % kGramTile;
        int i = ti * kGramTile + r, j = tj * kGramTile + c;
        if (i < a.K && j < a.K && i <= j) {
            if (pairs) {
                double gii = 0.0, gjj = 0.0;
#pragma unroll
                for (int k = 0; k < kFinishParts; ++k) { gii += diag[k][r]; gjj += diag[k][8 + c]; }
                int status = 0;
                const float d = i == j && gii > 0.0 ? 0.0f : (float)cosine_distance(s, gii, gjj, &status);
                a.dist_out[(size_t)i * a.K + j] = d;
                a.dist_out[(size_t)j * a.K + i] = d;
                if (a.gram_out) {
                    a.gram_out[(size_t)i * a.K + j] = s;
                    a.gram_out[(size_t)j * a.K + i] = s;
                }
                if (status) atomicOr(&a.ctl->status, status);
            } else {
                a.gram[(size_t)i * a.K + j] = s;
                a.gram[(size_t)j * a.K + i] = s;
            }
        }
    }
    if (pairs) return;
    __syncthreads();
    if (threadIdx.x == 0) is_last = take_last_ticket(&a.ctl->ticket, gridDim.x);
    __syncthreads();
    if (!is_last) return;
    const int K = a.K;
    const bool any_seed = a.ring.K > 0;
    // by processing step, or by original index (the ring orders start anywhere)
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
        const int t = e / K, u = e % K;
        const int i = any_seed ? t : a.replay.idx[t], j = any_seed ? u : a.replay.idx[u];
        sgram[e] = __ldcg(a.gram + (size_t)i * K + j);
    }
    __syncthreads();
    const double tau = any_seed ? a.ring.tau : a.replay.tau;
    int *counts = reinterpret_cast<int *>(&part[0][0]);
    const int seed = any_seed ? best_seed<2, FinishBlock>(sgram, K, tau, counts) : 0;
    if (threadIdx.x < 32) {
        WalkSteps<2> st;
        const WalkResult r = warp_walk<2>(sgram, K, seed, tau, st);
        if (any_seed) walk_outputs<2>(sgram, K, seed, r, st, nullptr, a.ring.mask_out, a.ring.dist_out, a.ring.count_out, a.ctl);
        else walk_outputs<2>(sgram, K, seed, r, st, a.replay.idx, a.replay.mask_out, a.replay.dist_out, a.replay.count_out, a.ctl);
        if (threadIdx.x == 0) {
            a.ctl->ring_seed = any_seed ? seed : -1;
            if (any_seed) *a.ring.seed_out = seed;
        }
    }
}

}  // namespace gaf
