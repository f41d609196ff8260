// Gram-first schedule of Algorithm 1 for 2 to 8 gradients in (mostly) ONE pass over the inputs.
//
// Every gradient is needed for the Gram matrix before the first decision of Algorithm 1 is known, and the
// accepted ones again for g/c (Eq. 5).  What that second pass fetches is most of what a call costs beyond reading
// the inputs once.  But WHICH gradients will be accepted can be told from a part of them: cosines estimated on m
// elements are off by about 1/sqrt(m), a thousandth on a million.  So:
//   stream   one CTA per SM; a producer thread keeps a ring of tiles (all K gradients x a chunk of D) in shared
//            memory filled with bulk copies (cp.async.bulk), about 200 KB in flight per SM;
//   sample   the first few tiles of every CTA are spread evenly over the vectors (every CTA at another phase, so
//            that all parts of a network are represented); the consumer warps take their Gram sums and KEEP them;
//   predict  CTA 0 totals the sample's sums, walks Algorithm 1 on them and tells every CTA, while the ring fills;
//   write    the mean under the predicted pattern is written for the kept tiles, and from then on for every
//            tile together with its Gram sums;
//   decide   at the end Algorithm 1 is walked on the full Gram matrix.  If it decides as predicted the
//            result is complete; otherwise the mean is formed again from the accepted gradients.
// The prediction decides which stores are made early, never a value: mask, distances and count come from the
// full sums, and the mean is the same additions in the same order (binary32, processing order, one division by
// c) whichever pass writes it.  Short vectors go without a prediction (see filter_shape in gaf_api.cu): after the
// decision the mean of the tiles that are still in the rings (25 MB of gradients) is written from there, and the
// others are fetched again, from L2 for the most part.
//
// Two forms of one kernel, with the same sums in the same order, hence the same outputs:
//   ONE      every CTA is resident at once.  At the end every CTA stores its partial sums; CTA 0 totals them, walks
//            Algorithm 1, writes the outputs and tells every CTA (bounded waits, GAF_STATUS_TIMEOUT).  After a wrong prediction the ring is run once more over the accepted gradients, the
//            last tiles first (what L2 still holds).
//   two      the last CTA to take a ticket decides, and masked_mean_kernel, launched behind, returns at once when
//            the result is already written.  The only wait for other CTAs is the prediction's, and it is short:
//            a CTA that does not get one goes on without.  The same form gives the pairwise distances.
// The kernel is launched with programmatic stream serialisation: it waits for whatever precedes it on the stream
// before it touches global memory, and lets the launch behind it be placed once its own streaming (two) or
// deciding (ONE) is over.
//
// Gram sums of a tile: up to 4 binary32 gradients in binary64 registers (products exact); otherwise binary32
// chains (64 products; 128 of bfloat16 values, whose products are exact), two to a register pair, widened to
// binary64 in shared memory; 7 and 8 bfloat16 gradients by warp-level MMAs (gaf_gram_mma.cuh's mapping, operands
// from shared memory, chains of 128).
#pragma once

#include <type_traits>

#include "gaf_device.cuh"
#include "gaf_gram_mma.cuh"
#include "gaf_gram_tc.cuh"
#include "gaf_gramfilter.cuh"

// Bound by HBM: (K b + 4) D bytes.  Measured (back to back, outputs of their own; before: second pass over the accepted
// gradients in every call): 4 x 11.2 M fp32 56 -> 46 us (225 MB: 4.8 TB/s), 8 x 40 M fp32 373 -> 244 us (5.9 TB/s), 8 x 124 M fp32
// 987 -> 750 us, 8 x 100 M bf16 515 -> 368 us (5.4 TB/s), 8 x 1 G bf16 4.66 -> 3.7 ms.  Of the 46 us, 4 pass until every CTA has its sample
// tiles, 6 more until the mean of the first is written (the ring is full after 4), 4 between the last CTA's last
// tile and the decision.  What decided the shape:
//   - with 8 consumer warps the Gram sums and the mean of a tile took longer than its copy (K = 8: 4.5 TB/s);
//   - a ring with fewer bytes in flight (3 tiles) cost 14 % with 8 gradients;
//   - not waiting for the prediction but fetching the tiles from before it again at the end: 70 against 46 us, because
//     a poll from an SM with a full ring in flight takes 4 us and more;
//   - CTAs that all read all partial sums, or all poll one counter, wait 3 to 6 us for the few lines that everybody reads.
namespace gaf {

constexpr unsigned int kFusedSpinLimit = 1u << 22;   // polls of an L2 round trip each: seconds
constexpr unsigned int kFusedSampleLimit = 64;       // two-launch form: polls for the prediction, some tens of microseconds
constexpr unsigned int kFusedCopyLimit = 1u << 19;   // attempts of up to 2 us at a ring barrier

// Test hook: no CTA is shown sums or patterns; none of the sample; no tile is copied; none from the second lap of the ring on.
constexpr int kWithholdAll = 1, kWithholdSample = 2, kWithholdTiles = 4, kWithholdLaterTiles = 8;

// Consumer warps work in groups; a tile belongs to one group, the groups take the tiles in turn.  One more warp
// produces.  15 warps of at most 128 registers.
constexpr int kFilterGroups = 2;
constexpr int kFilterGroupWarps = 7;
constexpr int kFilterGroupThreads = kFilterGroupWarps * 32;
constexpr int kFilterWarps = kFilterGroups * kFilterGroupWarps;
constexpr int kFilterConsumers = kFilterWarps * 32;
constexpr int kFilterThreads = kFilterConsumers + 32;
constexpr int kFilterMaxStages = 24;
constexpr int kFilterMaxCtas = 160;
// Two gradients: a shorter ring of smaller tiles, 112 KB in flight (2 x 30 M fp32: 63.3 us with 28 KB tiles in 172 KB, 62.1 with
// 14 KB tiles, 58.8 in the shorter ring as well; a third of the traffic are writes there).
constexpr int kFilterRingBytes = 206 << 10;
constexpr int kFilterPairRingBytes = 130 << 10;

// Tile of K gradients: kVecs groups of 4 elements per thread of a group and gradient, 20 to 43 KB in all.  Five and six gradients
// (50 M elements fp32): tiles of 18 and 21 KB in ten and eight stages took 167 and 190 us for all pairs, 222 and 239 for the
// filter, of twice that in four 141 and 170, 192 and 227; bfloat16 (60 M) 113 -> 88 and 127 -> 106, 153 -> 136 and 165 -> 160.
// But a filter call on a shorter bfloat16 input waits longer for its prediction behind large tiles (5 x 5.5 M 24.6 us with
// small ones, 26.8 with large ones; 6 x 8 M 33.9, 36.5): there the large ones are a form of their own (LONG).
template <typename T, int KT> constexpr bool kTwoTileForms = std::is_same<T, __nv_bfloat16>::value && (KT == 5 || KT == 6);
template <typename T, int KT, bool LONG = false> struct FilterTile {
    static constexpr bool kMma = std::is_same<T, __nv_bfloat16>::value && KT >= 7;
    static constexpr int kVecs = KT == 2 ? 8 / int(sizeof(T)) : (KT <= 4 || (KT <= 6 && (LONG || !kTwoTileForms<T, KT>)) ? 8 / int(sizeof(T)) : 4 / int(sizeof(T)));
    static constexpr int kElems = kVecs * 4 * kFilterGroupThreads;
    // (the MMA fragments of eight rows are read together: 64 bytes between rows keep them apart in the banks)
    static constexpr int kPitch = kElems * int(sizeof(T)) + (kMma ? 64 : 0);
    static constexpr int kBytes = KT * kPitch;
    // A multiple of the groups: a stage then always belongs to the same group, which has seen its previous tile land
    // before it waits for the next one (copies complete in any order; a barrier's parity tells only two phases apart).
    static constexpr int kRing = KT == 2 ? kFilterPairRingBytes : kFilterRingBytes;
    static constexpr int kFit = kRing / kBytes < kFilterMaxStages ? kRing / kBytes : kFilterMaxStages;
    static constexpr int kStages = kFit / kFilterGroups * kFilterGroups;
    static constexpr int kBatch = KT <= 4 ? 2 : 1;  // groups of 4 elements a thread loads together
};

struct GramFusedArgs {
    const void *g[kGsMaxK];                 // processing order (original order in any-seed and pairwise mode)
    int64_t D;
    int tile_elems;                         // elements of a tile per gradient (a multiple of 64, at most FilterTile::kElems)
    int rounds;                             // tiles per CTA
    int sample;                             // tiles per CTA in the sample; 0 = no prediction
    int evict_first;                        // what is read once gives way in L2 first
    void *partials;                         // [pair][kFilterMaxCtas]: TaggedSum (ONE) or double
    unsigned long long *sample_partials;    // [pair][kFilterMaxCtas]: binary32 sum and tag
    unsigned long long *verdicts;           // [2][kFilterMaxCtas][16]: a line per CTA for the predicted and one for the decided pattern
    unsigned int tag;                       // ONE: a number no other launch has
    float *out;                             // D floats
    ReplayArgs replay;                      // used when ring.K == 0
    RingArgs ring;                          // any-seed mode when ring.K > 0
    float *pair_dist_out;                   // pairwise mode: K x K distances instead of the walk and the mean
    double *pair_gram_out;                  // pairwise mode: optional copy of the Gram matrix
    unsigned int spin_limit;                // polls a waiting CTA makes before it gives up
    unsigned int copy_limit;                // attempts at a ring barrier before a wait gives up
    int test_withhold;                      // test hook, normally 0: what is never given or shown (kWithhold...)
};

// What CTAs tell one another carries the call's tag in every word, so that the reader polls the data itself: one
// trip to L2 and back after the last store, where an arrival counter (stores, release, counter, poll, then the
// loads) took three.  A binary64 sum travels as two words, half a sum and the tag or its complement each; a pattern as two
// words as well, whole in both; every word is written and read as a whole.  What an earlier call left in the place
// carries another tag, and 64 bits of a number that another operation left there would have to agree.  Every word
// has ONE reader: 148 CTAs that read the same lines at the same time wait 3 to 6 us for them.
// (The sample's sums travel as one word each, binary32 and the tag: all that can come of a stale one is a wrong prediction.)
__device__ __forceinline__ void st_word(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
struct TaggedSum { unsigned long long w[2]; };
__device__ __forceinline__ void st_tagged(TaggedSum *p, double v, unsigned int tag) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned long long lo = (b << 32) | tag, hi = (b & 0xFFFFFFFF00000000ull) | (unsigned int)~tag;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ TaggedSum ld_tagged(const TaggedSum *p) {
    TaggedSum t;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(t.w[0]), "=l"(t.w[1]) : "l"(p) : "memory");
    return t;
}
__device__ __forceinline__ bool tagged_value(const TaggedSum &t, double &v, unsigned int tag) {
    v = __longlong_as_double((long long)((t.w[0] >> 32) | (t.w[1] & 0xFFFFFFFF00000000ull)));
    return (unsigned int)t.w[0] == tag && (unsigned int)t.w[1] == (unsigned int)~tag;
}
__device__ __forceinline__ void st_pattern(unsigned long long *p, unsigned int pattern, unsigned int tag) {
    const unsigned long long hi = (unsigned long long)pattern << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(hi | tag), "l"(hi | (unsigned int)~tag) : "memory");
}
__device__ __forceinline__ bool ld_pattern(const unsigned long long *p, unsigned int &pattern, unsigned int tag) {
    unsigned long long a, b;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
    pattern = (unsigned int)(a >> 32);
    return (unsigned int)a == tag && (unsigned int)b == (unsigned int)~tag && (unsigned int)(b >> 32) == pattern;
}
// Bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) into shared memory, counted on `bar`.
__device__ __forceinline__ void bulk_load(uint32_t dst_smem, const void *src, uint32_t bytes, uint64_t *bar, uint64_t policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 ::"r"(dst_smem), "l"(src), "r"(bytes), "r"(tc_smem_u32(bar)), "l"(policy)
                 : "memory");
}

// The consumer warps among themselves (barrier 0 is the whole CTA's).
struct FilterConsumers {
    static __device__ __forceinline__ void sync() {
        asm volatile("barrier.cta.sync 1, %0;" ::"n"(kFilterConsumers) : "memory");
    }
    static __device__ __forceinline__ constexpr int threads() { return kFilterConsumers; }
};

// Two binary32 values in one register pair, and the two-wide instructions on them (each half rounds as the scalar
// instruction does).
typedef unsigned long long Pair;
__device__ __forceinline__ Pair pair_of(float lo, float hi) {
    Pair r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void pair_split(Pair p, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p)); }
__device__ __forceinline__ Pair pair_fma(Pair a, Pair b, Pair c) {
    Pair r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ Pair pair_add(Pair a, Pair b) {
    Pair r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ Pair pair_mul(Pair a, Pair b) {
    Pair r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

template <typename T> struct Quad;          // four consecutive elements as they lie in a tile, widened to two pairs
template <> struct Quad<float> {
    static __device__ __forceinline__ void load(const unsigned char *p, Pair (&x)[2]) {
        const ulonglong2 r = *reinterpret_cast<const ulonglong2 *>(p);
        x[0] = r.x; x[1] = r.y;
    }
};
template <> struct Quad<__nv_bfloat16> {
    static __device__ __forceinline__ void load(const unsigned char *p, Pair (&x)[2]) {
        const uint2 r = *reinterpret_cast<const uint2 *>(p);
        x[0] = pair_of(bf16_bits_to_float(r.x & 0xFFFFu), __uint_as_float(r.x & 0xFFFF0000u));
        x[1] = pair_of(bf16_bits_to_float(r.y & 0xFFFFu), __uint_as_float(r.y & 0xFFFF0000u));
    }
};

// Division of binary32 values by a count c of 1 to 8, correctly rounded.  A power of two: multiplication by its
// inverse.  Else x / c = RN(x zh + RN(x zl)) with zh = RN(1 / c), zl = RN(1 / c - zh) (Brisebarre, Muller and
// Raina, "Accelerating correctly rounded floating-point division when the divisor is known in advance", IEEE
// Trans. Computers 2004), which holds for c = 3, 5, 6 and 7 for every significand (all 2^23 checked) as long as x zl
// is a normal number; values outside [2^-90, 2^100] (zeros, infinities among them) take the division.
struct CountDivider {
    float c;
    Pair zh2, zl2;
    bool pow2;
    __device__ __forceinline__ explicit CountDivider(int count) {
        c = (float)count;
        const float zh = 1.0f / c, zl = fmaf(-zh, c, 1.0f) / c;
        zh2 = pair_of(zh, zh);
        zl2 = pair_of(zl, zl);
        pow2 = (count & (count - 1)) == 0;
    }
    __device__ __forceinline__ void divide(Pair (&x)[2]) const {
        if (pow2) {
            x[0] = pair_mul(x[0], zh2); x[1] = pair_mul(x[1], zh2);
            return;
        }
        float v[4];
        pair_split(x[0], v[0], v[1]);
        pair_split(x[1], v[2], v[3]);
        const float least = fminf(fminf(fabsf(v[0]), fabsf(v[1])), fminf(fabsf(v[2]), fabsf(v[3])));
        const float most = fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3])));
        if (least >= 8.077935669463161e-28f && most <= 1.2676506002282294e+30f) {      // 2^-90, 2^100
            x[0] = pair_fma(x[0], zh2, pair_mul(x[0], zl2));
            x[1] = pair_fma(x[1], zh2, pair_mul(x[1], zl2));
        } else {
            x[0] = pair_of(v[0] / c, v[1] / c);
            x[1] = pair_of(v[2] / c, v[3] / c);
        }
    }
};

// An accept pattern in one word: the rows, and the row the order starts at.  0 = not known.
__device__ __forceinline__ unsigned int pack_pattern(unsigned int bits, int start) {
    return 0x80000000u | ((unsigned int)start << 8) | bits;
}

// Order of a CTA's tiles: the S sample rounds (one in each of S segments of `seg` rounds, at the CTA's phase), then
// the others in ascending order.
__device__ __forceinline__ int round_of_visit(int v, int S, int seg, int phase) {
    if (v < S) return v * seg + phase;
    const int u = v - S, m = seg - 1;
    if (u >= S * m) return u + S;
    const int b = u / m, i = u - b * m;
    return b * seg + i + (i >= phase ? 1 : 0);
}

// Warp-wide sums of NP per-lane values by recursive halving, added to dst: in each round a lane keeps the half of its
// values chosen by one bit of its number, adding its partner's copy of that half, so about NP shuffles (not 5 NP)
// leave every sum in one lane.  A fixed tree.
template <int NP, int D, typename Acc>
struct HalvingSums {
    static constexpr int H = (NP + 1) / 2;
    static __device__ __forceinline__ void run(Acc *v, int lane, int base, int limit, double *dst) {
        const bool upper = (lane & D) != 0;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const Acc hi = i + H < NP ? v[i + H] : Acc(0);
            const Acc send = upper ? v[i] : hi, keep = upper ? hi : v[i];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, D);
        }
        // this lane now holds entries base .. of the half it chose; the upper half may be one shorter
        HalvingSums<H, D / 2, Acc>::run(v, lane, base + (upper ? H : 0), upper ? min(limit, base + NP) : min(limit, base + H), dst);
    }
};
template <int NP, typename Acc>
struct HalvingSums<NP, 0, Acc> {
    static __device__ __forceinline__ void run(Acc *v, int, int base, int limit, double *dst) {
#pragma unroll
        for (int i = 0; i < NP; ++i)
            if (base + i < limit) dst[base + i] += (double)v[i];
    }
};

template <typename T, int KT, bool ONE, bool LONG>
__global__ void __launch_bounds__(kFilterThreads, 1)
gram_filter_kernel(const __grid_constant__ GramFusedArgs a) {
    using Tile = FilterTile<T, KT, LONG>;
    using Sync = FilterConsumers;
    constexpr int NP = KT * (KT + 1) / 2;
    constexpr int CW = kFilterWarps, NG = kFilterGroups, kStages = Tile::kStages, kPitch = Tile::kPitch;
    extern __shared__ __align__(128) unsigned char ring[];      // [stage][gradient][pitch]
    __shared__ uint64_t full[kStages], empty[kStages];
    // the tile in a stage, written by the producer: first element, and from kTileShift on its length.  One word, so that a consumer
    // that stopped waiting for it sees one tile or another (at the start: none), never the start of one and the length of another.
    __shared__ unsigned long long stage_tile[kStages];
    constexpr int kTileShift = 48;
    static_assert(Tile::kElems < 1 << (64 - kTileShift), "a tile's length fits above its first element");
    __shared__ double ssum[CW][NP];         // per-warp sums
    __shared__ double sgram[KT * KT];
    __shared__ int seed_counts[KT];
    __shared__ const T *list[kGsMaxK];      // accepted gradients in the order they are added
    __shared__ int n_list;                  // c
    __shared__ int sh_ok, sh_again;         // outcome of a wait; how many tiles are fetched a second time
    __shared__ int sh_done;                 // two launches: every CTA has written the decided mean
    __shared__ unsigned int sh_pred;        // predicted and decided pattern
    __shared__ volatile unsigned int sh_final;
    __shared__ volatile int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Control *ctl = a.replay.ctl;

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) { tc_mbar_init(&full[s], 1); tc_mbar_init(&empty[s], kFilterGroupWarps); stage_tile[s] = 0ull; }
        sh_pred = 0u; sh_final = 0u; sh_ok = 1; sh_again = 0; sh_done = 1; abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = tid; i < CW * NP; i += kFilterThreads) (&ssum[0][0])[i] = 0.0;
    __syncthreads();
    // Launched with programmatic stream serialisation, this grid may be placed while the launch before
    // it on the stream is still winding down: nothing that launch (or the producer of the gradients)
    // wrote may be touched before it has completed.  A no-op after an ordinary predecessor.
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const int rounds = a.rounds, S = a.sample;
    constexpr int kAlign = 16 / (int)sizeof(T);
    const int64_t Dv = a.D / kAlign * kAlign;                   // what the copies cover

    if (warp == CW) {
        // ------------------------------------------------------------------ producer ----
        const int te = a.tile_elems, seg = S > 0 ? rounds / S : 1, phase = S > 0 ? (int)blockIdx.x % seg : 0;
        const int given = a.test_withhold & kWithholdTiles ? 0 : (a.test_withhold & kWithholdLaterTiles ? min(rounds, kStages) : rounds);
        int it = 0;                         // tiles since the start, of both passes
        // (bulk copies whose lines give way first are the better ones while the gradients of a call are of L2's size; see the host)
        const uint64_t once = a.evict_first ? l2_policy_evict_first() : l2_policy_evict_normal();
        // no prediction: the tiles that leave the ring are read again soon (4 x 2 M fp32 14.0 -> 12.8 us, 8 x 2 M 27.5 -> 27.0)
        const uint64_t again = ONE && S == 0 ? l2_policy_evict_last() : once;
        auto fill = [&](int v, const void *const *rows, int n_rows) {
            const int s = it % kStages;
            if (it >= kStages && !tc_mbar_wait(&empty[s], (uint32_t)((it / kStages - 1) & 1), &abort_flag, a.copy_limit))
                return false;
            const int r = round_of_visit(v, S, seg, phase);
            const int64_t e0 = ((int64_t)r * gridDim.x + blockIdx.x) * te, left = Dv - e0;
            const int n = left >= te ? te : (left > 0 ? (int)left : 0);
            *reinterpret_cast<volatile unsigned long long *>(&stage_tile[s]) = (unsigned long long)e0 | (unsigned long long)n << kTileShift;
            if (n > 0) {
                const uint32_t bytes = (uint32_t)n * (uint32_t)sizeof(T), dst = tc_smem_u32(ring + (size_t)s * Tile::kBytes);
                tc_mbar_arrive_expect_tx(&full[s], bytes * (uint32_t)n_rows);
                for (int g = 0; g < n_rows; ++g)
                    bulk_load(dst + (uint32_t)(g * kPitch), static_cast<const T *>(rows[g]) + e0, bytes, &full[s], it < rounds - kStages ? again : once);
            } else {
                tc_mbar_arrive(&full[s]);
            }
            ++it;
            return true;
        };
        if (lane == 0)
            for (int v = 0; v < given; ++v)
                if (!fill(v, a.g, KT)) break;
        __syncwarp();
        __syncthreads();                    // the consumers have decided whether there is a second pass
        if (ONE && lane == 0 && !abort_flag)
            for (int v = sh_again - 1; v >= 0; --v)
                if (!fill(v, reinterpret_cast<const void *const *>(list), n_list)) break;
        // after a wait that gave up, which may be one of the second pass: the copies in flight must land before the CTA leaves
        // its shared memory
        if (lane == 0 && (abort_flag || sh_again > 0))
            for (int i = it > kStages ? it - kStages : 0; i < it; ++i)
                for (unsigned int spin = 0; spin < kFusedCopyLimit; ++spin)
                    if (tc_mbar_try(&full[i % kStages], (uint32_t)((i / kStages) & 1), 2000u)) break;
        return;
    }

    // ---------------------------------------------------------------------- consumers ----
    const int group = warp / kFilterGroupWarps, gwarp = warp - group * kFilterGroupWarps, gtid = gwarp * 32 + lane;
    if (blockIdx.x == 0 && tid == 0) ctl->status = 0;
    // Two launches may be replayed from a graph: their tag is the number of the call among such calls on the workspace, from 1 on
    // (gaf_workspace_init clears the words that carry it); the count moves on when every CTA of the call has taken its ticket.
    // (The tags of the one-launch form have the upper bit set.)
    const unsigned int tag = ONE ? a.tag | 0x80000000u : (__ldcg(&ctl->two_launch_calls) + 1u) & 0x7FFFFFFFu;

    // Accumulators: binary64, pairs of binary32 chains, or (MMA) this lane's fragment of the 8 x 8 matrix.
    constexpr bool kF64 = !GsAcc<T, KT>::kPeriodicFlush;
    using Acc = typename std::conditional<kF64, double, Pair>::type;
    constexpr int NA = Tile::kMma ? 1 : NP;
    // tiles between flushes: each half of a pair sums 64 products (128 of bfloat16 values)
    constexpr int kChainTiles = 128 / int(sizeof(T)) / Tile::kVecs > 0 ? 128 / int(sizeof(T)) / Tile::kVecs : 1;
    Acc acc[NA];
#pragma unroll
    for (int p = 0; p < NA; ++p) acc[p] = Acc(0);
    float frag[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    double frag_sum[2] = {0.0, 0.0};
    int chain = 0;
    auto flush = [&]() {
        if constexpr (Tile::kMma) {
            const int g = lane >> 2, t = lane & 3;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = 2 * t + h;
                if (g <= j && j < KT) ssum[warp][g * KT - g * (g - 1) / 2 + (j - g)] += frag_sum[h];
                frag_sum[h] = 0.0;
            }
        } else if constexpr (kF64) {
            HalvingSums<NP, 16, double>::run(acc, lane, 0, NP, ssum[warp]);
#pragma unroll
            for (int p = 0; p < NP; ++p) acc[p] = 0.0;
        } else {
            float v[NP];
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                float lo, hi;
                pair_split(acc[p], lo, hi);
                v[p] = lo + hi;
                acc[p] = Pair(0);
            }
            HalvingSums<NP, 16, float>::run(v, lane, 0, NP, ssum[warp]);
        }
        chain = 0;
    };
    // One tile: its Gram sums (GRAM) and the mean of its rows under a pattern (MEAN).
    auto process = [&](auto gram_tag, auto mean_tag, int s, unsigned int from, unsigned int before, const CountDivider &div) {
        constexpr bool GRAM = decltype(gram_tag)::value, MEAN = decltype(mean_tag)::value;
        constexpr int B = Tile::kBatch;
        const unsigned char *tile = ring + (size_t)s * Tile::kBytes;
        const unsigned long long where = *reinterpret_cast<volatile unsigned long long *>(&stage_tile[s]);
        const int n = (int)(where >> kTileShift);
        float *out = a.out + (where & ((1ull << kTileShift) - 1ull));
        if constexpr (GRAM && Tile::kMma) {
            const int g = lane >> 2, t = lane & 3;
            const unsigned char *row = tile + (g < KT ? g : 0) * kPitch;
#pragma unroll
            for (int u = 0; u < Tile::kElems / 32 / kFilterGroupWarps; ++u) {
                const int e = (u * kFilterGroupWarps + gwarp) * 32 + t * 8;
                uint4 r = make_uint4(0u, 0u, 0u, 0u);
                if (g < KT && e < n) r = *reinterpret_cast<const uint4 *>(row + e * 2);
                mma_bf16_16816(frag, r.x, r.y);
                mma_bf16_16816(frag, r.z, r.w);
                if (u % 4 == 3) {
                    frag_sum[0] += (double)frag[0]; frag_sum[1] += (double)frag[1];
                    frag[0] = frag[1] = frag[2] = frag[3] = 0.0f;
                }
            }
            static_assert(!Tile::kMma || Tile::kElems / 32 / kFilterGroupWarps % 4 == 0, "chains end inside a tile");
        }
        if constexpr (MEAN || !Tile::kMma) {
            constexpr bool SUMS = GRAM && !Tile::kMma;
#pragma unroll
            for (int u0 = 0; u0 < Tile::kVecs; u0 += B) {
                Pair x[B][KT][2];
                int e[B];
#pragma unroll
                for (int b = 0; b < B; ++b) {
                    e[b] = ((u0 + b) * kFilterGroupThreads + gtid) * 4;
                    if (e[b] < n) {
#pragma unroll
                        for (int g = 0; g < KT; ++g)
                            if (SUMS || (((from | before) >> g) & 1u)) Quad<T>::load(tile + g * kPitch + e[b] * (int)sizeof(T), x[b][g]);
                    }
                }
#pragma unroll
                for (int b = 0; b < B; ++b)
                    if (SUMS && e[b] < n) {
                        if constexpr (kF64) {
                            float f[KT][4];
#pragma unroll
                            for (int g = 0; g < KT; ++g) { pair_split(x[b][g][0], f[g][0], f[g][1]); pair_split(x[b][g][1], f[g][2], f[g][3]); }
                            int p = 0;
#pragma unroll
                            for (int g = 0; g < KT; ++g)
#pragma unroll
                                for (int h = g; h < KT; ++h, ++p)
#pragma unroll
                                    for (int k = 0; k < 4; ++k) acc[p] = gs_fma(f[g][k], f[h][k], acc[p]);
                        } else if constexpr (!Tile::kMma) {
                            int p = 0;
#pragma unroll
                            for (int g = 0; g < KT; ++g)
#pragma unroll
                                for (int h = g; h < KT; ++h, ++p)
                                    acc[p] = pair_fma(x[b][g][1], x[b][h][1], pair_fma(x[b][g][0], x[b][h][0], acc[p]));
                        }
                    }
                if constexpr (MEAN) {
                    // in processing order (-0 + x = x for every x, so the first addition is a copy)
                    Pair v[B][2];
#pragma unroll
                    for (int b = 0; b < B; ++b) v[b][0] = v[b][1] = 0x8000000080000000ull;
#pragma unroll
                    for (int g = 0; g < KT; ++g)
                        if ((from >> g) & 1u) {
#pragma unroll
                            for (int b = 0; b < B; ++b) { v[b][0] = pair_add(v[b][0], x[b][g][0]); v[b][1] = pair_add(v[b][1], x[b][g][1]); }
                        }
                    if (before) {
#pragma unroll
                        for (int g = 0; g < KT; ++g)
                            if ((before >> g) & 1u) {
#pragma unroll
                                for (int b = 0; b < B; ++b) { v[b][0] = pair_add(v[b][0], x[b][g][0]); v[b][1] = pair_add(v[b][1], x[b][g][1]); }
                            }
                    }
#pragma unroll
                    for (int b = 0; b < B; ++b)
                        if (e[b] < n) {
                            div.divide(v[b]);
                            float4 r;
                            pair_split(v[b][0], r.x, r.y);
                            pair_split(v[b][1], r.z, r.w);
                            __stcs(reinterpret_cast<float4 *>(out + e[b]), r);
                        }
                }
            }
        }
        if constexpr (GRAM && !Tile::kMma && !kF64) {
            if (++chain == kChainTiles) flush();
        }
    };
    using std::false_type;
    using std::true_type;
    // (After a wait that ran out the warp goes on with whatever the stage holds: the call is not valid, but every word that stage_tile
    // can hold lies inside the output.)
    auto wait_full = [&](int it) {
        const uint32_t parity = (uint32_t)((it / kStages) & 1);
        if (!tc_mbar_try(&full[it % kStages], parity, 2000u) &&
            !tc_mbar_wait(&full[it % kStages], parity, &abort_flag, a.copy_limit) && lane == 0)
            atomicOr(&ctl->status, GAF_STATUS_TIMEOUT);
        __syncwarp();
    };
    auto release = [&](int it) {
        __syncwarp();
        if (lane == 0) tc_mbar_arrive(&empty[it % kStages]);
    };
    // This CTA's sum of pair `tid` so far, over its warps in a fixed order (threads below NP).
    auto cta_sum = [&]() {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < CW; ++w) s += ssum[w][tid];
        return s;
    };
    // row-major pair index -> (i, j), i <= j
    auto pair_at = [](int p, int &i, int &j) {
        i = 0;
        while (p >= KT - i) { p -= KT - i; ++i; }
        j = i + p;
    };
    // Sums of all CTAs in a fixed order into sgram: warp w takes the pairs w, w + CW, ...  `load(pair, cta)` fetches a sum,
    // `value(raw, x)` returns whether it is there; every warp polls its own at most `limit` times.  All of a warp's
    // loads are issued before any is looked at: this is a wait for L2 that every CTA shares (one pair after the other, and one
    // load after the other, 8 bf16 gradients of 5 M took 35.0 us, now 32.2; 8 fp32 of 16 M 109.6, now 105.5).
    auto total = [&](auto load, auto value, unsigned int limit) {
        constexpr int R = (kFilterMaxCtas + 31) / 32, M = (NP + CW - 1) / CW;
        double part[M][R];
        bool all = false;
        for (unsigned int polls = 0; polls <= limit && !all; ++polls) {
            decltype(load(0, 0)) raw[M][R];
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int k = 0; k < R; ++k)
                    raw[m][k] = load(min(warp + m * CW, NP - 1), min(lane + 32 * k, (int)gridDim.x - 1));
            bool mine = true;
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    double x;
                    mine = value(raw[m][k], x) && mine;
                    part[m][k] = lane + 32 * k < (int)gridDim.x ? x : 0.0;
                }
            all = __all_sync(0xFFFFFFFFu, mine);
        }
        if (!all) {
            if (lane == 0) sh_ok = 0;
        } else {
            double s[M];
#pragma unroll
            for (int m = 0; m < M; ++m) {
                s[m] = 0.0;
#pragma unroll
                for (int k = 0; k < R; ++k) s[m] += part[m][k];
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1)
#pragma unroll
                for (int m = 0; m < M; ++m) s[m] += shfl_down_f64(s[m], d);
#pragma unroll
            for (int m = 0; m < M; ++m)
                if (lane == 0 && warp + m * CW < NP) {
                    int i, j;
                    pair_at(warp + m * CW, i, j);
                    sgram[i * KT + j] = s[m];
                    sgram[j * KT + i] = s[m];
                }
        }
        Sync::sync();
        return sh_ok != 0;
    };

    // CTA 0, one warp: a pattern to every CTA's line; the other CTAs, one thread: wait for it (0 = it did not come).
    auto tell = [&](unsigned long long *lines, unsigned int pattern) {
        for (int cta = lane; cta < (int)gridDim.x; cta += 32) st_pattern(lines + cta * 16, pattern, tag);
    };
    auto hear = [&](const unsigned long long *lines, unsigned int limit, bool withheld) {
        for (unsigned int polls = 0; polls <= limit; ++polls) {
            unsigned int pattern;
            if (ld_pattern(lines + blockIdx.x * 16, pattern, tag) && !withheld) return pattern;
        }
        return 0u;
    };

    // Algorithm 1 (or its order-indifferent variant) on sgram, by all consumers: decided pattern into sh_final and, if
    // there are lines, to every CTA; mask, distances and count to their places.
    auto decide = [&](unsigned long long *lines) {
        const bool any_seed = a.ring.K > 0;
        const double tau = any_seed ? a.ring.tau : a.replay.tau;
        const int seed = any_seed ? best_seed<1, Sync>(sgram, KT, tau, seed_counts) : 0;
        if (warp == 0) {
            WalkSteps<1> st;
            const WalkResult r = warp_walk<1>(sgram, KT, seed, tau, st);
            const unsigned int final = pack_pattern((unsigned int)r.bits, seed);
            if (lines != nullptr) tell(lines, final);
            if (lane == 0) {
                sh_final = final;
                ctl->ring_seed = any_seed ? seed : -1;
                if (any_seed) *a.ring.seed_out = seed;
            }
            if (any_seed) walk_outputs<1>(sgram, KT, seed, r, st, nullptr, a.ring.mask_out, a.ring.dist_out, a.ring.count_out, ctl);
            else walk_outputs<1>(sgram, KT, seed, r, st, a.replay.idx, a.replay.mask_out, a.replay.dist_out, a.replay.count_out, ctl);
        }
        Sync::sync();
    };

    // Two gradients (ONE): the result is the mean of both or the first alone.  When the latest two calls on this workspace
    // ended alike, that pattern is taken instead of a sample's, and nobody waits for one (0 both, 1 the first alone; from 2 on: they
    // differed, bit 0 the latest).  Read before this CTA hands in its sums, hence before CTA 0 can have decided.
    const unsigned int hint = KT == 2 && ONE && S > 0 ? __ldcg(&ctl->pair_hint) : 2u;
    const bool sampling = S > 0 && hint >= 2u;
    // (a group's tiles have its number modulo NG, in a second pass too)
    auto next_of_group = [&](int it) { return it + (group + NG - it % NG) % NG; };
    unsigned int pred = hint < 2u ? pack_pattern(hint == 1u ? 1u : 3u, 0) : 0u;
    int v = group;
    if (sampling) {
        const CountDivider none(1);
        for (; v < S; v += NG) {
            wait_full(v);
            process(true_type(), false_type(), v % kStages, 0u, 0u, none);
        }
    }
    if (sampling) {
        flush();
        Sync::sync();
        if (tid < NP)
            st_word(a.sample_partials + (size_t)tid * kFilterMaxCtas + blockIdx.x,
                    ((unsigned long long)__float_as_uint((float)cta_sum()) << 32) | tag);
        const unsigned int limit = ONE && !(a.test_withhold & kWithholdSample) ? a.spin_limit : kFusedSampleLimit;
        const bool withheld = (a.test_withhold & (kWithholdAll | kWithholdSample)) != 0;
        if (blockIdx.x == 0) {
            const bool known = total(
                [&](int p, int cta) { return ld_word(a.sample_partials + (size_t)p * kFilterMaxCtas + cta); },
                [&](unsigned long long w, double &x) {
                    x = (double)__uint_as_float((unsigned int)(w >> 32));
                    return (unsigned int)w == tag && !withheld;
                }, limit);
            const bool any_seed = a.ring.K > 0;
            const double tau = any_seed ? a.ring.tau : a.replay.tau;
            const int seed = known && any_seed ? best_seed<1, Sync>(sgram, KT, tau, seed_counts) : 0;
            if (warp == 0 && known) {
                WalkSteps<1> st;
                const unsigned int guess = pack_pattern((unsigned int)warp_walk<1>(sgram, KT, seed, tau, st).bits, seed);
                if (lane == 0) sh_pred = guess;
                tell(a.verdicts, guess);
            }
        } else if (tid == 0) {
            sh_pred = hear(a.verdicts, limit, withheld);
        }
        Sync::sync();
        pred = sh_pred;
        if (tid == 0) sh_ok = 1;
    }
    if (pred) {
        const unsigned int bits = pred & 0xFFu, before = bits & ((1u << ((pred >> 8) & 0xFu)) - 1u), from = bits ^ before;
        const CountDivider div(__popc(bits));
        for (int w = group; sampling && w < S; w += NG) {
            process(false_type(), true_type(), w % kStages, from, before, div);
            release(w);
        }
        if constexpr (KT == 2 && ONE) {
            // without a sample the sums are cut where a call that takes one cuts them: same bits whatever the calls before it left
            // (as a condition inside the loop below: 0.3 to 2 us more per call)
            if (S > 0 && !sampling) {
                for (; v < S; v += NG) {
                    wait_full(v);
                    process(true_type(), true_type(), v % kStages, from, before, div);
                    release(v);
                }
                flush();
            }
        }
        for (; v < rounds; v += NG) {
            wait_full(v);
            process(true_type(), true_type(), v % kStages, from, before, div);
            release(v);
        }
    } else {
        // (the last tiles stay in the ring: their mean is written from there)
        const CountDivider none(1);
        for (int w = group; sampling && w < S && w < rounds - kStages; w += NG) release(w);
        for (; v < rounds; v += NG) {
            wait_full(v);
            process(true_type(), false_type(), v % kStages, 0u, 0u, none);
            if (v < rounds - kStages) release(v);
        }
    }
    flush();
    if constexpr (!ONE) {
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        __syncthreads();                    // (lets the producer go)
    } else {
        Sync::sync();
    }
    if (tid < NP) {
        double s = cta_sum();
        if (blockIdx.x == 0 && Dv < a.D) {
            // the last elements, which no copy covers
            int i, j;
            pair_at(tid, i, j);
            const T *x = static_cast<const T *>(a.g[i]), *y = static_cast<const T *>(a.g[j]);
            for (int64_t e = Dv; e < a.D; ++e) s += (double)load1<T>(x, e) * (double)load1<T>(y, e);
        }
        if constexpr (ONE) st_tagged(static_cast<TaggedSum *>(a.partials) + (size_t)tid * kFilterMaxCtas + blockIdx.x, s, tag);
        else static_cast<double *>(a.partials)[(size_t)tid * kFilterMaxCtas + blockIdx.x] = s;
    }
    // two launches: the pattern under which this CTA wrote its share of the mean, for the CTA that decides (in the CTA's line,
    // behind the words that carry a tag)
    if constexpr (!ONE) {
        if (tid == 0 && a.pair_dist_out == nullptr) a.verdicts[blockIdx.x * 16 + 8] = pred;
    }

    // ---- decide ----
    if constexpr (ONE) {
        unsigned long long *const lines = a.verdicts + kFilterMaxCtas * 16;
        if (blockIdx.x == 0) {
            if (total([&](int p, int cta) { return ld_tagged(static_cast<const TaggedSum *>(a.partials) + (size_t)p * kFilterMaxCtas + cta); },
                      [&](const TaggedSum &w, double &x) { return tagged_value(w, x, tag) && !(a.test_withhold & kWithholdAll); },
                      a.spin_limit)) {
                decide(lines);
            }
        } else if (tid == 0) {
            sh_final = hear(lines, a.spin_limit, (a.test_withhold & kWithholdAll) != 0);
        }
        Sync::sync();
        if (sh_final == 0u) {
            if (tid == 0) atomicOr(&ctl->status, GAF_STATUS_TIMEOUT);
            __syncthreads();
            return;
        }
    } else {
        Sync::sync();
        if (tid == 0) sh_ok = take_last_ticket(&ctl->ticket, gridDim.x) ? 1 : 0;
        Sync::sync();
        if (!sh_ok) return;
        if (tid == 0) ctl->two_launch_calls = tag;
        const unsigned int share = a.pair_dist_out == nullptr && tid < (int)gridDim.x ? (unsigned int)__ldcg(a.verdicts + tid * 16 + 8) : 0u;
        total([&](int p, int cta) { return __ldcg(static_cast<const double *>(a.partials) + (size_t)p * kFilterMaxCtas + cta); },
              [](double w, double &x) { x = w; return true; }, 0u);
        if (a.pair_dist_out != nullptr) {
            // pairwise mode: Eq. 4 for every pair
            if (tid < KT * KT) {
                const int i = tid / KT, j = tid % KT;
                const double gii = sgram[i * KT + i], gjj = sgram[j * KT + j], gij = sgram[tid];
                int status = 0;
                const double d = (i == j && gii > 0.0) ? 0.0 : cosine_distance(gij, gii, gjj, &status);
                a.pair_dist_out[tid] = (float)d;
                if (a.pair_gram_out) a.pair_gram_out[tid] = gij;
                if (status) atomicOr(&ctl->status, status);
            }
            return;
        }
        decide(nullptr);
        // the result is complete if EVERY CTA wrote its share under the decided pattern, wherever it had the pattern from
        if (tid < (int)gridDim.x && share != sh_final) sh_done = 0;
    }
    const int kept = pred ? 0 : min(rounds, kStages);           // tiles that are still in the ring
    if (tid == 0) {
        const unsigned int bits = sh_final & 0xFFu;
        const int start = (int)((sh_final >> 8) & 0xFu);
        int n = 0;
        for (int t = 0; t < KT; ++t) {
            const int i = start + t >= KT ? start + t - KT : start + t;
            if ((bits >> i) & 1u) list[n++] = static_cast<const T *>(a.g[i]);
        }
        n_list = n;
        if (KT == 2 && ONE && S > 0 && blockIdx.x == 0) {
            const unsigned int outcome = n == 1 ? 1u : 0u;
            ctl->pair_hint = outcome == (hint & 1u) ? outcome : (2u | outcome);
        }
        if (ONE) sh_again = sh_final != pred ? rounds - kept : 0;
    }
    Sync::sync();
    const int c = n_list;
    if constexpr (!ONE) {
        if (tid == 0) ctl->mean_done = sh_done;
    } else {
        // the launch behind this one on the stream may be placed from here on (it waits for this grid itself)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        __syncthreads();                    // the producer learns whether it is wanted again
    }
    // the last elements, which no copy covers (two launches: the second may have nothing to do)
    if ((!ONE || blockIdx.x == 0) && Dv + tid < a.D) {
        const int64_t e = Dv + tid;
        float x = load1<T>(list[0], e);
        for (int i = 1; i < c; ++i) x += load1<T>(list[i], e);
        a.out[e] = x / (float)c;
    }
    if constexpr (ONE) {
        if (sh_final == pred) return;
        const CountDivider div(c);
        const unsigned int bits = sh_final & 0xFFu, before = bits & ((1u << ((sh_final >> 8) & 0xFu)) - 1u);
        for (int w = next_of_group(rounds - kept); w < rounds; w += NG) {
            process(false_type(), true_type(), w % kStages, bits ^ before, before, div);
            release(w);
        }
        // the accepted gradients of the other tiles again, compacted to the first rows in the order they are added
        for (int it = next_of_group(rounds); it < 2 * rounds - kept; it += NG) {
            wait_full(it);
            process(false_type(), true_type(), it % kStages, (1u << c) - 1u, 0u, div);
            release(it);
        }
    }
}

}  // namespace gaf
