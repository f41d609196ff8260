// Gram matrix G = X X^T of binary32 gradients (one, or 9 to 64 of them; 2 to 8 go to the one-pass kernel of gaf_fused.cuh)
// on the 5th-generation tensor cores, every gradient read ONCE, with sums that are exact integers.
//
// A binary32 value is brought to 31-bit fixed point under a power of two of its gradient and cut into four signed
// base-256 digits, x 2^k = d0 2^24 + d1 2^16 + d2 2^8 + d3.  The digits of all K gradients are the rows of ONE 8-bit
// matrix, row s KP + i = digit s of gradient i (KP = K rounded up to 8, 16 at least), so that its product with itself
// (tcgen05.mma.kind::i8, 8-bit x 8-bit -> 32-bit integers) holds every product of digits of every pair.  Integer sums
// are exact and do not depend on their order, up to 2^17 products a sum; they are put together in 64-bit integers and
// binary64 at the end.  What is rounded at all is the value to fixed point, by half a unit of 2^-k at most: a fixed part of the largest
// magnitudes, so that elements far below them lose bits, the smallest all.  For normal values half a unit is about 2^-23 of their
// root mean square.  Largest error of all pairs, of the norms' product, against the chains of 64 rounded products of a kernel on the binary32
// pipes (24 x 3 M): normal values 1e-10 / 3e-9, Student's t of 3 degrees 3e-10 / 7e-9, lognormal of sigma 2 2e-9 / 8e-8, 200 tensors of
// lognormal scales 7e-12 / 5e-9.  (A gradient with one element of 1 and all others 2^-26, against one of ones: 4e-6 of the norms' product, where
// chains leave 3e-9.)
//
// The power of two.  A CTA takes its share in periods of at most 1023 x 128 elements.  At the start of each it looks at the first tile of
// each of its teams and allows for elements 2^5 times as large: half a unit is at most 2^-25 of the largest magnitude that the CTA sampled of
// the gradient.  A tile with anything beyond that is noticed in the conversion and left out of the sums; at the end of the period the
// tiles left out come again, under scales that hold the largest of their values (half a unit: 2^-30 of it), and
// their sums are added.  Which tiles these are depends on the values alone, so that results repeat bit for bit.
// Gradients with infinities or NaNs are left out of the digits, the products of their infinities found afterwards.
// What values of many sizes cost (all pairs of 16 x 11.2 M, 24 x 3 M, 32 x 11.2 M, 64 x 3 M, us, short runs; when a tile beyond its bound was
// noticed at the end only, the CTA did its whole share again):
//                                                          here            whole share           binary32 pipes
//     normal values                                  121  57 238 140     122   54  237  139     140  89 459 522
//     one element of 10^6                            122  58 239 142     470  145  686  496     141  89 459 522
//     lognormal, sigma 2                             121  60 238 145     480  151  743  524     141  89 459 522
//     97 % of all rows of 512 elements zero          128  69 246 158     492  160  742  521     140  89 459 522
//     200 tensors with lognormal scales, sigma 2     124  60 245 145     485  157  766  530     140  89 459 522
//     6 % of the vector 1000 times as large          117  64 260 155     494   55  240  529     140  89 459 522
//     one gradient of NaNs                           119  58 247 141    3417 1201 7912 2905     141  89 459 523
//     infinities in a gradient                       135  79 274 196    1309  546 2588 1522     141  89 459 523
// Work split.  One CTA per SM.  A tile is 128 consecutive elements of all K gradients (256 up to 16); tiles are dealt round-robin to the
// CTAs, and inside a CTA to teams of KP / 8 warps.  Every warp of a team has eight gradients for the whole kernel (their
// addresses and scales stay in registers); it reads 512 consecutive bytes of each, writes their digits into the team's tile
// buffer in shared memory (128-byte swizzle, K-major: the operand format; 192 KB in all), and the team hands the tile to the one
// thread that issues the MMAs, in whatever order the tiles come:
// 4 MMAs of 128 rows x 4 KP columns x 32 elements, and beyond 32 gradients 4 more for the products of d2 and d3
// among themselves (what is missing of the 4 KP x 4 KP products then is the mirror image of something present).
// Rows of absent gradients, and the rows of the 128 beyond 4 KP, hold whatever the memory holds: their sums are not read.
//
// Bound by HBM in short runs (of the copy rate: 16 gradients 0.91, 24 to 40 0.86 to 0.92, 64 0.88; up to 12, whose rows are padded to 16, 0.61 to 0.76; 24 x 3 M 0.77,
// with 8 us of launch, first tiles and last sums), by the power cap in long ones (24 x 3 M: tensor pipe 33 % busy, issue slots 52 %).  All
// pairs, D = 11.2 M, against the kernel on the binary32 pipes (bound by these and by shared memory), us:
//     gradients                    9    15    16    24    32    40    64
//     short runs                 102   118   121   183   238   320   501    (binary32 pipes 143  141  140  306  459  901  1905)
//     a second of calls on end   112   135   138   211   277   369   581    (142  143  145  306  459  901  1947; the SM clock falls to 1.1 to 1.5 GHz)
// What decided the shape: loads under a branch, or in a ring of single registers, wait for one another (32 gradients: 900 us; a warp with
// absent gradients loads under predicates and converts zeros for them, without a branch: 15 / 31 x 8.2 M 108 / 220 us with branches,
// 100 / 198 so, binary32 pipes 105 / 338); eight gradients for the whole kernel per warp, 20 warps and more (300 -> 265); the MMAs issued by a
// converged warp with an elected lane (their operands are scalars then; 16 gradients 147 -> 118 with two chunks a product); shared memory of
// less than 196 KB in all, beyond which the first-level cache that loads in flight need shrinks (64 x 4.1 M 230 -> 245).  Products of 64 rows,
// which waste less, cost the same time and no less power.  The mean written meanwhile under the pattern of a sample: 16 x 11.2 M 199 us, 179 with a
// pass of its own.
#pragma once

#include "gaf_device.cuh"
#include "gaf_fused.cuh"
#include "gaf_gram_tc.cuh"
#include "gaf_gramfilter.cuh"
#include "gaf_pairwise.cuh"

namespace gaf {

constexpr int kDgChunk = 128;                   // elements of a digit row in one swizzle block
constexpr int kDgHeadroom = 5;                  // bits between the largest sampled magnitude and the bound
constexpr unsigned int kDgPollLimit = 1u << 23; // looks at all barriers without a tile: a second
constexpr int kDgMaxChain = 1023;               // chunks: 1023 x 128 products of at most 2^14 fit a 32-bit sum

// How a warp goes through a tile: all of its eight gradients; some of them, loads under predicates and zeros for the others; or none beyond the fourth.
enum { kDgAll, kDgSome, kDgFour };
template <int FORM> using DigitsForm = std::integral_constant<int, FORM>;

template <int KP> struct DigitsShape {
    // Chunks of 128 elements of a tile.  Up to 16 gradients two of them lie one above the other in the 128 rows of a product, each
    // a diagonal block of it (the thread that issues cannot keep up with products of 64 columns: 16 x 11.2 M 147 us, 118).
    static constexpr int kChunks = KP <= 16 ? 2 : 1;
    static constexpr int kTeam = KP / 8;                        // warps of a team
    static constexpr int kTeams = KP == 64 ? 3 : 23 / kTeam;
    static constexpr int kTeamBuffers = 2 / kChunks;
    static constexpr int kWarps = kTeams * kTeam;
    static constexpr int kThreads = (kWarps + 1) * 32;
    static constexpr bool kTwo = KP > 32;                       // two products
    static constexpr int kColumns = kChunks * 4 * KP;           // of a product
    static constexpr int kRowsValid = kTwo ? 2 * KP : kColumns;
    static constexpr int kChunkBytes = 4 * KP * kDgChunk;
    static constexpr int kTileBytes = kChunks * kChunkBytes;
    static constexpr int kBuffers = kTeams * kTeamBuffers;
    // an operand of 128 rows read from the last tile may reach past it
    static constexpr int kRowsRead = kTwo ? 2 * KP + 128 : 128;
    static constexpr int kPad = kRowsRead > kColumns ? (kRowsRead - kColumns) * 128 : 0;
    static constexpr int kDyn = kBuffers * kTileBytes + kPad + 1024;
    static constexpr int kCols = kTwo ? 512 : 128;              // tensor memory
    static constexpr int kPeriodTiles = kDgMaxChain / kChunks / kTeams * kTeams;
    static_assert(kBuffers <= 32, "a lane of the issuing warp per buffer");
    static_assert(4 * KP * (KP + 1) * 8 <= kBuffers * kTileBytes, "the tile buffers hold the sums at the end");
};

struct GramDigitsArgs {
    const float *g[GAF_MAX_K];
    int K;
    int64_t D;
    int tiles;                  // T = ceil(K / 8)
    int pairs;                  // T (T + 1) / 2
    double *partials;           // [tile pair][slice][64]
    Control *ctl;
    unsigned int wait_limit;
    int test_extra_arrival;     // test hook, normally 0: warp 0's barrier expects an arrival that never comes
};

// One attempt at waiting for the phase with the given parity, for as long as the hardware suspends a thread by itself.
__device__ __forceinline__ bool dg_mbar_try(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(tc_smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool dg_mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag, unsigned int limit) {
    for (unsigned int spin = 0; spin < limit; ++spin) {
        if (dg_mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
// True in one lane of a whole warp, the same one every time.
__device__ __forceinline__ bool dg_elect() {
    uint32_t is;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(is)::"memory");
    return is != 0;
}
__device__ __forceinline__ bool dg_mbar_test(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(tc_smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// 8-bit signed x 8-bit signed -> 32-bit integer, both operands K-major, M = 128.
__device__ __forceinline__ void dg_mma(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__host__ __device__ constexpr uint32_t dg_idesc(int n) {
    return (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}
// 16 bytes if `wanted`, else r stays as it is: a load under a predicate.  (Under a branch the loads of a tile wait for one another.)
__device__ __forceinline__ void dg_ld16_if(uint4 &r, bool wanted, const void *p, uint64_t policy) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "@p ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;\n\t}"
        : "+r"(r.x), "+r"(r.y), "+r"(r.z), "+r"(r.w)
        : "l"(p), "l"(policy), "r"((unsigned int)wanted));
}
// 32 lanes x 4 columns of 32-bit accumulators.
__device__ __forceinline__ void dg_tmem_ld4(uint32_t taddr, int (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr)
                 : "memory");
}
template <int OFFSET> __device__ __forceinline__ void dg_st(uint32_t addr, unsigned int v) {
    asm volatile("st.shared.b32 [%0 + %2], %1;" ::"r"(addr), "r"(v), "n"(OFFSET) : "memory");
}
// The largest of m and the magnitudes of a pair; NaN if any is one.
__device__ __forceinline__ float dg_max_abs(float m, float a, float b) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ double dg_pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }   // |k| <= 1022

// 2^k under which a magnitude of 2^headroom times the given one is at most 2^30 (all zeros: the largest such power there is).
__device__ __forceinline__ int dg_exponent(unsigned int max_bits, int headroom) {
    const int e = (int)(max_bits >> 23) - 126;          // the magnitude is below 2^e
    return max_bits == 0u ? 126 : min(30 - e - headroom, 126);
}

// What the 32 lanes' pieces v of gradient r hold: the largest finite magnitude, a NaN, an infinity.  (Called where little else goes on; inlined at
// every call it is half of the kernel's code.)
__device__ __noinline__ void dg_note(uint4 v, int r, unsigned int *top, unsigned long long *nan_rows, unsigned long long *inf_rows) {
    const unsigned int m[4] = {v.x & 0x7FFFFFFFu, v.y & 0x7FFFFFFFu, v.z & 0x7FFFFFFFu, v.w & 0x7FFFFFFFu};
    unsigned int finite = 0u;
    bool nan = false, inf = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        finite = m[i] < 0x7F800000u ? max(finite, m[i]) : finite;
        nan |= m[i] > 0x7F800000u;
        inf |= m[i] == 0x7F800000u;
    }
    finite = __reduce_max_sync(0xFFFFFFFFu, finite);
    nan = __any_sync(0xFFFFFFFFu, nan);
    inf = __any_sync(0xFFFFFFFFu, inf);
    if ((threadIdx.x & 31) == 0) {
        if (nan) atomicOr(nan_rows, 1ull << r);
        if (inf) atomicOr(inf_rows, 1ull << r);
        atomicMax(&top[r], finite);
    }
}

template <int KP>
__global__ void __launch_bounds__(DigitsShape<KP>::kThreads, 1) gram_digits_kernel(const __grid_constant__ GramDigitsArgs a) {
    using S = DigitsShape<KP>;
    constexpr int W = S::kWarps, TEAMS = S::kTeams, TEAM = S::kTeam, NB = S::kBuffers, TB = S::kTeamBuffers, CH = S::kChunks;
    extern __shared__ unsigned char dg_smem[];
    __shared__ uint64_t full[NB], empty[NB], drained;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s, issued_s;
    __shared__ int expo[KP];                            // value = fixed point x 2^-expo
    __shared__ unsigned int rowmax[KP];                 // largest finite magnitude of the period's sample,
    __shared__ unsigned int rowtop[KP];                 // and of what was found beyond the bound
    __shared__ unsigned int beyond_map[32];             // the period's tiles with a value beyond its bound,
    __shared__ int beyond_buffer[NB];                   // and the buffers that hold one
    __shared__ unsigned long long nan_rows[2], inf_rows[2];     // gradients with a NaN, an infinity: [0] known before the period, [1] found in it
    // (the warp's number from a shuffle: known to be the same in all lanes, so that a row's address is a scalar and the lane's part 32 bits)
    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    unsigned char *tiles = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(dg_smem) + 1023) & ~uintptr_t(1023));
    const uint32_t tiles_u32 = tc_smem_u32(tiles);
    volatile int *const abort_flag = &abort_s;

    auto clear_period = [&]() {
        if (tid < KP) { rowmax[tid] = 0u; rowtop[tid] = 0u; }
        if (tid < 32) beyond_map[tid] = 0u;
    };
    clear_period();
    if (tid == 0) {
        for (int b = 0; b < NB; ++b) {
            tc_mbar_init(&full[b], TEAM + (b == 0 && a.test_extra_arrival ? 1 : 0));
            tc_mbar_init(&empty[b], 1);
            beyond_buffer[b] = 0;
        }
        tc_mbar_init(&drained, 1);
        abort_s = 0;
        nan_rows[0] = nan_rows[1] = inf_rows[0] = inf_rows[1] = 0ull;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(&tmem_base_s)),
                     "r"(S::kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_base_s;
    // a programmatic dependent of what precedes it on the stream: nothing global is touched before that has completed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (blockIdx.x == 0 && tid == 0) a.ctl->status = 0;          // first kernel of the operation

    const int K = a.K;
    const int64_t n_quads = a.D / 4, G = gridDim.x;
    const int64_t n_tiles = (n_quads + CH * 32 - 1) / (CH * 32);
    const int n_mine = blockIdx.x < n_tiles ? (int)((n_tiles - blockIdx.x + G - 1) / G) : 0;
    const uint64_t policy = l2_policy_evict_first();
    auto quad_of = [&](int n) { return ((int64_t)n * G + blockIdx.x) * (CH * 32); };      // first four elements of the CTA's tile n
    // this warp's eight gradients (absent ones: never read)
    const int team = warp / TEAM, row0 = (warp - team * TEAM) * 8;
    auto row = [&](int u) { return reinterpret_cast<const unsigned char *>(a.g[row0 + u]); };
    // The team takes its tiles of a period [n0, n1) (n0 a multiple of the teams) in ascending order, but for one that changes places
    // with its first: the first tiles of all teams, from which the scales are taken, are spread over the CTA's share, one in every
    // TEAMS-th part of it at an uneven place (equal distances fall in step with rows of 2^n elements), the same in all CTAs: places
    // of their own cost a page each (24 x 3 M: 1.5 us).
    const unsigned int place = ((unsigned int)team * 2654435761u + 1234567u) >> 20;
    auto tiles_of = [&](int n0, int n1) { return n1 - n0 > team ? (n1 - n0 - team + TEAMS - 1) / TEAMS : 0; };
    auto first_of = [&](int count) { return (int)((unsigned int)count * ((unsigned int)team * 4096u + place) / (TEAMS * 4096u)); };
    uint4 x[8] = {};
    // The warp's gradients that take part: those that are there and hold no NaN or infinity, as far as the CTA knows.  (All products of a
    // gradient that does are NaN or infinite, whatever the digits say.)
    unsigned int live = 0u;
    auto update_live = [&](unsigned long long odd) {
        const int here = min(max(K - row0, 0), 8);
        const unsigned int mask = warp < W ? ((1u << here) - 1u) & ~(unsigned int)(odd >> row0) : 0u;
        live = __shfl_sync(0xFFFFFFFFu, mask, 0);           // (known to be the same in all lanes, as `warp` is)
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (!((live >> u) & 1u)) x[u] = make_uint4(0u, 0u, 0u, 0u);         // (and stays so: loads are under predicates)
    };
    auto fetch = [&](auto form, int n, int chunk) {
        constexpr int ROWS = decltype(form)::value == kDgFour ? 4 : 8;
        const int64_t q = quad_of(n) + chunk * 32, left = n_quads - q;
        // lanes past the end of the vectors read the last four elements and count them as zeros
        const bool inside = lane < left;
        const int mine = inside ? lane * 16 : ((int)left - 1) * 16;
#pragma unroll
        for (int u = 0; u < ROWS; ++u) {
            if constexpr (decltype(form)::value == kDgAll) x[u] = ld16_policy(row(u) + q * 16 + mine, policy);
            else dg_ld16_if(x[u], (live >> u) & 1u, row(u) + q * 16 + mine, policy);
        }
        if (left < 32) {
#pragma unroll
            for (int u = 0; u < ROWS; ++u) x[u] = inside ? x[u] : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    // dg_note of all that x holds, for the sample: one operation a gradient where everything is finite.
    auto note_all = [&]() {
        unsigned int most[8], mine = 0u;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            most[u] = __reduce_max_sync(0xFFFFFFFFu, max(max(x[u].x & 0x7FFFFFFFu, x[u].y & 0x7FFFFFFFu), max(x[u].z & 0x7FFFFFFFu, x[u].w & 0x7FFFFFFFu)));
#pragma unroll
        for (int u = 0; u < 8; ++u) mine = lane == u ? most[u] : mine;
        const bool takes_part = lane < 8 && ((live >> lane) & 1u);
        if (__builtin_expect(!__any_sync(0xFFFFFFFFu, takes_part && mine >= 0x7F800000u), 1)) {
            if (takes_part) atomicMax(&rowmax[row0 + lane], mine);
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if ((live >> u) & 1u) dg_note(x[u], row0 + u, rowmax, &nan_rows[0], &inf_rows[0]);
        }
    };
    // The period's scales come from the first tiles of its teams, and for a gradient that has nothing but zeros there, from single pieces of
    // 16 bytes, 32 times as many places.
    auto sample = [&](int n0, int n1) {
        update_live(nan_rows[0] | inf_rows[0]);
        const int count = tiles_of(n0, n1);
        if (warp < W && count > 0) {
            const int n = n0 + team + first_of(count) * TEAMS;
            if (live == 0xFFu) fetch(DigitsForm<kDgAll>(), n, 0);
            else fetch(DigitsForm<kDgSome>(), n, 0);
            note_all();
        }
        __syncthreads();
        const unsigned long long odd = nan_rows[0] | inf_rows[0];
        auto zeros = [&](int r) { return r < K && rowmax[r] == 0u && !((odd >> r) & 1ull); };
        if (__builtin_expect(!__any_sync(0xFFFFFFFFu, zeros(lane) || zeros(lane + 32)), 1)) return;      // (the same for all warps)
        unsigned int dark = 0u;
        for (int u = 0; u < 8; ++u) dark |= warp < W && count > 0 && zeros(row0 + u) ? 1u << u : 0u;
        __syncthreads();
        if (dark) {
            const int at = (int)((unsigned int)count * ((unsigned int)lane * 4096u + place) / (32u * 4096u));
            const int64_t q = min(quad_of(n0 + team + at * TEAMS) + (int)((place + (unsigned int)lane * 11u) % (CH * 32u)), n_quads - 1);
            for (int u = 0; u < 8; ++u)
                if ((dark >> u) & 1u) dg_note(ld16_policy(row(u) + q * 16, policy), row0 + u, rowmax, &nan_rows[0], &inf_rows[0]);
        }
        __syncthreads();
    };
    auto is_beyond = [&](int t) { return (beyond_map[t >> 5] >> (t & 31)) & 1u; };

    uint32_t done_tiles = 0;                            // tiles this warp's team has handed over so far
    uint32_t phase = 0, n_drained = 0;                  // issuing warp: parity of the next tile in buffer `lane`; drains so far
    // This warp's digits of the team's tiles of [n0, n1), into the team's buffers in turn: of all of them under the sample's scales (the
    // first is in x already), or, EXACT, of those with a value beyond its bound under scales that hold every finite value in them.
    auto convert_tiles = [&](auto exact_tag, auto form, int n0, int n1) {
        constexpr bool EXACT = decltype(exact_tag)::value;
        constexpr int ROWS = decltype(form)::value == kDgFour ? 4 : 8;
        float scale[ROWS];
#pragma unroll
        for (int u = 0; u < ROWS; ++u) {
            const int sampled = dg_exponent(rowmax[row0 + u], kDgHeadroom);
            const int k = EXACT ? min(sampled, dg_exponent(rowtop[row0 + u], 0)) : sampled;
            scale[u] = __uint_as_float((unsigned int)(k + 127) << 23);
        }
        const int count = tiles_of(n0, n1);
        // v: how many tiles the team is through; EXACT: its tile, counted within the period
        const int first = first_of(count), end = EXACT ? n1 - n0 : count;
        auto tile_at = [&](int v) { return EXACT ? v : team + (v == 0 ? first : v == first ? 0 : v) * TEAMS; };
        auto next_beyond = [&](int t) {
            while (t < end && !is_beyond(t)) t += TEAMS;
            return t;
        };
        int v = EXACT ? next_beyond(team) : 0;
        if (EXACT && v < end) fetch(form, n0 + v, 0);
        for (int chunk = 0; v < end;) {
            const int buffer = team * TB + (int)(done_tiles % TB);
            // the MMAs on what this buffer held before are complete
            if (chunk == 0 && done_tiles >= TB && !__all_sync(0xFFFFFFFFu, dg_mbar_wait(&empty[buffer], (done_tiles / TB - 1) & 1u, abort_flag, kDgPollLimit))) break;
            const uint32_t block = tiles_u32 + (uint32_t)(buffer * S::kTileBytes + chunk * S::kChunkBytes + row0 * 128);
            float most = 0.0f;
#pragma unroll
            for (int u = 0; u < ROWS; ++u) {
                float f[4] = {__uint_as_float(x[u].x), __uint_as_float(x[u].y), __uint_as_float(x[u].z), __uint_as_float(x[u].w)};
#pragma unroll
                for (int i = 0; i < 4; ++i) f[i] *= scale[u];
                if constexpr (!EXACT) most = dg_max_abs(dg_max_abs(most, f[0], f[1]), f[2], f[3]);
                // signed digits: carries by an addition, then the lower three bytes without their bias
                unsigned int d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) d[i] = (unsigned int)__float2int_rn(f[i]) + 0x00808080u;
                // 4 x 4 bytes turned: word s = digit s of the four elements
                const unsigned int t0 = __byte_perm(d[0], d[1], 0x5140), t1 = __byte_perm(d[0], d[1], 0x7362);
                const unsigned int t2 = __byte_perm(d[2], d[3], 0x5140), t3 = __byte_perm(d[2], d[3], 0x7362);
                const uint32_t dst = block + (uint32_t)(u * 128) + (uint32_t)((lane * 4) ^ (u << 4));
                dg_st<0>(dst, __byte_perm(t1, t3, 0x7632));
                dg_st<KP * 128>(dst, __byte_perm(t1, t3, 0x5410) ^ 0x80808080u);
                dg_st<2 * KP * 128>(dst, __byte_perm(t0, t2, 0x7632) ^ 0x80808080u);
                dg_st<3 * KP * 128>(dst, __byte_perm(t0, t2, 0x5410) ^ 0x80808080u);
            }
            if constexpr (!EXACT) {
                if (__builtin_expect(__any_sync(0xFFFFFFFFu, !(most <= 1073741824.0f)), 0)) {
                    // beyond the bound (or not finite): the tile is left out, and comes again under other scales
#pragma unroll
                    for (int u = 0; u < ROWS; ++u)
                        if ((live >> u) & 1u) dg_note(x[u], row0 + u, rowtop, &nan_rows[1], &inf_rows[1]);
                    if (lane == 0) {
                        const int t = tile_at(v);
                        atomicOr(&beyond_map[t >> 5], 1u << (t & 31));
                        *(volatile int *)&beyond_buffer[buffer] = 1;
                    }
                    __syncwarp();
                }
            }
            if (++chunk == CH) {
                tc_fence_async_smem();
                __syncwarp();
                if (lane == 0) tc_mbar_arrive(&full[buffer]);
                ++done_tiles;
                chunk = 0;
                v = EXACT ? next_beyond(v + TEAMS) : v + 1;
            }
            if (v < end) fetch(form, n0 + tile_at(v), chunk);
        }
    };
    // MMAs of `total` tiles in the order they come, by lane 0 of the issuing warp; back when all are complete (or a wait gave
    // up).  Tiles with a value beyond its bound are passed over.  Lane b looks at buffer b's barrier.  (In a fixed order the teams wait for one another: 32 x 2 M 69 us for 59.)
    auto issue_tiles = [&](int total) {
        uint32_t accumulate = 0;
        while (total > 0) {
            unsigned int ready = 0;
            bool beyond = false;
            for (unsigned int idle = 0; idle <= a.wait_limit; ++idle) {
                const bool here = dg_mbar_test(&full[lane < NB ? lane : 0], phase) && lane < NB;
                beyond = *(volatile int *)&beyond_buffer[lane < NB ? lane : 0] != 0 && here;
                ready = __ballot_sync(0xFFFFFFFFu, here);
                if (ready || __any_sync(0xFFFFFFFFu, *abort_flag)) break;
                __nanosleep(32);                        // (without it the polls take issue slots from the conversion: 3 us on short calls)
            }
            if (!ready) {
                *abort_flag = 1;
                break;
            }
            phase ^= (ready >> lane) & 1u;
            total -= __popc(ready);
            if (beyond) {
                // (no MMA reads this buffer: it is free at once)
                *(volatile int *)&beyond_buffer[lane] = 0;
                tc_mbar_arrive(&empty[lane]);
            }
            ready &= ~__ballot_sync(0xFFFFFFFFu, beyond);
            __syncwarp();
            tc_fence_after_sync();
            for (; ready; ready &= ready - 1u) {
                // (everything but the instructions themselves by the whole warp: scalars, which they want their operands to be)
                const int b = __ffs(ready) - 1;
                const uint32_t tile = tiles_u32 + (uint32_t)(b * S::kTileBytes);
                const uint64_t d0 = tc_smem_desc(tile), d2 = tc_smem_desc(tile + 2 * KP * 128);
                if (dg_elect()) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        // 32 elements = 32 bytes further along K inside the swizzle atom
                        dg_mma(tmem, d0 + (uint64_t)(2 * k), d0 + (uint64_t)(2 * k), dg_idesc(S::kColumns), k == 0 ? accumulate : 1u);
                        if (S::kTwo) dg_mma(tmem + 4 * KP, d2 + (uint64_t)(2 * k), d2 + (uint64_t)(2 * k), dg_idesc(2 * KP), k == 0 ? accumulate : 1u);
                    }
                    tc_commit(&empty[b]);
                }
                accumulate = 1;
                __syncwarp();
            }
        }
        if (dg_elect()) tc_commit(&drained);            // (the lane that issued the MMAs)
        __syncwarp();
        if (lane == 0) {
            issued_s = (int)accumulate;
            // (this last commit arrives when everything issued so far has completed: also before tensor memory is freed after a
            // wait that gave up)
            bool complete = false;
            for (unsigned int spin = 0; spin < kTcSpinLimit && !complete; ++spin) complete = tc_mbar_try(&drained, n_drained & 1u, 2000u);
            if (!complete) *abort_flag = 1;
        }
        ++n_drained;
    };

    // The sums of what was issued out of tensor memory, put together and added to what came before.
    auto collect = [&](bool first) {
        const bool any = issued_s != 0;
        constexpr int P = KP + 1;                       // (a pitch of 2 banks between rows)
        double *red = reinterpret_cast<double *>(tiles);
        if (any && warp < W) {
            const int row = (warp & 3) * 32 + lane, s = row / KP % 4;
            const bool valid = row < S::kRowsValid;
            const double weight = dg_pow2(24 - 8 * s), weight2 = dg_pow2(8 - 8 * s);
            // (of the rows' own chunk: a warp's rows are of one)
            const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(CH > 1 ? (warp & 3) * 32 / (4 * KP) * (4 * KP) : 0);
            for (int jb = warp >> 2; jb < KP / 4; jb += (W - (warp & 3) + 3) / 4) {
                int d[4][4], d2[2][4];
#pragma unroll
                for (int t = 0; t < 4; ++t) dg_tmem_ld4(lanes + (uint32_t)(t * KP + jb * 4), d[t]);
                if (S::kTwo) {
#pragma unroll
                    for (int t = 0; t < 2; ++t) dg_tmem_ld4(lanes + (uint32_t)((4 + t) * KP + jb * 4), d2[t]);
                }
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (valid) {
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) {
                        const long long hi = (long long)d[0][jj] * 16777216ll + (long long)d[1][jj] * 65536ll;
                        const long long lo = (long long)d[2][jj] * 256ll + (long long)d[3][jj];
                        double *const at = red + (size_t)row * P + jb * 4 + jj;
                        if constexpr (S::kTwo) {
                            // rows of d0, d1 against all columns (the upper two digits' columns, the lower two's), and rows of
                            // d2, d3 against columns of d2, d3
                            const long long lo2 = (long long)d2[0][jj] * 256ll + (long long)d2[1][jj];
                            at[0] = (double)hi * weight + (double)lo2 * weight2;
                            at[(size_t)2 * KP * P] = (double)lo * weight;
                        } else {
                            at[0] = (double)(hi + lo) * weight;
                        }
                    }
                }
            }
        }
        tc_fence_before_sync();
        __syncthreads();
        tc_fence_after_sync();
        for (int e = tid; e < a.pairs * 64; e += S::kThreads) {
            int ti, tj;
            tile_pair(e >> 6, a.tiles, ti, tj);
            const int i = ti * 8 + ((e >> 3) & 7), j = tj * 8 + (e & 7);
            if (i > j || j >= K) continue;
            double v = 0.0;
            if (any) {
                if constexpr (S::kTwo) {
                    const double *const low = red + (size_t)2 * KP * P;
#pragma unroll
                    for (int s = 0; s < 2; ++s)
                        v += red[(s * KP + i) * P + j] + (low[(s * KP + i) * P + j] + low[(s * KP + j) * P + i]);
                } else {
#pragma unroll
                    for (int s = 0; s < 4 * CH; ++s) v += red[(s * KP + i) * P + j];
                }
                v *= dg_pow2(-(expo[i] + expo[j]));
            }
            double *const dst = a.partials + ((size_t)(e >> 6) * gridDim.x + blockIdx.x) * 64 + (e & 63);
            if (first) {
                // fewer than 4 leftover elements: plain binary64 products
                if (blockIdx.x == 0)
                    for (int64_t el = n_quads * 4; el < a.D; ++el) v += (double)a.g[i][el] * (double)a.g[j][el];
                *dst = v;
            } else {
                *dst += v;
            }
        }
        __syncthreads();
    };

    // Gradients with NaNs and infinities: NaN for all products of the former; the products of infinities with the other gradients, infinite or
    // NaN whatever the order, from the period's tiles beyond their bounds or, of a gradient that was left out from the start, from all.
    // Once all products of a gradient are known to be NaN, or infinite of both signs, it is not looked at any more.
    auto nonfinite_products = [&](int n0, int n1) {
        unsigned long long *const pos_of = reinterpret_cast<unsigned long long *>(tiles), *const neg_of = pos_of + KP, *const nan_of = neg_of + KP;
        for (int r = tid; r < 3 * KP; r += S::kThreads) pos_of[r] = 0ull;       // (bit j of word i; the tile buffers are free here)
        __syncthreads();
        const unsigned long long nans = nan_rows[0] | nan_rows[1], infs = inf_rows[0] | inf_rows[1], all = K == 64 ? ~0ull : (1ull << K) - 1ull;
        for (int t = warp; warp < W && infs && t < (n1 - n0) * CH; t += W) {
            const int64_t q = quad_of(n0 + t / CH) + (t % CH) * 32 + lane;
            const bool inside = q < n_quads;
            unsigned long long rows = (inf_rows[0] | (is_beyond(t / CH) ? inf_rows[1] : 0ull)) & ~nans;
            for (; rows; rows &= rows - 1ull) {
                const int r = __ffsll((long long)rows) - 1;
                const unsigned long long known = *(volatile unsigned long long *)&nan_of[r] |
                    (*(volatile unsigned long long *)&pos_of[r] & *(volatile unsigned long long *)&neg_of[r]) | (1ull << r) | nans;
                if (!__any_sync(0xFFFFFFFFu, (~known & all) != 0ull)) continue;
                const float4 f = inside ? reinterpret_cast<const float4 *>(a.g[r])[q] : make_float4(0.f, 0.f, 0.f, 0.f);
                const float xs[4] = {f.x, f.y, f.z, f.w};
                if (!__any_sync(0xFFFFFFFFu, isinf(xs[0]) || isinf(xs[1]) || isinf(xs[2]) || isinf(xs[3]))) continue;
                for (int j0 = 0; j0 < K; j0 += 4) {
                    float4 g[4];                    // (loads in flight together)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        g[k] = inside && j0 + k < K ? reinterpret_cast<const float4 *>(a.g[j0 + k])[q] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float ys[4] = {g[k].x, g[k].y, g[k].z, g[k].w};
                        bool pos = false, neg = false, nan = false;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float p = isinf(xs[i]) ? xs[i] * ys[i] : 0.0f;
                            pos |= p > 0.0f; neg |= p < 0.0f; nan |= isnan(p);
                        }
                        pos = __any_sync(0xFFFFFFFFu, pos); neg = __any_sync(0xFFFFFFFFu, neg); nan = __any_sync(0xFFFFFFFFu, nan);
                        const unsigned long long bit = lane == 0 && j0 + k < K ? 1ull << (j0 + k) : 0ull;
                        if (pos && bit) atomicOr(&pos_of[r], bit);
                        if (neg && bit) atomicOr(&neg_of[r], bit);
                        if (nan && bit) atomicOr(&nan_of[r], bit);
                    }
                }
            }
        }
        __syncthreads();
        for (int e = tid; e < a.pairs * 64; e += S::kThreads) {      // (the slots that this thread wrote)
            int ti, tj;
            tile_pair(e >> 6, a.tiles, ti, tj);
            const int i = ti * 8 + ((e >> 3) & 7), j = tj * 8 + (e & 7);
            if (i > j || j >= K) continue;
            double *const dst = a.partials + ((size_t)(e >> 6) * gridDim.x + blockIdx.x) * 64 + (e & 63);
            const double inf = __longlong_as_double(0x7FF0000000000000ll);
            auto bit = [&](const unsigned long long *w) { return (((w[i] >> j) | (w[j] >> i)) & 1ull) != 0ull; };
            const bool pos = i == j ? (infs >> i) & 1ull : bit(pos_of), neg = i != j && bit(neg_of);
            if (((nans >> i) | (nans >> j)) & 1ull || (i != j && bit(nan_of))) *dst = __longlong_as_double(0x7FF8000000000000ll);
            else *dst += (pos ? inf : 0.0) - (neg ? inf : 0.0);
        }
        __syncthreads();
    };
    // (every thread takes the same turns: the conditions are read behind a barrier)
    auto convert_and_issue = [&](auto exact_tag, int n0, int n1, int total) {
        if (warp < W) {
            if (decltype(exact_tag)::value) convert_tiles(exact_tag, DigitsForm<kDgSome>(), n0, n1);
            else if (live == 0xFFu) convert_tiles(std::false_type(), DigitsForm<kDgAll>(), n0, n1);
            else if (live < 16u) convert_tiles(std::false_type(), DigitsForm<kDgFour>(), n0, n1);
            else convert_tiles(std::false_type(), DigitsForm<kDgSome>(), n0, n1);
        } else {
            issue_tiles(total);
        }
        __syncwarp();
        tc_fence_before_sync();
        __syncthreads();
        tc_fence_after_sync();
    };
    for (int n0 = 0; n0 == 0 || n0 < n_mine; n0 += S::kPeriodTiles) {
        const int n1 = min(n_mine, n0 + S::kPeriodTiles);
        if (n0 > 0) {
            clear_period();
            if (tid == 0) { nan_rows[0] |= nan_rows[1]; inf_rows[0] |= inf_rows[1]; }
            __syncthreads();
        }
        sample(n0, n1);
        update_live(nan_rows[0] | inf_rows[0]);
        if (tid < KP) expo[tid] = dg_exponent(rowmax[tid], kDgHeadroom);        // (read behind the next barrier)
        convert_and_issue(std::false_type(), n0, n1, n1 - n0);
        if (abort_s) break;
        const int beyond = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned int)__popc(beyond_map[lane]));
        collect(n0 == 0);
        if (__builtin_expect(beyond != 0, 0)) {
            update_live(nan_rows[0] | nan_rows[1] | inf_rows[0] | inf_rows[1]);
            if (tid < KP) expo[tid] = min(expo[tid], dg_exponent(rowtop[tid], 0));
            convert_and_issue(std::true_type(), n0, n1, beyond);
            if (abort_s) break;
            collect(false);
        }
        if (__builtin_expect((nan_rows[0] | nan_rows[1] | inf_rows[0] | inf_rows[1]) != 0ull, 0)) nonfinite_products(n0, n1);
    }
    // the streaming part of this CTA is over: the finishing kernel may be placed (it waits for this grid)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();
    if (warp == W) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::kCols) : "memory");
    }
    if (abort_s) {
        if (tid == 0) atomicOr(&a.ctl->status, kStatusTimeoutBit);
        return;
    }
}

}  // namespace gaf
