// Global beam selection (Section 2.1: every active beam is expanded over the codebook and the global top-k
// candidates are kept): from the previous beams' cumulative scores and this step's candidate log-probabilities,
// the W_new best (parent, code) pairs per request, best first, parents in the form onela_reorder_beams takes - so
// selection, reorder and the layers' decode launches of a step can run back to back on the device (one CUDA graph).
//
// A candidate's rank is a 64-bit composite: its fp32 score (parent score + log-probability, mapped to
// order-preserving bits; NaN lowest, -0 = +0) in the high word, 0xffffffff - flat index in the low word, so
// composites are distinct and "larger" means "better, ties to the smaller flat index".
//
// The candidates are cut into shares, the shares' largest give a bound that at least k of them reach - so at least k candidates
// reach it, and hardly more do (1094 expected for k = 1024 of a million) - and only the shares that reach it are looked into:
//   * up to 16 384 candidates (32 768 where more than 256 survive), fewer than 48 per survivor, or without scratch, a share is a
//     thread's, in a cluster of up to eight CTAs of 1024 threads per request (`select_kernel`): the first CTA finds the bound, what
//     reaches it is gathered in its shared memory (distributed shared memory, one remote atomic per CTA), ordered through a histogram
//     of the scores and written out best first;
//   * beyond, shares of sixteen are spread over all SMs by a launch of their own (`spread_shares_kernel`), and the cluster goes on
//     from their largest (`select_kernel<true>`).  A cluster alone waited 7.7 us for 512 x 256 candidates out of HBM;
//   * where few survive (k <= 256), one CTA does the rest without a cluster's barriers, from shares of neighbours, whose members
//     one CTA can fetch in full lines (`select_shares_kernel`, `select_of_shares_kernel`).
// What bounds it: latency - the shares (2 us), then for a cluster four barriers (4 us of 12) and a dozen of a CTA's; the code runs
// once per launch, so loops stay rolled.  (As two launches - every 4096 candidates by an eight-pass radix select of their own, one
// CTA to merge the parts' lists - the 512 x 256 -> 512 selection took 36 - 43 us, one cluster 14 warm and 18 out of HBM.)
#include <mutex>

#include "onela_internal.h"

namespace onela {

namespace {

constexpr int SEL_THREADS = 1024;
constexpr int SEL_CAP = ONELA_SELECT_CAP;      // survivors per request (W_new <= SEL_CAP)
constexpr int SEL_LIST = 4096;                 // candidates that reach the bound: room in shared memory
constexpr int SEL_CTAS = 8;                    // CTAs per cluster at most
constexpr int SEL_HELD = 16;                   // scores a thread keeps in registers
constexpr int SEL_SHARE = 16;                  // consecutive candidates of a share
constexpr int SEL_SHARES = ONELA_SELECT_PARTS * 4096 / SEL_SHARE;     // shares of the largest request; the list behind them in the
                                               // scratch takes all candidates of the k + k / 8 threads the bound may leave
constexpr int SEL_BINS = 2048;
constexpr int SEL_ROTATE = 977;                // a thread's place moves by this much from stripe to stripe, so that one code's
                                               // candidates (a multiple of C apart) do not all fall to the same threads

__device__ __forceinline__ uint32_t score_bits(float s) {
    if (s != s) return 0u;                              // NaN: below every number
    const uint32_t u = __float_as_uint(s + 0.0f);       // -0.0 + 0.0 = +0.0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

struct ScoreSource {     // composites computed from the caller's scores; item i is flat index i
    const float* bs;
    const float* lp;
    uint32_t magic;      // i / C as (i magic / 2^32) >> shift, exactly (see divide_by)
    int shift, C;
    __device__ __forceinline__ uint32_t parent(uint32_t i) const { return magic ? __umulhi(i, magic) >> shift : i; }
    __device__ __forceinline__ float score(uint32_t i) const { return __ldg(bs + parent(i)) + __ldg(lp + i); }
    __device__ __forceinline__ unsigned long long join(uint32_t bits, uint32_t i) const {
        return ((unsigned long long)bits << 32) | (unsigned long long)(0xffffffffu - i);
    }
    __device__ __forceinline__ unsigned long long operator()(uint32_t i) const { return join(score_bits(score(i)), i); }
};
// i / C for i < 2^20: with m = ceil(2^t / C), i m / 2^t has the right integer part while i C < 2^t - t = 32 serves C <= 4096,
// t = 40 (m below 2^32 then) the larger ones; C = 1 is no division.
void divide_by(int32_t C, uint32_t& magic, int& shift) {
    shift = C > 4096 ? 8 : 0;
    magic = C == 1 ? 0u : (uint32_t)(((1ull << (32 + shift)) + (unsigned long long)C - 1ull) / (unsigned long long)C);
}
struct SelectShared {
    unsigned int hist[SEL_BINS];
    unsigned long long sel[SEL_CAP];           // (the exhaustive selection's result)
    unsigned long long prefix, lo, hi;
    unsigned long long part_min[32], part_max[32];
    unsigned int k, count, equal, part_sum[32];
};

// Leaves the k largest composites of item(0 .. n-1) in sh.sel[0 .. k) (unordered); k <= min(n, SEL_CAP).
// `item(j, i)` returns composite i = tid + j * SEL_THREADS: from the source itself, or from the thread's registers.
// MAXJ > 0: at most MAXJ items per thread, loops unrolled (so that a register array can be indexed); 0: any number.
template <int MAXJ, class Item>
__device__ void select_passes(const Item& item, uint32_t n, int k, SelectShared& sh) {
    const int tid = threadIdx.x;
    if (tid == 0) { sh.prefix = 0ull; sh.k = (unsigned)k; sh.count = 0u; }
    if (tid < 256) sh.hist[tid] = 0u;
    __syncthreads();
    // after the pass over byte p, sh.prefix holds bytes 7..p of the k-th largest composite and sh.k how many
    // survivors are still to be found among the candidates that share those bytes
    const uint32_t n_padded = (n + SEL_THREADS - 1) / SEL_THREADS * SEL_THREADS;
    for (int p = 7; p >= 0; --p) {             // two block-wide barriers per pass
        const unsigned long long prefix = sh.prefix;
        const unsigned want = sh.k;               // (read here: the bin search below rewrites it)
        const unsigned long long hi_mask = p == 7 ? 0ull : (~0ull << (8 * (p + 1)));
        auto count_item = [&](int j, uint32_t i) {
            // whole warps stay in the loop (padding iterations carry no candidate) so the peer vote is complete
            const bool live = i < n;
            const unsigned long long c = live ? item(j, i) : 0ull;
            const bool in = live && ((c & hi_mask) == prefix);
            const unsigned bin = (unsigned)(c >> (8 * p)) & 255u;
            // one atomic per distinct bin in the warp: scores cluster, so most lanes share a bin in the early passes
            const unsigned vote = __ballot_sync(0xffffffffu, in);
            if (in) {
                const unsigned peers = __match_any_sync(vote, bin);
                if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&sh.hist[bin], __popc(peers));
            }
        };
        if constexpr (MAXJ > 0) {
#pragma unroll
            for (int j = 0; j < MAXJ; ++j) {
                const uint32_t i = tid + (uint32_t)j * SEL_THREADS;
                if (i < n_padded) count_item(j, i);
            }
        } else {
            for (uint32_t i = tid; i < n_padded; i += SEL_THREADS) count_item(0, i);
        }
        __syncthreads();
        // the bin that holds the k-th largest, by the first warp alone: lane l takes bins 8 l .. 8 l + 7, suffix counts
        // (candidates in bins >= b) across the lanes by shuffles; it also clears the histogram for the next pass
        if (tid < 32) {
            unsigned h[8], mine = 0;
#pragma unroll
            for (int t = 0; t < 8; ++t) { h[t] = sh.hist[8 * tid + t]; mine += h[t]; }
#pragma unroll
            for (int t = 0; t < 8; ++t) sh.hist[8 * tid + t] = 0u;
            unsigned incl = mine;                                   // counts of lanes >= this one
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned up = __shfl_down_sync(0xffffffffu, incl, off);
                if (tid + off < 32) incl += up;
            }
            unsigned here = incl;                                   // candidates in bins >= 8 tid + t, from t = 0 down
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const unsigned next = here - h[t];                  // ... in bins > 8 tid + t
                if (here >= want && next < want) {                  // exactly one bin qualifies
                    sh.prefix = prefix | ((unsigned long long)(8 * tid + t) << (8 * p));
                    sh.k = want - next;
                    sh.equal = h[t];
                }
                here = next;
            }
        }
        __syncthreads();
        // the score word is fixed and exactly the candidates that share it are still wanted: no tie straddles the cut
        if (p == 4 && sh.equal == sh.k) break;
    }
    const unsigned long long threshold = sh.prefix;   // (low bytes zero after an early exit: every equal score is kept)
    auto keep_item = [&](int j, uint32_t i) {
        const unsigned long long c = item(j, i);
        if (c >= threshold) {
            const unsigned pos = atomicAdd(&sh.count, 1u);
            if (pos < SEL_CAP) sh.sel[pos] = c;
        }
    };
    if constexpr (MAXJ > 0) {
#pragma unroll
        for (int j = 0; j < MAXJ; ++j) {
            const uint32_t i = tid + (uint32_t)j * SEL_THREADS;
            if (i < n) keep_item(j, i);
        }
    } else {
        for (uint32_t i = tid; i < n; i += SEL_THREADS) keep_item(0, i);
    }
    __syncthreads();
}
// The exhaustive selection.  The passes read every candidate four to eight times: up to ITEMS * SEL_THREADS candidates are
// fetched once, all loads in flight together, and kept in registers; longer lists are re-read from the source.
template <int ITEMS, class Src>
__device__ void select_topk(const Src& src, uint32_t n, int k, SelectShared& sh) {
    if (n <= (uint32_t)ITEMS * SEL_THREADS) {
        unsigned long long held[ITEMS];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t i = threadIdx.x + (uint32_t)j * SEL_THREADS;
            held[j] = i < n ? src(i) : 0ull;
        }
        auto item = [&](int j, uint32_t) { return held[j]; };      // j is a compile-time constant in the unrolled loops
        select_passes<ITEMS>(item, n, k, sh);
    } else {
        auto item = [&](int, uint32_t i) { return src(i); };
        select_passes<0>(item, n, k, sh);
    }
}

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t in_first_cta(const void* p) {      // shared address in the cluster's first CTA
    uint32_t at;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(p)));
    return at;
}
__device__ __forceinline__ void st_cluster64(uint32_t at, unsigned long long x) { asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(at), "l"(x) : "memory"); }
__device__ __forceinline__ unsigned long long ld_cluster64(uint32_t at) {
    unsigned long long x;
    asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(x) : "r"(at) : "memory");
    return x;
}
__device__ __forceinline__ unsigned add_cluster(uint32_t at, unsigned x) {
    unsigned old;
    asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(at), "r"(x) : "memory");
    return old;
}

// The histogram step of bound_of: bins of the CTA's items counted in sh.hist, the bin that holds the want-th largest is
// found; sh.equal = that bin, sh.count = items in it and above, sh.k = items above.  Ends with a barrier.
__device__ __forceinline__ void bin_of_kth(unsigned want, SelectShared& sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __syncthreads();
    // counts of the bins from the top: thread t takes bins 2 t and 2 t + 1
    const uint2 h = reinterpret_cast<const uint2*>(sh.hist)[tid];
    unsigned incl = h.x + h.y;                                        // lanes >= this one
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned up = __shfl_down_sync(0xffffffffu, incl, o);
        if (lane + o < 32) incl += up;
    }
    if (lane == 0) sh.part_sum[warp] = incl;
    __syncthreads();
    const unsigned above = __reduce_add_sync(0xffffffffu, lane > warp ? sh.part_sum[lane] : 0u);      // warps above this one
    const unsigned ge0 = above + incl, ge1 = ge0 - h.x, gt1 = ge1 - h.y;
    if (ge1 >= want && gt1 < want) {
        sh.equal = 2 * tid + 1;
        sh.count = ge1;
        sh.k = gt1;
    } else if (ge0 >= want && ge1 < want) {
        sh.equal = 2 * tid;
        sh.count = ge0;
        sh.k = ge1;
    }
    __syncthreads();
}

// A bound that at least k, and as a rule little more, of the CTA's composites reach (COUNT per thread, 0 where there is
// none; all threads call).  A histogram over the span of the scores at hand; where the bin that holds the k-th largest holds
// too many more, further rounds look into that bin alone, on whole composites, down to single ones if they must.
template <int COUNT>
__device__ unsigned long long bound_of(const unsigned long long (&held)[COUNT], int k, SelectShared& sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned want = (unsigned)k;
    const unsigned slack = max(32u, want / 8);
    unsigned long long lo, hi;
    {
        uint32_t mn = 0xffffffffu, mx = 0u;
#pragma unroll
        for (int j = 0; j < COUNT; ++j)
            if (held[j]) {
                mn = min(mn, (uint32_t)(held[j] >> 32));
                mx = max(mx, (uint32_t)(held[j] >> 32));
            }
        mn = __reduce_min_sync(0xffffffffu, mn);
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) { sh.part_min[warp] = mn; sh.part_max[warp] = mx; }
        reinterpret_cast<uint2*>(sh.hist)[tid] = make_uint2(0u, 0u);
        __syncthreads();
        mn = __reduce_min_sync(0xffffffffu, (uint32_t)sh.part_min[lane]);
        mx = __reduce_max_sync(0xffffffffu, (uint32_t)sh.part_max[lane]);
        const int shift = max(0, 32 - __clz(mx - mn) - 11);
#pragma unroll
        for (int j = 0; j < COUNT; ++j)
            if (held[j]) atomicAdd(&sh.hist[((uint32_t)(held[j] >> 32) - mn) >> shift], 1u);
        bin_of_kth(want, sh);
        const uint32_t first = mn + (sh.equal << shift);
        lo = (unsigned long long)first << 32;
        hi = ((unsigned long long)(first + ((1u << shift) - 1u)) << 32) | 0xffffffffull;
    }
    while (sh.count - want > slack) {
        want -= sh.k;
        unsigned long long mn = ~0ull, mx = 0ull;
#pragma unroll
        for (int j = 0; j < COUNT; ++j)
            if (held[j] >= lo && held[j] <= hi) {
                mn = min(mn, held[j]);
                mx = max(mx, held[j]);
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        if (lane == 0) { sh.part_min[warp] = mn; sh.part_max[warp] = mx; }
        reinterpret_cast<uint2*>(sh.hist)[tid] = make_uint2(0u, 0u);
        __syncthreads();
        mn = sh.part_min[lane];
        mx = sh.part_max[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        const int shift = max(0, 64 - __clzll((long long)(mx - mn)) - 11);
#pragma unroll
        for (int j = 0; j < COUNT; ++j)
            if (held[j] >= lo && held[j] <= hi) atomicAdd(&sh.hist[(unsigned)((held[j] - mn) >> shift)], 1u);
        bin_of_kth(want, sh);
        lo = mn + ((unsigned long long)sh.equal << shift);
        hi = lo + (1ull << shift) - 1ull;
        if (shift == 0) break;
    }
    return lo;
}

// Writes survivor x, which is the `rank`-th best, out.
__device__ __forceinline__ void emit(unsigned long long x, int rank, const ScoreSource& src, int32_t* parents, int32_t* codes, float* scores) {
    const uint32_t idx = 0xffffffffu - (uint32_t)(x & 0xffffffffull), par = src.parent(idx);
    parents[rank] = (int)par;
    codes[rank] = (int)(idx - par * (uint32_t)src.C);
    // the score is in the composite, but for NaNs' payloads and the sign of zero (0 and 0x80000000 there)
    const uint32_t u = (uint32_t)(x >> 32);
    scores[rank] = (u & 0x7fffffffu) == 0u ? __ldg(src.bs + par) + __ldg(src.lp + idx) : __uint_as_float((u & 0x80000000u) ? u ^ 0x80000000u : ~u);
}

// Orders list[0 .. n) best first (n <= 1024 E; `spare`: as much room again) and writes the k best out.  The scores at hand are
// spread over SEL_BINS bins: an element's rank is the count of the bins before its own plus the number of larger ones in it,
// as a rule one or two.  Where a bin holds many (equal scores): runs of 32 are sorted by their warp (shuffles), then merged
// pairwise, an element's place being its own in its run plus the number of elements of the other run that come before it,
// found by bisection.  (600 survivors: 2.5 us with bins; 6.7 us merged, whose scattered 64-bit reads conflict; 9.2 us as a
// bitonic sort.)
template <int E>
__device__ void sort_and_emit(unsigned long long* list, unsigned long long* spare, int n, int k, SelectShared& sh, const ScoreSource& src,
                              int32_t* parents, int32_t* codes, float* scores) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long x[E];
    {
        uint32_t mn = 0xffffffffu, mx = 0u;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const bool live = e * SEL_THREADS + tid < n;
            x[e] = live ? list[e * SEL_THREADS + tid] : 0ull;
            if (live) {
                mn = min(mn, (uint32_t)(x[e] >> 32));
                mx = max(mx, (uint32_t)(x[e] >> 32));
            }
        }
        mn = __reduce_min_sync(0xffffffffu, mn);
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) { sh.part_min[warp] = mn; sh.part_max[warp] = mx; }
        reinterpret_cast<uint2*>(sh.hist)[tid] = make_uint2(0u, 0u);
        __syncthreads();
        mn = __reduce_min_sync(0xffffffffu, (uint32_t)sh.part_min[lane]);
        mx = __reduce_max_sync(0xffffffffu, (uint32_t)sh.part_max[lane]);
        const int shift = max(0, 32 - __clz(mx - mn) - 11);
        unsigned at[E];
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (e * SEL_THREADS + tid < n) at[e] = atomicAdd(&sh.hist[(mx - (uint32_t)(x[e] >> 32)) >> shift], 1u);
        __syncthreads();
        const uint2 h = reinterpret_cast<const uint2*>(sh.hist)[tid];
        unsigned incl = h.x + h.y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        const unsigned most = __reduce_max_sync(0xffffffffu, max(h.x, h.y));
        if (lane == 31) { sh.part_sum[warp] = incl; sh.part_min[warp] = most; }
        __syncthreads();
        const unsigned before = incl - h.x - h.y + __reduce_add_sync(0xffffffffu, lane < warp ? sh.part_sum[lane] : 0u);
        const bool few = __reduce_max_sync(0xffffffffu, (uint32_t)sh.part_min[lane]) <= 32u;
        reinterpret_cast<uint2*>(sh.hist)[tid] = make_uint2(before, before + h.x);       // where the bins start
        __syncthreads();
        if (few) {
            unsigned bin[E];
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (e * SEL_THREADS + tid < n) {
                    bin[e] = (mx - (uint32_t)(x[e] >> 32)) >> shift;
                    spare[sh.hist[bin[e]] + at[e]] = x[e];
                }
            __syncthreads();
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (e * SEL_THREADS + tid < n) {
                    const unsigned first = sh.hist[bin[e]], end = bin[e] + 1 < SEL_BINS ? sh.hist[bin[e] + 1] : (unsigned)n;
                    unsigned rank = first;
                    if (first < (unsigned)k) {
                        for (unsigned q = first; q < end; ++q) rank += spare[q] > x[e];
                        if (rank < (unsigned)k) emit(x[e], (int)rank, src, parents, codes, scores);
                    }
                }
            return;
        }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (e * SEL_THREADS + (tid & ~31) >= n) continue;    // (the whole warp: nothing to sort)
        // loops, not unrolled: the code runs once per launch, and fetching it is what it would cost
#pragma unroll 1
        for (int size = 2; size <= 32; size <<= 1)
#pragma unroll 1
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                const unsigned long long y = __shfl_xor_sync(0xffffffffu, x[e], stride);
                const bool keep_large = ((lane & size & 31) == 0) == ((lane & stride) == 0);      // (size 32: descending)
                x[e] = (x[e] > y) == keep_large ? x[e] : y;
            }
    }
    unsigned long long *from = spare, *to = list;
    __syncthreads();                                         // the list has been read
#pragma unroll
    for (int e = 0; e < E; ++e) from[e * SEL_THREADS + tid] = x[e];
    __syncthreads();
    for (int run = 32; run < n; run <<= 1) {
#pragma unroll 1
        for (int e = 0; e < E; ++e) {
            const int i = e * SEL_THREADS + tid, at = i & (run - 1), other = (i ^ run) & ~(run - 1);
            const bool right = (i & run) != 0;               // equals (padding) keep their order: the left run's first
            const unsigned long long me = from[i];
            int lo = 0, len = run;                           // elements of the other run before this one: in [lo, lo + len]
            while (len > 0) {
                const int half = len >> 1;
                const unsigned long long y = from[other + lo + half];
                const bool before = right ? y >= me : y > me;
                lo = before ? lo + half + 1 : lo;
                len = before ? len - half - 1 : half;
            }
            to[(i & ~(2 * run - 1)) + at + lo] = me;
        }
        __syncthreads();
        unsigned long long* t = from;
        from = to;
        to = t;
    }
#pragma unroll
    for (int e = 0; e < E; ++e) x[e] = from[e * SEL_THREADS + tid];
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (e * SEL_THREADS + tid < k) emit(x[e], e * SEL_THREADS + tid, src, parents, codes, scores);
}

// ... of a list of at most SEL_LIST in `room`, the sort buffer behind it.
__device__ __forceinline__ void order_and_emit(unsigned long long* room, int n, int k, SelectShared& sh, const ScoreSource& src, int32_t* parents, int32_t* codes, float* scores) {
    if (n <= SEL_THREADS) sort_and_emit<1>(room, room + SEL_LIST, n, k, sh, src, parents, codes, scores);
    else if (n <= 2 * SEL_THREADS) sort_and_emit<2>(room, room + SEL_LIST, n, k, sh, src, parents, codes, scores);
    else sort_and_emit<SEL_LIST / SEL_THREADS>(room, room + SEL_LIST, n, k, sh, src, parents, codes, scores);
}

// Running maximum of a thread's candidates in increasing index order: the larger score, the earlier one of equals, NaN below
// every number (the order of the composites, on floats: a third of the instructions).
struct Best {
    float s = 0.f;
    uint32_t i = 0xffffffffu;      // none
    __device__ __forceinline__ void take(float x, uint32_t at) {
        const bool better = x > s || i == 0xffffffffu || (s != s && x == x);
        s = better ? x : s;
        i = better ? at : i;
    }
    __device__ __forceinline__ unsigned long long composite(const ScoreSource& src) const { return i == 0xffffffffu ? 0ull : src.join(score_bits(s), i); }
};

// Where candidate j of place `me` lies when `span` (a power of two) threads share a range: consecutive threads take
// consecutive candidates of a stripe, turned by SEL_ROTATE from stripe to stripe.
__device__ __forceinline__ uint32_t place_of(int j, uint32_t me, uint32_t span) { return (uint32_t)j * span + ((me + (uint32_t)j * SEL_ROTATE) & (span - 1)); }

// A request's scratch is one selection's at a time, and selections of one request may be in flight on several streams: who uses it
// has claimed it.  The claim (a word per request, zero when the context starts): the address the claimant's parents go to, which is
// its alone while it is in flight, and how many CTAs of its launch of shares found the claim theirs, so that one word says all.
// Nobody waits for a claim: a launch of shares that does not get it for all of its CTAs leaves the next launch to select
// exhaustively from the candidates themselves, by one CTA - slow, but two selections of one request at a time are rare.  (Cost, us a
// selection: 0.3 for the claim, 0.3 for the code beside the path; marks in the shares' entries in place of a claim, read and written
// with them as 128 bits, 0.7 for the cluster and 1.8 for one CTA.)
struct Claim {
    static constexpr int COUNT_BITS = 11;                    // of at most ONELA_SELECT_PARTS * 4 CTAs
    static_assert(ONELA_SELECT_PARTS * 4 < 1 << COUNT_BITS, "CTAs of a launch of shares");
    unsigned long long *word, token;
    __device__ __forceinline__ Claim(unsigned long long* claims, int req, const int32_t* parents_of_request)
        : word(claims + req), token(reinterpret_cast<unsigned long long>(parents_of_request) >> 2 << COUNT_BITS) {}
    // one thread of a CTA: ask, and later (the answer takes as long as a load) settle
    __device__ __forceinline__ unsigned long long ask() const { return atomicCAS(word, 0ull, token + 1); }
    __device__ __forceinline__ bool settle(unsigned long long answer) const {
        if (answer == 0ull) return true;
        if ((answer ^ token) >> COUNT_BITS) return false;
        atomicAdd(word, 1ull);
        return true;
    }
    __device__ __forceinline__ unsigned long long state() const { return __ldcg(word); }
    __device__ __forceinline__ bool mine(unsigned long long state) const { return ((state ^ token) >> COUNT_BITS) == 0ull; }
    __device__ __forceinline__ void release() const { __stcg(word, 0ull); }      // one thread, when the scratch has been read
};

// The largest of every share of SEL_HELD candidates, to scratch[request][share].  Share t of 16 384 candidates has its members at
// place_of(m, t, 1024); a CTA finds 64 shares' largest, four members per thread, so that the loads spread over all SMs.
constexpr int SHARE_THREADS = 256, SHARES_PER_CTA = 64;
__global__ void __launch_bounds__(SHARE_THREADS) spread_shares_kernel(const float* __restrict__ beam_scores, const float* __restrict__ cand_logp, int W_prev, int C,
                                                                      uint32_t magic, int shift, int k, unsigned long long* __restrict__ scratch,
                                                                      unsigned long long* claims, const int32_t* parents) {
    constexpr int MEMBERS = SEL_HELD * SHARES_PER_CTA / SHARE_THREADS;
    static_assert(SEL_THREADS % SHARES_PER_CTA == 0 && SHARES_PER_CTA % 32 == 0 && MEMBERS * SHARE_THREADS == SEL_HELD * SHARES_PER_CTA, "shares of a CTA");
    __shared__ unsigned long long part[SHARE_THREADS];
    __shared__ bool s_mine;
    const int tid = threadIdx.x, req = blockIdx.y;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Claim claim(claims, req, parents + (long long)req * k);
    const unsigned long long answer = tid == 0 ? claim.ask() : 0ull;      // (comes while the candidates do)
    const uint32_t N = (uint32_t)W_prev * (uint32_t)C, share = blockIdx.x * SHARES_PER_CTA + (tid & (SHARES_PER_CTA - 1));
    const uint32_t first = share / SEL_THREADS * (SEL_HELD * SEL_THREADS);
    const ScoreSource src{beam_scores + (long long)req * W_prev, cand_logp + (long long)req * N, magic, shift, C};
    Best best;
#pragma unroll
    for (int j = 0; j < MEMBERS; ++j) {
        const uint32_t i = first + place_of(tid / SHARES_PER_CTA * MEMBERS + j, share & (SEL_THREADS - 1), SEL_THREADS);
        if (i < N) best.take(src.score(i), i);
    }
    part[tid] = best.composite(src);
    if (tid == 0) s_mine = claim.settle(answer);
    __syncthreads();
    if (s_mine && tid < SHARES_PER_CTA) {
        unsigned long long x = part[tid];
#pragma unroll
        for (int j = SHARES_PER_CTA; j < SHARE_THREADS; j += SHARES_PER_CTA) x = max(x, part[j + tid]);
        scratch[(long long)req * (ONELA_SELECT_PARTS * SEL_CAP) + share] = x;
    }
}

// The largest of every share of 16 V consecutive candidates, to scratch[request][share]: V candidates per thread and step, the
// largest of sixteen threads' by shuffles; a CTA takes 1024 candidates, so that the loads spread over all SMs.
template <int V>
__global__ void __launch_bounds__(SHARE_THREADS) select_shares_kernel(const float* __restrict__ beam_scores, const float* __restrict__ cand_logp, int W_prev, int C,
                                                                      uint32_t magic, int shift, int k, unsigned long long* __restrict__ scratch,
                                                                      unsigned long long* claims, const int32_t* parents) {
    __shared__ bool s_mine;
    const int tid = threadIdx.x, req = blockIdx.y;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Claim claim(claims, req, parents + (long long)req * k);
    const unsigned long long answer = tid == 0 ? claim.ask() : 0ull;      // (comes while the candidates do)
    const uint32_t N = (uint32_t)W_prev * (uint32_t)C;
    const ScoreSource src{beam_scores + (long long)req * W_prev, cand_logp + (long long)req * N, magic, shift, C};
    scratch += (long long)req * (ONELA_SELECT_PARTS * SEL_CAP);
    unsigned long long best[4 / V];
#pragma unroll
    for (int j = 0; j < 4 / V; ++j) {
        best[j] = 0ull;
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const uint32_t i = blockIdx.x * 1024u + (j * SHARE_THREADS + tid) * V + e;
            if (i < N) best[j] = max(best[j], src(i));
        }
    }
    if (tid == 0) s_mine = claim.settle(answer);
    __syncthreads();
    if (!s_mine) return;
#pragma unroll
    for (int j = 0; j < 4 / V; ++j) {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) best[j] = max(best[j], __shfl_xor_sync(0xffffffffu, best[j], o));
        const uint32_t share = blockIdx.x * (64u / V) + (j * SHARE_THREADS + tid) / 16;
        if ((tid & 15) == 0 && share * (16u * V) < N) scratch[share] = best[j];
    }
}

// The k best of a request from its shares' largest (at most 16 384), one CTA: a bound that at least k of the shares reach, the
// candidates of those shares that reach it, their order.  (A cluster that shared this work out spent 4 us of 14 in its barriers.)
__global__ void __launch_bounds__(SEL_THREADS) select_of_shares_kernel(const float* __restrict__ beam_scores, const float* __restrict__ cand_logp, int W_prev, int C,
                                                                       uint32_t magic, int shift, int k, int log2_share, unsigned long long* __restrict__ scratch,
                                                                       unsigned long long* claims, unsigned parts, int32_t* __restrict__ parents,
                                                                       int32_t* __restrict__ codes, float* __restrict__ scores) {
    extern __shared__ unsigned long long room[];             // [2][SEL_LIST]: list and sort buffer; the shares that reach the bound
    __shared__ SelectShared sh;
    __shared__ unsigned n_list, n_hits;
    const int tid = threadIdx.x, req = blockIdx.x;
    if (tid == 0) n_list = n_hits = 0u;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t N = (uint32_t)W_prev * (uint32_t)C, shares = (N + (1u << log2_share) - 1) >> log2_share;
    const ScoreSource src{beam_scores + (long long)req * W_prev, cand_logp + (long long)req * N, magic, shift, C};
    parents += (long long)req * k;
    codes += (long long)req * k;
    scores += (long long)req * k;
    scratch += (long long)req * (ONELA_SELECT_PARTS * SEL_CAP);
    const Claim claim(claims, req, parents);
    const unsigned long long state = claim.state();
    unsigned long long held[SEL_HELD];
#pragma unroll
    for (int j = 0; j < SEL_HELD; ++j) {
        const uint32_t i = (uint32_t)j * SEL_THREADS + tid;
        held[j] = i < shares ? __ldcg(scratch + i) : 0ull;
    }
    unsigned n = N;                                          // candidates that the exhaustive selection has to look at: all of them
    const unsigned long long* list = nullptr;                // ... or those of a list
    if (state == claim.token + parts) {
        const unsigned long long bound = bound_of(held, k, sh);
        uint16_t* hits = reinterpret_cast<uint16_t*>(room + 2 * SEL_LIST);
#pragma unroll
        for (int j = 0; j < SEL_HELD; ++j)
            if (held[j] >= bound) hits[atomicAdd(&n_hits, 1u)] = (uint16_t)(j * SEL_THREADS + tid);
        __syncthreads();
        auto each = [&](auto&& put) {
            const uint32_t todo = n_hits << log2_share;
#pragma unroll 4
            for (uint32_t x = tid; x < todo; x += SEL_THREADS) {
                const uint32_t i = ((uint32_t)hits[x >> log2_share] << log2_share) + (x & ((1u << log2_share) - 1u));
                if (i < N) {
                    const unsigned long long c = src(i);
                    if (c >= bound) put(c);
                }
            }
        };
        each([&](unsigned long long c) {
            const unsigned at = atomicAdd(&n_list, 1u);
            if (at < SEL_LIST) room[at] = c;
        });
        __syncthreads();
        n = n_list;
        if (n <= SEL_LIST) {
            if (tid == 0) claim.release();
            order_and_emit(room, (int)n, k, sh, src, parents, codes, scores);
            return;
        }
        // too many for shared memory (candidates that gather in few shares): the list again, to global memory
        __syncthreads();
        if (tid == 0) n_list = 0u;
        __syncthreads();
        unsigned long long* out = scratch + SEL_SHARES;
        each([&](unsigned long long c) { out[atomicAdd(&n_list, 1u)] = c; });
        __threadfence_block();
        list = out;
    }
    __syncthreads();
    select_topk<SEL_HELD>([&](uint32_t i) { return list ? __ldcg(list + i) : src(i); }, n, k, sh);
    if (tid == 0 && claim.mine(state)) claim.release();      // (select_topk ends with a barrier; a claim that not all CTAs got ends too)
    sort_and_emit<1>(sh.sel, room, k, k, sh, src, parents, codes, scores);
}

constexpr unsigned N_ALL = 0xffffffffu;       // no list of those that reach the bound

// grid (CTAs of a cluster, requests).  SHARES: the shares' largest come from scratch (spread_shares_kernel),
// and only the shares that reach the bound are looked into.  `scratch` ([request][ONELA_SELECT_PARTS * SEL_CAP], or null): also
// where the candidates that reach the bound go when they do not fit in shared memory (behind the shares).
template <bool SHARES>
__global__ void __launch_bounds__(SEL_THREADS) select_kernel(const float* __restrict__ beam_scores, const float* __restrict__ cand_logp, int W_prev, int C,
                                                             uint32_t magic, int shift, int k, unsigned long long* __restrict__ scratch,
                                                             unsigned long long* claims, unsigned parts, int32_t* __restrict__ parents,
                                                             int32_t* __restrict__ codes, float* __restrict__ scores) {
    extern __shared__ unsigned long long room[];             // [8][1024]: the threads' largest; later list and sort
    __shared__ SelectShared sh;
    __shared__ unsigned n_list, n_mine, n_hits, s_at, s_claimed;
    __shared__ unsigned long long s_bound;
    const int tid = threadIdx.x;
    const int ctas = gridDim.x, rank = blockIdx.x, req = blockIdx.y;
    if (tid == 0) n_mine = n_hits = 0u;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t N = (uint32_t)W_prev * (uint32_t)C;
    const ScoreSource src{beam_scores + (long long)req * W_prev, cand_logp + (long long)req * N, magic, shift, C};
    parents += (long long)req * k;
    codes += (long long)req * k;
    scores += (long long)req * k;
    if (scratch) scratch += (long long)req * (ONELA_SELECT_PARTS * SEL_CAP);
    const uint32_t span = (uint32_t)ctas * SEL_THREADS, me = (uint32_t)rank * SEL_THREADS + tid;
    const uint32_t items = SHARES ? (N + SEL_HELD * SEL_THREADS - 1) / (SEL_HELD * SEL_THREADS) * SEL_THREADS : N;     // candidates, or shares
    const int stripes = (int)((items + span - 1) / span);
    const Claim claim(claims, req, parents);
    unsigned long long state = 0ull;
    if constexpr (SHARES) state = claim.state();
    const bool shared = !SHARES || state == claim.token + parts;      // (the same for the whole cluster: only its first CTA ends its claim)
    // 1. this thread's candidates (shares)
    unsigned long long best = 0ull;
    if constexpr (SHARES) {
#pragma unroll 8
        for (int j = 0; j < stripes; ++j) {
            const uint32_t i = place_of(j, me, span);
            if (i < items) best = max(best, __ldcg(scratch + i));
        }
    } else {
        Best top;
#pragma unroll 8
        for (int j = 0; j < stripes; ++j) {
            const uint32_t i = place_of(j, me, span);
            if (i < N) top.take(src.score(i), i);
        }
        best = top.composite(src);
    }
    unsigned n = N_ALL;
    bool listed = false;
    if (shared) {
        // 2. the bound
        unsigned long long bound = 1ull;                         // (a composite is never 0: the index word of a candidate is not)
        if (ctas > 1) {
            st_cluster64(in_first_cta(room + rank * SEL_THREADS + tid), best);
            cluster_barrier();
            if (rank == 0) {
                unsigned long long mine[SEL_CTAS];
#pragma unroll
                for (int c = 0; c < SEL_CTAS; ++c) mine[c] = c < ctas ? room[c * SEL_THREADS + tid] : 0ull;
                bound = bound_of(mine, k, sh);
                if (tid == 0) { s_bound = bound; n_list = 0u; }
            }
            cluster_barrier();
            if (rank != 0) bound = ld_cluster64(in_first_cta(&s_bound));
        } else {
            if (stripes > 1) {
                const unsigned long long mine[1] = {best};
                bound = bound_of(mine, k, sh);
            }
            if (tid == 0) n_list = 0u;
            __syncthreads();
        }
        // 3. the candidates that reach it: the shares whose largest does are listed, then all threads look into their members;
        // what they find goes to a list of this CTA's, which is then appended to the first CTA's
        uint16_t* hits = reinterpret_cast<uint16_t*>(room + 2 * SEL_LIST);      // thread (+ 1024 x stripe: share), of this CTA
        if constexpr (SHARES) {
            if (best >= bound)
                for (int j = 0; j < stripes; ++j) {
                    const uint32_t i = place_of(j, me, span);
                    if (i < items && __ldcg(scratch + i) >= bound) hits[atomicAdd(&n_hits, 1u)] = (uint16_t)(j * SEL_THREADS + tid);
                }
        } else if (best >= bound) {
            hits[atomicAdd(&n_hits, 1u)] = (uint16_t)tid;
        }
        __syncthreads();
        const int members = SHARES ? SEL_HELD : stripes;
        auto each = [&](auto&& put) {
            const int todo = (int)n_hits * members;
#pragma unroll 2
            for (int x = tid; x < todo; x += SEL_THREADS) {
                const int q = x / members, m = x - q * members;
                uint32_t i = hits[q];
                if constexpr (SHARES) {                          // share i of stripe j: member m among the 16 384 candidates it lies in
                    i = place_of((int)(i / SEL_THREADS), (uint32_t)rank * SEL_THREADS + (i & (SEL_THREADS - 1)), span);
                    i = i / SEL_THREADS * (SEL_HELD * SEL_THREADS) + place_of(m, i & (SEL_THREADS - 1), SEL_THREADS);
                } else {
                    i = place_of(m, (uint32_t)rank * SEL_THREADS + i, span);
                }
                if (i < N) {
                    const unsigned long long c = src(i);
                    if (c >= bound) put(c);
                }
            }
        };
        unsigned long long* mine = room + SEL_LIST;              // (beside the first CTA's list)
        each([&](unsigned long long c) {
            const unsigned at = atomicAdd(&n_mine, 1u);
            if (at < SEL_LIST) mine[at] = c;
        });
        __syncthreads();
        const unsigned cnt = n_mine;
        if (tid == 0) s_at = add_cluster(in_first_cta(&n_list), cnt);
        __syncthreads();
        {
            const unsigned at = s_at;
            const uint32_t list_at = in_first_cta(room);
            for (unsigned i = tid; i < min(cnt, (unsigned)SEL_LIST); i += SEL_THREADS)
                if (at + i < SEL_LIST) st_cluster64(list_at + (at + i) * 8, mine[i]);
        }
        cluster_barrier();
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(n) : "r"(in_first_cta(&n_list)) : "memory");
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");       // this thread has read the first CTA's memory
        if (n > SEL_LIST && scratch) {
            // too many for shared memory (candidates that gather in few threads' shares): the list again, to global memory
            asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
            if (rank == 0 && tid == 0) {
                n_list = 0u;
                s_claimed = SHARES || claim.settle(claim.ask());
            }
            cluster_barrier();
            unsigned claimed;
            asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(claimed) : "r"(in_first_cta(&s_claimed)) : "memory");
            listed = claimed != 0u;
            unsigned long long* out = scratch + SEL_SHARES;
            if (listed) each([&](unsigned long long c) { out[add_cluster(in_first_cta(&n_list), 1u)] = c; });
            __threadfence();
            asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        }
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
    if (rank != 0) return;
    if (n <= SEL_LIST) {
        if (SHARES && tid == 0) claim.release();             // (the cluster is through with the shares)
        order_and_emit(room, (int)n, k, sh, src, parents, codes, scores);
    } else {                                                 // exhaustively, over the list or over all candidates
        if (listed) {
            const unsigned long long* list = scratch + SEL_SHARES;
            select_topk<SEL_HELD>([&](uint32_t i) { return __ldcg(list + i); }, n, k, sh);
        } else {
            __syncthreads();
            select_topk<SEL_HELD>(src, N, k, sh);
        }
        if (tid == 0 && (SHARES ? claim.mine(state) : listed)) claim.release();      // (select_topk ends with a barrier)
        sort_and_emit<1>(sh.sel, room, k, k, sh, src, parents, codes, scores);
    }
}

}  // namespace

// Whether the shares' largest come from a launch of their own.  The shares have to be a few times as many as the survivors for
// their bound to leave little more than those (three times: 1.2 k candidates expected).  Where the lines lie, measured as whole
// generations (select, index, decode; us, one cluster reading all candidates / from shares): one CTA for the rest - 128 x 1000 ->
// 128 115 / 101, 4 x 200 x 512 -> 200 98.5 / 94.2; a cluster for the rest - 2 x 512 x 128 -> 512 127.5 / 121.4, 8 x 512 x 512 -> 512
// 215 / 193, 3 x 333 x 512 -> 333 281 / 250.  One CTA at 512 survivors of 8 x 512 x 512 198, at 1000 of 4 x 1000 x 1000 194 against the
// cluster's 152: it then fetches 16 000 candidates by itself.  (Before the scratch was claimed, 0.5 us a selection.)
// Between 12 800 and 16 384 candidates it depends on how many survive (as a graph, one cluster / from shares): 8 x 60 x 256 -> 60 51.8 /
// 50.0, 1 x 16 x 1000 -> 16 49.2 / 47.1, 4 x 13 x 1000 -> 13 50.2 / 49.1; 1 x 100 x 160 -> 100 49.2 / 50.2, 4 x 128 x 100 -> 128 63.5 / 64.9, 2 x
// 200 x 65 -> 200 49.1 / 51.2; issued eagerly the first three gain less, the last three lose up to 6 %.  Below, from shares is slower even
// where few survive (8 x 16 x 512 -> 16 63.7 / 65.5, 4 x 60 x 100 -> 60 61.4 / 64.5, both eagerly).
constexpr int SHARES_FROM = 16384, ONE_CTA_TO = 256;
bool from_shares(long long candidates, int k) { return candidates > (k <= ONE_CTA_TO ? SHARES_FROM : 2 * SEL_HELD * SEL_THREADS) && candidates >= 3ll * SEL_SHARE * k; }
int select_launches(long long candidates, int32_t W_new) { return from_shares(candidates, W_new) ? 2 : 1; }

cudaError_t launch_select(const float* beam_scores, const float* cand_logp, int32_t req_count, int32_t W_prev, int32_t C,
                          int32_t W_new, unsigned long long* scratch, unsigned long long* claims, int32_t* parents, int32_t* codes,
                          float* scores, cudaStream_t stream) {
    const long long N = (long long)W_prev * C;
    if (N > (long long)ONELA_SELECT_PARTS * 4096) return cudaErrorInvalidValue;
    // CTAs per request: one while the candidates are at most four per thread (the exchange between CTAs costs more than the
    // loads it shares out), then as many as keep them in registers, up to a portable cluster
    const bool shares = scratch && from_shares(N, W_new);
    const long long blocks = (N + SEL_HELD * SEL_THREADS - 1) / (SEL_HELD * SEL_THREADS);       // of 1024 shares
    const int ctas = shares ? (blocks <= 4 ? 4 : SEL_CTAS)
                            : N <= 4 * SEL_THREADS ? 1 : N <= 2 * SEL_HELD * SEL_THREADS ? 2 : N <= 4 * SEL_HELD * SEL_THREADS ? 4 : SEL_CTAS;
    // the threads' largest, later list and sort buffer: 64 KB; the shares that reach the bound: 16 KB
    constexpr int SMEM = SEL_CTAS * SEL_THREADS * (int)sizeof(unsigned long long) + SEL_SHARES / SEL_CTAS * (int)sizeof(uint16_t);
    static_assert(ONE_CTA_TO + 32 <= SEL_SHARES / SEL_CTAS && ONE_CTA_TO / 8 <= 32, "shares that the bound may leave to one CTA");
    static_assert(2 * SEL_LIST == SEL_CTAS * SEL_THREADS, "list and sort buffer");
    static_assert(SEL_SHARES + (SEL_CAP + SEL_CAP / 8) * (ONELA_SELECT_PARTS * 4096 / (SEL_CTAS * SEL_THREADS)) <= ONELA_SELECT_PARTS * SEL_CAP, "scratch");
    // one-time set-up per device (function attributes belong to a device's context)
    constexpr int MAX_DEVICES = 64;
    static std::mutex setup_mutex;
    static bool ready[MAX_DEVICES] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(setup_mutex);
        if (!ready[dev]) {
            cudaError_t e = cudaFuncSetAttribute(select_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(select_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(select_of_shares_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
            if (e != cudaSuccess) return e;
            ready[dev] = true;
        }
    }
    uint32_t magic;
    int shift;
    divide_by(C, magic, shift);
    unsigned parts = 0;                  // CTAs per request of the launch of shares
    if (shares) {
        cudaError_t e;
        if (W_new <= ONE_CTA_TO) {       // shares of 16 candidates; of 64 where the CTA's threads would not hold that many
            const bool wide = N > 1ll * SEL_SHARE * SEL_HELD * SEL_THREADS;
            static_assert(4ll * SEL_SHARE * SEL_HELD * SEL_THREADS >= (long long)ONELA_SELECT_PARTS * 4096, "the shares of the largest request");
            parts = (unsigned)((N + 1023) / 1024);
            e = launch_dependent(wide ? select_shares_kernel<4> : select_shares_kernel<1>, dim3(parts, req_count), dim3(SHARE_THREADS), 0, stream, beam_scores, cand_logp,
                                 W_prev, C, magic, shift, W_new, scratch, claims, parents);
            if (e != cudaSuccess) return e;
            return launch_dependent(select_of_shares_kernel, dim3(req_count), dim3(SEL_THREADS), SMEM, stream, beam_scores, cand_logp, W_prev, C, magic, shift,
                                    W_new, wide ? 6 : 4, scratch, claims, parts, parents, codes, scores);
        }
        parts = (unsigned)(blocks * (SEL_THREADS / SHARES_PER_CTA));
        e = launch_dependent(spread_shares_kernel, dim3(parts, req_count), dim3(SHARE_THREADS), 0, stream, beam_scores, cand_logp, W_prev, C, magic, shift, W_new,
                             scratch, claims, parents);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas, req_count);
    cfg.blockDim = dim3(SEL_THREADS);
    cfg.dynamicSmemBytes = SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = ctas;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, shares ? select_kernel<true> : select_kernel<false>, beam_scores, cand_logp, W_prev, C, magic, shift, W_new, scratch, claims, parts, parents,
                              codes, scores);
}

}  // namespace onela

// ---------------------------------------------------------------------------------------------------------------
// Beam selection without a workspace (declared in onela.h as onela_select_beams_static): the same launch, which needs no
// device memory beyond the CTAs' own; where too many candidates reach the bound for shared memory, the exhaustive selection
// runs over the candidates themselves.
extern "C" onela_status onela_select_beams_static(const float* beam_scores_dev, const float* cand_logp_dev, int32_t req_count,
                                                  int32_t W_prev, int32_t C, int32_t W_new, int32_t* parents_out_dev,
                                                  int32_t* codes_out_dev, float* scores_out_dev, void* stream) {
    using namespace onela;
    if (!beam_scores_dev || !cand_logp_dev || !parents_out_dev || !codes_out_dev || !scores_out_dev) return ONELA_E_INVAL;
    if (req_count < 1 || W_prev < 1 || C < 1 || W_new < 1) return ONELA_E_INVAL;
    // the call's documented limits: beyond them the caller has to use onela_select_beams, or split the batch
    constexpr int STATIC_REQUESTS = 2;
    if (req_count > STATIC_REQUESTS) return ONELA_E_CAPACITY;
    if ((int64_t)W_prev * C > (int64_t)ONELA_SELECT_PARTS * 4096) return ONELA_E_CAPACITY;
    if (W_new > ONELA_SELECT_CAP || W_new > (int64_t)W_prev * C) return ONELA_E_CAPACITY;
    if (launch_select(beam_scores_dev, cand_logp_dev, req_count, W_prev, C, W_new, nullptr, nullptr, parents_out_dev, codes_out_dev,
                      scores_out_dev, static_cast<cudaStream_t>(stream)) != cudaSuccess)
        return ONELA_E_CUDA;
    return ONELA_OK;
}
