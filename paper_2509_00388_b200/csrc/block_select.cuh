// Selections by one CTA of 512 threads (or groups of them) over values in its shared memory.
//
// Bound: latency.  A barrier costs 45 clocks, a dependent load from shared memory 30 to 80, a warp reduction 25 to 45,
// an addition with a result 110, an integer division by a variable 150; a selection is a chain of these over a few elements
// per thread.  So: one histogram over the range the values are known to lie in instead of digits of their
// bits, its threshold bin ranked by counting; sizes of groups are constants; no scan where a reduction will do.
// Measured for 1003 values on one SM: the 32 largest in order 4000 -> 1900 clocks.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace graphkv {
namespace bs {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kBins = 1024;
constexpr int kRankCap = 128;           // elements of the threshold bin ranked by counting
constexpr int kTopMax = 32;             // elements group_top takes at most
constexpr uint32_t kAllTies = 0xffffffffu;

__device__ __forceinline__ uint32_t incl_scan(uint32_t v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// What a selection keeps: keys above thr, and of those equal to it the first `ties` by position (kAllTies: all).
struct Kept {
    uint32_t thr, ties;
};

// The least and the greatest key of val[0 .. n).  wcnt: 2 * kWarps words.  Starts after and ends with a barrier.
__device__ __forceinline__ void block_range(const float *val, int n, uint32_t *wcnt, uint32_t &lo, uint32_t &hi)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    lo = 0xffffffffu;
    hi = 0u;
    for (int i = threadIdx.x; i < n; i += kThreads) {
        const uint32_t key = float_to_key(val[i]);
        lo = min(lo, key);
        hi = max(hi, key);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
        wcnt[warp] = lo;
        wcnt[kWarps + warp] = hi;
    }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, wcnt[lane & (kWarps - 1)]);
    hi = __reduce_max_sync(0xffffffffu, wcnt[kWarps + (lane & (kWarps - 1))]);
    __syncthreads();
}

// The k largest (1 <= k <= n) of val[0 .. n).  Where the threshold is expected to lie, lo .. hi in keys, is cut into
// bins; the lowest bin takes all below, the highest all above, so any lo <= hi gives the right result.  hist: kBins words
// and kRankCap words behind them; wcnt: kWarps, misc: 8 words.  Starts after and ends with a barrier.
__device__ __noinline__ Kept block_kth(const float *val, int n, uint32_t k, uint32_t lo, uint32_t hi, uint32_t *hist,
                                       uint32_t *wcnt, uint32_t *misc)
{
    static_assert(kBins == 2 * kThreads, "two bins per thread");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t *list = hist + kBins;
    uint32_t from = 0u, to = 0xffffffffu;           // the keys still in question: those in from .. to
    uint32_t left = k;                              // of them, how many are kept
    while (true) {
        const int shift = max(0, 22 - __clz(hi - lo));              // (hi - lo) >> shift < kBins
        const uint32_t last = (hi - lo) >> shift;
        auto bin_of = [&](uint32_t key) { return key < lo ? 0u : min((key - lo) >> shift, last); };
        reinterpret_cast<uint2 *>(hist)[tid] = make_uint2(0u, 0u);
        if (tid == 0) misc[3] = 0u;
        __syncthreads();
#pragma unroll 4
        for (int i = tid; i < n; i += kThreads) {
            const uint32_t key = float_to_key(val[i]);
            if (key >= from && key <= to) atomicAdd(&hist[bin_of(key)], 1u);
        }
        __syncthreads();
        // the bin that holds the left-th largest: the warps from the first on hold the highest bins
        const uint2 c = reinterpret_cast<const uint2 *>(hist)[kThreads - 1 - tid];      // bins 2 (511 - tid) and + 1
        const uint32_t sum = __reduce_add_sync(0xffffffffu, c.x + c.y);
        if (lane == 0) wcnt[warp] = sum;
        __syncthreads();
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? wcnt[lane & (kWarps - 1)] : 0u);
        if (before < left && before + sum >= left) {
            const uint32_t run = before + incl_scan(c.x + c.y, lane) - (c.x + c.y);
            const uint32_t bin = 2u * (uint32_t)(kThreads - 1 - tid);
            if (run < left && run + c.y >= left) misc[0] = bin + 1u, misc[1] = run, misc[2] = c.y;
            else if (run + c.y < left && run + c.y + c.x >= left) misc[0] = bin, misc[1] = run + c.y, misc[2] = c.x;
        }
        __syncthreads();
        const uint32_t bin = misc[0], in = misc[2];
        left -= misc[1];
        const uint32_t bin_lo = bin == 0u ? from : max(from, lo + (bin << shift));
        const uint32_t bin_hi = bin == last ? to : min(to, lo + (bin << shift) + ((1u << shift) - 1u));
        if (in == left || bin_lo == bin_hi) {       // the whole bin, or ties of one value
            __syncthreads();
            return Kept{bin_lo, in == left ? kAllTies : left};
        }
        if (in <= (uint32_t)kRankCap) {
#pragma unroll 4
            for (int i = tid; i < n; i += kThreads) {
                const uint32_t key = float_to_key(val[i]);
                if (key >= bin_lo && key <= bin_hi) list[atomicAdd(&misc[3], 1u)] = key;
            }
            __syncthreads();
            const int i = tid >> 2, sub = tid & 3;                  // four threads per element
            if (warp * 8 < (int)in) {
                const uint32_t me = i < (int)in ? list[i] : 0u;
                uint32_t gt = 0, ge = 0;                            // larger ones; larger or equal
#pragma unroll 4
                for (int u = sub; u < (int)in; u += 4) {
                    const uint32_t x = list[u];
                    gt += x > me;
                    ge += x >= me;
                }
                uint32_t both = gt | ge << 16;
                both += __shfl_xor_sync(0xffffffffu, both, 1);
                both += __shfl_xor_sync(0xffffffffu, both, 2);
                gt = both & 0xffffu;
                ge = both >> 16;
                if (i < (int)in && gt < left && ge >= left) {       // (ties write the same)
                    misc[4] = me;
                    misc[5] = ge == left ? kAllTies : left - gt;
                }
            }
            __syncthreads();
            return Kept{misc[4], misc[5]};
        }
        lo = from = bin_lo;
        hi = to = bin_hi;
        __syncthreads();
    }
}

// put(t, i) for every element i that is kept, t its rank by position: every warp owns a contiguous run of elements.
// wcnt: 2 * kWarps words.  Starts after a barrier; the words are free after the caller's next.
__device__ __forceinline__ int run_length(int n) { return (ceil_div(n, kWarps) + 31) & ~31; }
// ... where only the first of the ties are kept
template <typename Put>
__device__ __forceinline__ void emit_with_ties(const float *val, int n, Kept th, uint32_t *wcnt, Put put)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, seg = run_length(n), lo = min(warp * seg, n), hi = min(lo + seg, n);
    const unsigned below = (1u << lane) - 1u;
    uint32_t gt = 0, eq = 0;
    for (int pass = 0; pass < 2; ++pass) {
        if (pass == 1) {
            if (lane == 0) {
                wcnt[warp] = gt;
                wcnt[kWarps + warp] = eq;
            }
            __syncthreads();
            gt = __reduce_add_sync(0xffffffffu, lane < warp ? wcnt[lane] : 0u);
            eq = __reduce_add_sync(0xffffffffu, lane < warp ? wcnt[kWarps + lane] : 0u);
        }
        for (int i0 = lo; i0 < hi; i0 += 32) {
            const int i = i0 + lane;
            const uint32_t key = i < hi ? float_to_key(val[i]) : 0u;
            const bool is_gt = i < hi && key > th.thr, is_eq = i < hi && key == th.thr;
            const unsigned bg = __ballot_sync(0xffffffffu, is_gt), be = __ballot_sync(0xffffffffu, is_eq);
            const uint32_t g = gt + __popc(bg & below), e = eq + __popc(be & below);
            if (pass == 1 && (is_gt || (is_eq && e < th.ties))) put((int)(g + min(e, th.ties)), i);
            gt += __popc(bg);
            eq += __popc(be);
        }
    }
}
template <typename Put>
__device__ __forceinline__ void emit_kept(const float *val, int n, Kept th, uint32_t *wcnt, Put put)
{
    if (th.ties != kAllTies) {
        emit_with_ties(val, n, th, wcnt, put);
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, seg = run_length(n);
    const int lo = min(warp * seg, n), hi = min(lo + seg, n);
    constexpr int kQ = 4;
    unsigned bm[kQ];
    uint32_t c = 0;
    auto look = [&](int i0) {
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const int i = i0 + q * 32 + lane;
            bm[q] = __ballot_sync(0xffffffffu, i < hi && float_to_key(i < hi ? val[i] : 0.f) >= th.thr);
        }
    };
    for (int i0 = lo; i0 < hi; i0 += 32 * kQ) {
        look(i0);
#pragma unroll
        for (int q = 0; q < kQ; ++q) c += __popc(bm[q]);
    }
    if (lane == 0) wcnt[warp] = c;
    __syncthreads();
    uint32_t at = __reduce_add_sync(0xffffffffu, lane < warp ? wcnt[lane & (kWarps - 1)] : 0u);
    for (int i0 = lo; i0 < hi; i0 += 32 * kQ) {
        if (hi - lo > 32 * kQ) look(i0);
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            if (bm[q] >> lane & 1u) put((int)(at + __popc(bm[q] & ((1u << lane) - 1u))), i0 + q * 32 + lane);
            at += __popc(bm[q]);
        }
    }
}

// The m <= kTopMax largest of x[0 .. n), ties to the lower position, by a group of T threads (t: this one's number): as
// edge keys in descending order in top[0 .. m), 0 where there are fewer.  The m-th largest of 64 disjoint parts'
// maxima bounds the m-th element from below, and about 1.4 m elements reach it; they are listed and ranked by
// counting.  Returns the number of listed elements: above T (ties) the list is incomplete and `top` not written.
// Starts after and ends with a barrier of the group.
template <int T> struct GroupScratch {
    unsigned long long *cand, *top;             // [T], [kTopMax]
    uint32_t *gm;                               // [64] maxima
    uint32_t *word;                             // [0] listed, [1] the bound
    static constexpr int kBytes = 8 * T + 8 * kTopMax + 4 * 64 + 16;
    __device__ __forceinline__ GroupScratch(uint8_t *p)
        : cand(reinterpret_cast<unsigned long long *>(p)), top(cand + T), gm(reinterpret_cast<uint32_t *>(top + kTopMax)),
          word(gm + 64) {}
};
template <int T> __device__ __forceinline__ void group_bar(int bar)
{
    if constexpr (T == kThreads) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(T) : "memory");
}
// The listed elements cand[0 .. n), n <= T, ranked.
template <int T>
__device__ __forceinline__ void group_rank(const GroupScratch<T> &s, int n, int m, int bar, int t)
{
    constexpr int kShare = T == kThreads ? 4 : 2;
    auto rank = [&](auto share_c) {
        constexpr int share = decltype(share_c)::value;
        const int i = t / share, sub = t % share;
        if ((t & ~31) / share >= n) return;
        const unsigned long long me = i < n ? s.cand[i] : ~0ull;
        int r = 0;
#pragma unroll 4
        for (int u = sub; u < n; u += share) r += s.cand[u] > me;
#pragma unroll
        for (int o = 1; o < share; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        if (i < n && sub == 0 && r < m) s.top[r] = me;
    };
    if (n * kShare <= T) rank(std::integral_constant<int, kShare>{});
    else rank(std::integral_constant<int, 1>{});
    if (t >= n && t < m) s.top[t] = 0ull;
    group_bar<T>(bar);
}
template <int T>
__device__ __forceinline__ int group_top(const float *x, int n, int m, int bar, int t, const GroupScratch<T> &s)
{
    constexpr int kPerWarp = 2048 / T, kQ = T == kThreads ? 4 : 8;
    const int lane = t & 31;
    uint32_t key[kQ], mx = 0u;
    auto load = [&](int i0) {
#pragma unroll
        for (int q = 0; q < kQ; ++q) key[q] = i0 + q * T < n ? float_to_key(x[i0 + q * T]) : 0u;
    };
    for (int i0 = t; i0 - t < n; i0 += kQ * T) {
        load(i0);
#pragma unroll
        for (int q = 0; q < kQ; ++q) mx = max(mx, key[q]);
    }
    // (a part: the lanes of a warp that agree in their low bits, so that a plateau of neighbours is spread)
#pragma unroll
    for (int o = 16; o >= kPerWarp; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    // (the part's number takes the last bits, so that no two are equal)
    if (lane < kPerWarp) s.gm[(t >> 5) * kPerWarp + lane] = (mx & ~63u) | (63u - (uint32_t)((t >> 5) * kPerWarp + lane));
    if (t == 0) s.word[0] = 0u;
    group_bar<T>(bar);
    if (t < 64) {
        const uint32_t me = s.gm[t];
        int r = 0;
#pragma unroll
        for (int u = 0; u < 64; u += 4) {
            const uint4 g = *reinterpret_cast<const uint4 *>(s.gm + u);
            r += (g.x > me) + (g.y > me) + (g.z > me) + (g.w > me);
        }
        if (r == m - 1) s.word[1] = me & ~63u;
    }
    group_bar<T>(bar);
    const uint32_t bound = s.word[1];
    for (int i0 = t; i0 - t < n; i0 += kQ * T) {
        if (n > kQ * T) load(i0);
        unsigned bm[kQ];
        uint32_t c = 0;
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            bm[q] = __ballot_sync(0xffffffffu, i0 + q * T < n && key[q] >= bound);
            c += __popc(bm[q]);
        }
        if (c == 0u) continue;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(s.word, c);
        at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            const uint32_t p = at + __popc(bm[q] & ((1u << lane) - 1u));
            if ((bm[q] >> lane & 1u) && p < (uint32_t)T)
                s.cand[p] = (unsigned long long)key[q] << 32 | (0xffffffffu - (uint32_t)(i0 + q * T));
            at += __popc(bm[q]);
        }
    }
    group_bar<T>(bar);
    const int have = (int)s.word[0];
    if (have <= T) group_rank(s, have, m, bar, t);
    return have;
}

}  // namespace bs
}  // namespace graphkv
