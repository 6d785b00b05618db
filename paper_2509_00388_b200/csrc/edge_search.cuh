// The edges of one source that can be among its m largest, found by one warp over a row of cosines in
// shared memory.
#pragma once

#include "common.cuh"

namespace graphkv {

// The edges of x(0 .. n) (lane-strided: element i * 32 + lane, kCandEmpty where there is none) that reach a
// bound at which between m and kCandCap of them do; with too many near-ties, exactly the m largest (lowest
// positions first; kOrdered = false, where i is in no order of position: none, and -1 returned).  put(slot, e, i).  Returns their number, and in *bound a value that m of them reach (-1
// with fewer than m).  `from`: -1, or a value that at least m of them are known to reach.  Rolled loops over
// shared memory: the code runs once per source.
template <bool kOrdered = true, typename At, typename Put>
__device__ __forceinline__ int warp_list_top(int n, int m, float from, At x, Put put, float *bound)
{
    const int lane = threadIdx.x & 31;
    // how many reach t0, t1 (packed)
    auto reach2 = [&](float t0, float t1) {
        uint32_t c = 0;
#pragma unroll 4
        for (int i = lane; i < n; i += 32) {
            const float e = x(i);
            c += (e >= t0 ? 1u : 0u) + (e >= t1 ? 0x10000u : 0u);
        }
        return __reduce_add_sync(0xffffffffu, c);
    };
    float lo = from, hi = 1.0f;
    const float half = from + 0.5f * (1.0f - from);
    uint32_t c = reach2(from, half);
    int have = (int)(c & 0xffffu);
    *bound = -1.0f;
    if ((int)(c >> 16) >= m) lo = half, have = (int)(c >> 16);
    else hi = half;
    for (int it = 0; have > kCandCap && it < 16; ++it) {
        const float t0 = lo + (hi - lo) * (1.0f / 3.0f), t1 = lo + (hi - lo) * (2.0f / 3.0f);
        c = reach2(t0, t1);
        if ((int)(c >> 16) >= m) {
            lo = t1;
            have = (int)(c >> 16);
        } else if ((int)(c & 0xffffu) >= m) {
            lo = t0;
            hi = t1;
            have = (int)(c & 0xffffu);
        } else {
            hi = t0;
        }
    }
    if (have >= m) *bound = lo;
    if (!kOrdered && have > kCandCap) return -1;
    uint32_t exact = 0;                         // with too many near-ties: the key of the m-th largest
    int ties = 0;                               // and how many of its ties belong to the m
    if (have > kCandCap) {
        uint32_t klo = float_to_key(lo), khi = float_to_key(1.0f) + 1u;
        while (khi - klo > 1u) {
            const uint32_t mid = klo + (khi - klo) / 2u;
            uint32_t q = 0;
            for (int i = lane; i < n; i += 32) q += float_to_key(x(i)) >= mid;
            if ((int)__reduce_add_sync(0xffffffffu, q) >= m) klo = mid;
            else khi = mid;
        }
        exact = klo;
        uint32_t q = 0;
        for (int i = lane; i < n; i += 32) q += float_to_key(x(i)) > exact;
        ties = m - (int)__reduce_add_sync(0xffffffffu, q);
    }
    int at = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const float e = i0 + lane < n ? x(i0 + lane) : kCandEmpty;
        bool keep = e >= lo;
        if (exact) {
            const uint32_t key = float_to_key(e);
            const unsigned eq = __ballot_sync(0xffffffffu, key == exact);
            keep = key > exact || (key == exact && __popc(eq & ((1u << lane) - 1u)) < ties);
            ties -= min(ties, __popc(eq));
        }
        const unsigned bm = __ballot_sync(0xffffffffu, keep);
        if (keep) put(at + __popc(bm & ((1u << lane) - 1u)), e, i0 + lane);
        at += __popc(bm);
    }
    return at;
}

// A cosine from the products, which may leave [-1, 1] by a rounding or be NaN (no edge).
__device__ __forceinline__ float clamped_edge(float raw)
{
    return raw == raw ? fminf(fmaxf(raw, -1.0f), 1.0f) : kCandEmpty;
}

// A lower bound of the m-th largest edge of a row, from the maxima best[0 .. kParts) of disjoint parts of it
// (unclamped cosines; -inf for a part without an edge; kParts 256 or 512): the (m + 1)-th largest of them,
// or a little less, whatever the source's own place (one of the m + 1) holds.  About as many edges reach it.
// An interpolating search on the logarithm of the count, eight maxima per lane, two tries per step.
template <int kParts>
__device__ __forceinline__ float warp_bound_of_maxima(const float *best, int m)
{
    const int lane = threadIdx.x & 31;
    const float4 *b4 = reinterpret_cast<const float4 *>(best);
    float v[8];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        float4 s = b4[q * 32 + lane];
        if constexpr (kParts == 512) {          // (two parts in one)
            const float4 t = b4[(q + 2) * 32 + lane];
            s = make_float4(fmaxf(s.x, t.x), fmaxf(s.y, t.y), fmaxf(s.z, t.z), fmaxf(s.w, t.w));
        }
        v[4 * q] = s.x; v[4 * q + 1] = s.y; v[4 * q + 2] = s.z; v[4 * q + 3] = s.w;
    }
    auto reach2 = [&](float t0, float t1) {
        uint32_t c = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) c += (v[q] >= t0 ? 1u : 0u) + (v[q] >= t1 ? 0x10000u : 0u);
        return __reduce_add_sync(0xffffffffu, c);
    };
    // (a bound above 1 would tell apart cosines that clamp to the same value, and so would one at or below -1)
    float a = fminf(fminf(fminf(v[0], v[1]), fminf(v[2], v[3])), fminf(fminf(v[4], v[5]), fminf(v[6], v[7])));
    float b = fmaxf(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])), fmaxf(fmaxf(v[4], v[5]), fmaxf(v[6], v[7])));
    // (clamped to [-1, 1], the floats shifted to [1, 3] are ordered like their bits)
    a = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(fmaxf(a, -1.0f) + 2.0f))) - 2.0f;
    b = fminf(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(b, -1.0f) + 2.0f))) - 2.0f, 1.0f);
    uint32_t c = reach2(a, b);
    int ca = (int)(c & 0xffffu), cb = (int)(c >> 16);
    float lo = -INFINITY;                       // fewer than m + 1 parts with an edge
    if (cb > m) lo = b;
    else if (ca > m) {
        lo = a;
        const float w0 = __log2f(1.2f * (float)m + 1.5f), w1 = __log2f(1.06f * (float)m + 1.0f);
        for (int it = 0; it < 10; ++it) {
            const float la = __log2f((float)ca), lb = __log2f(fmaxf((float)cb, 0.5f)), r = __fdividef(b - a, la - lb);
            const float t0 = it < 6 ? a + fmaxf(la - w0, 0.04f * (la - lb)) * r : a + (b - a) * (1.0f / 3.0f);
            const float t1 = it < 6 ? a + fminf(la - w1, 0.96f * (la - lb)) * r : a + (b - a) * (2.0f / 3.0f);
            c = reach2(t0, t1);
            const int c0 = (int)(c & 0xffffu), c1 = (int)(c >> 16);
            if (c1 > m) {
                lo = a = t1;
                ca = c1;
            } else if (c0 > m) {
                lo = a = t0;
                ca = c0;
                b = t1;
                cb = c1;
            } else {
                b = t0;
                cb = c0;
            }
            if (ca <= m + (m >> 2) + 2) break;
        }
    }
    return lo <= -1.0f ? -INFINITY : lo;
}

}  // namespace graphkv
