// Decode-side use of a cache: the attention of one new token's queries over `rows` cached keys
// and values per KV head (the full cache, or the compact cache this library builds), as a
// micro-benchmark of what the compression buys at decoding time (Efficiency Analysis: the paper's
// only latency table is decoding latency).
//
//   out[b][hq][:] = sum_j softmax_j(q[b][hq] . K[b][h][j] / sqrt(D)) * V[b][h][j],  h = hq / G
//
// Bound: the cache is read once and nothing else is large, so HBM.  A unit's rows are cut into
// blocks of 8 KB of K and V (16 bf16 or 8 fp32 rows) and its blocks into equal runs, one per CTA.  A
// warp takes whole blocks through a ring of asynchronous copies of its own (two blocks: twelve warps
// keep 96 to 192 KB in flight per SM) and keeps a running softmax of its own, so the loop has no
// barrier.  The warps of a CTA merge in shared memory; a unit that several CTAs share is merged by
// the first of them where they fit a cluster, else by the last to finish, in the same launch.
//
// Measured on one B200, bf16, 8 KV heads, 4 query heads each (plain loads, a barrier per 32 rows and
// a second kernel for the merge before -> now): 32800 rows 145 -> 28 us (4.8 TB/s), 16 x 2080 rows
// 137 -> 25.5 us (5.4 TB/s), 4 x 32800 rows 89 us (6.0 TB/s, 92 % of the copy bandwidth), 544 rows
// 15.4 -> 5.8 us.  About 8 us of a launch are its start, the first
// loads' latency and the merge.  Runs of blocks cut without regard to units (an equal share for
// every SM, but two units in some CTAs, one after the other) measured 34 and 28 us.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"

namespace graphkv {

// Warps of a CTA: 12 where a CTA has an SM to itself, 6 where two share it.
constexpr int kDecWarps = 12, kDecWarps2 = 6;
constexpr int kDecStages = 2;          // blocks in a warp's ring
constexpr int kDecHalf = 4096;         // bytes of K, and of V, in a block
constexpr int kDecStage = 2 * kDecHalf;
template <typename T> __host__ __device__ constexpr int dec_rows() { return kDecHalf / (kHeadDim * (int)sizeof(T)); }
// Fewest blocks a CTA of a shared unit takes (8224 rows: 13.2, 12.8, 13.0 us with 3, 6, 10; 544 rows, merged
// through the workspace: 6.9, 6.9, 7.6): below it more CTAs only mean more parts to merge.
constexpr int kDecMinBlocks = 6;
constexpr int kDecMaxG = 8;            // query heads per KV head this kernel serves
constexpr int kDecPart = 4 + kHeadDim; // floats of a partial result of one query head: max, sum, 2 unused, accumulator
template <int kWarps> __host__ __device__ constexpr size_t dec_smem_bytes() { return (size_t)kWarps * kDecStages * kDecStage; }
static_assert(kDecMaxG * kDecPart * 4 <= kDecStages * kDecStage, "a warp's result takes the place of its ring");

struct DecodeArgs {
    int batch, hq, hkv, G, rows;
    int blocks_per_unit;               // blocks of a unit
    int splits;                        // CTAs that share a unit
    int cluster;                       // they are one cluster
    int two;                           // two CTAs per SM
    long long qs[2];                   // element strides of q: batch, head
    long long ks[3], vs[3];            // element strides of K and V: batch, head, row
    unsigned long long *arrived;       // [units] (call tag, count of CTAs that left their part), splits > 1; the call
                                       // leaves zeros, so that a captured call, whose tag is the same at every
                                       // replay, starts its count again
    float *part;                       // [units][splits][G][kDecPart], splits > 1
    float *out;                        // [batch][hq][D]
    uint32_t call_tag;                 // a nonzero value no other call on this workspace used
};

// 16 bytes global -> shared, zeros when `in` is false.
__device__ __forceinline__ void dec_copy16(uint32_t dst, const void *src, bool in)
{
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ uint4 lds16(uint32_t p)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(p));
    return v;
}

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
                 "{%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Two floats as a bf16 pair (first in the low half), and what the rounding left over.
__device__ __forceinline__ uint32_t take_bf16x2(float &x, float &y)
{
    uint32_t w;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(y), "f"(x));
    x -= __uint_as_float(w << 16);
    y -= __uint_as_float(w & 0xffff0000u);
    return w;
}

// The running softmax of one warp over bf16 rows, on the tensor cores.  The row operands come from
// registers as the loads deliver them: a dot product does not care about the order of its terms, so
// the eight consecutive dimensions of a 16-byte load stand for eight terms of the contraction in
// both operands.  Scores: S = Q K^T, query heads on the 16 rows of the product (repeated).  Values:
// O = P V with P in three bf16 parts (8 + 8 + 8 bits, the whole fp32 significand), each part on
// rows of the product of its own: for up to four heads, rows 0-3 / 4-7 / 8-11 hold the high, middle
// and low parts, so one product per 16 rows of V serves them all; five to eight heads take two.
// (With fp32 FMAs and shuffles instead the same loop needs about six times the instructions.)
template <int kG> struct DecodeTc {
    uint32_t q[4][4];                  // [32-dimension group]: this lane's query row, 16 bytes each
    float acc[16][4];
    float m, l;

    __device__ __forceinline__ void load_q(const __nv_bfloat16 *q0, long long stride, int G)
    {
        const int lane = threadIdx.x & 31, g = (lane >> 2) & (kG - 1), t = lane & 3;
        // (q may start at any element)
        const unsigned short *src = reinterpret_cast<const unsigned short *>(q0) + g * stride + t * 8;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int w = 0; w < 4; ++w)
                q[c][w] = g < G ? src[c * 32 + 2 * w] | (uint32_t)src[c * 32 + 2 * w + 1] << 16 : 0u;
    }
    __device__ __forceinline__ void clear()
    {
        m = kNegBig;
        l = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
    }
    // Where 16-byte piece c of row r of the block goes: the lanes that read together (rows 8n + g of
    // K, rows 2t + e of V) find their pieces in different banks.
    __device__ __forceinline__ static uint32_t k_at(int r, int c) { return r * 256 + ((c ^ ((r & 1) << 2)) << 4); }
    __device__ __forceinline__ static uint32_t v_at(int r, int c) { return r * 256 + ((c ^ (r & 6)) << 4); }
    // the block at shared address `st`, rows r0 .. r0+15 of the unit (those below `rows` count)
    __device__ __forceinline__ void block(uint32_t st, int r0, int rows, float scale)
    {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        float s[2][4];
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            s[n][0] = s[n][1] = s[n][2] = s[n][3] = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint4 k = lds16(st + k_at(n * 8 + g, c * 4 + t));
                const uint32_t a0[4] = {q[c][0], q[c][0], q[c][1], q[c][1]}, a1[4] = {q[c][2], q[c][2], q[c][3], q[c][3]};
                mma_bf16_16816(s[n], a0, k.x, k.y);
                mma_bf16_16816(s[n], a1, k.z, k.w);
            }
        }
        // this lane: head g % kG, rows 2t, 2t+1 of both halves
        float p[4];
        float mx = m;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = r0 + 2 * t + (e & 1) + (e >> 1) * 8;
            p[e] = r < rows ? s[e >> 1][e & 1] * scale : -INFINITY;
            mx = fmaxf(mx, p[e]);
        }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        if (__any_sync(0xffffffffu, mx > m)) {
            const float sc = exp2f(m - mx);
            l *= sc;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                acc[i][0] *= sc; acc[i][1] *= sc; acc[i][2] *= sc; acc[i][3] *= sc;
            }
            m = mx;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            p[e] = exp2f(p[e] - mx);
            l += p[e];
        }
        uint32_t part[3][2];           // [high, middle, low][row half]
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            part[x][0] = take_bf16x2(p[0], p[1]);
            part[x][1] = take_bf16x2(p[2], p[3]);
        }
        uint32_t a[4], a2[4];
        if constexpr (kG == 4) {
            const bool low4 = g < 4;
            a[0] = low4 ? part[0][0] : part[1][0];
            a[1] = low4 ? part[2][0] : 0u;
            a[2] = low4 ? part[0][1] : part[1][1];
            a[3] = low4 ? part[2][1] : 0u;
        } else {
            a[0] = part[0][0]; a[1] = part[1][0]; a[2] = part[0][1]; a[3] = part[1][1];
            a2[0] = part[2][0]; a2[1] = 0u; a2[2] = part[2][1]; a2[3] = 0u;
        }
        // column n of product i stands for dimension 8 n + i (i < 8), 64 + 8 n + i - 8 above
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint32_t w[4][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint4 v = lds16(st + kDecHalf + v_at(2 * t + (e & 1) + (e >> 1) * 8, c * 8 + g));
                w[e][0] = v.x; w[e][1] = v.y; w[e][2] = v.z; w[e][3] = v.w;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t sel = (i & 1) ? 0x7632u : 0x5410u;
                const uint32_t b0 = __byte_perm(w[0][i >> 1], w[1][i >> 1], sel);
                const uint32_t b1 = __byte_perm(w[2][i >> 1], w[3][i >> 1], sel);
                mma_bf16_16816(acc[c * 8 + i], a, b0, b1);
                if constexpr (kG == 8) mma_bf16_16816(acc[c * 8 + i], a2, b0, b1);
            }
        }
    }
    // (max, sum, accumulator) of the warp's rows -> dst [kG][kDecPart]
    __device__ __forceinline__ void store(float *dst)
    {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        l += __shfl_xor_sync(0xffffffffu, l, 1);
        l += __shfl_xor_sync(0xffffffffu, l, 2);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float x = acc[i][0] + acc[i][2], y = acc[i][1] + acc[i][3];
            if constexpr (kG == 4) {
                x += __shfl_xor_sync(0xffffffffu, x, 16);
                y += __shfl_xor_sync(0xffffffffu, y, 16);
            }
            if (g < kG) {
                const int d0 = (i >> 3) * 64 + 16 * t + (i & 7);
                dst[g * kDecPart + 4 + d0] = x;
                dst[g * kDecPart + 4 + d0 + 8] = y;
            }
        }
        if (t == 0 && g < kG) {
            dst[g * kDecPart] = m;
            dst[g * kDecPart + 1] = l;
        }
    }
};

// The same over fp32 rows, on the FMA pipe: half a warp takes kR rows at a time, a lane eight of
// the 128 dimensions; the 16 (row, head) sums are reduced over the half by exchanging halves of the
// set, which leaves one sum per lane.
template <int kG> struct DecodeSimt {
    static constexpr int kR = 16 / kG;
    const float *q;                    // [kG][128] in shared memory
    float acc[kG][8];
    float m, l;                        // of head lane % kG

    __device__ __forceinline__ void clear()
    {
        m = kNegBig;
        l = 0.f;
#pragma unroll
        for (int g = 0; g < kG; ++g)
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[g][e] = 0.f;
    }
    __device__ __forceinline__ static uint32_t k_at(int r, int c) { return r * 512 + (c << 4); }
    __device__ __forceinline__ static uint32_t v_at(int r, int c) { return r * 512 + (c << 4); }
    // this lane's dimensions: 4 sub .. and 64 + 4 sub ..
    __device__ __forceinline__ static void load_row(uint32_t p, float (&v)[8])
    {
        const uint4 a = lds16(p), b = lds16(p + 256);
        v[0] = __uint_as_float(a.x); v[1] = __uint_as_float(a.y); v[2] = __uint_as_float(a.z); v[3] = __uint_as_float(a.w);
        v[4] = __uint_as_float(b.x); v[5] = __uint_as_float(b.y); v[6] = __uint_as_float(b.z); v[7] = __uint_as_float(b.w);
    }
    __device__ __forceinline__ void block(uint32_t st, int r0, int rows, float scale)
    {
        const int lane = threadIdx.x & 31, half = lane >> 4, sub = lane & 15;
        constexpr int kHalfRows = dec_rows<float>() / 2;
#pragma unroll 1
        for (int step = 0; step < kHalfRows; step += kR) {
            const int rl = half * kHalfRows + step, rb = r0 + rl;
            float k[kR][8], v[kR][8];
#pragma unroll
            for (int r = 0; r < kR; ++r) {
                load_row(st + k_at(rl + r, sub), k[r]);
                load_row(st + kDecHalf + v_at(rl + r, sub), v[r]);
            }
            float s[16];               // [row][head]
#pragma unroll
            for (int g = 0; g < kG; ++g) {
                const float4 qa = *reinterpret_cast<const float4 *>(q + g * kHeadDim + 4 * sub);
                const float4 qb = *reinterpret_cast<const float4 *>(q + g * kHeadDim + 64 + 4 * sub);
#pragma unroll
                for (int r = 0; r < kR; ++r) {
                    float x = qa.x * k[r][0];
                    x = fmaf(qa.y, k[r][1], x); x = fmaf(qa.z, k[r][2], x); x = fmaf(qa.w, k[r][3], x);
                    x = fmaf(qb.x, k[r][4], x); x = fmaf(qb.y, k[r][5], x); x = fmaf(qb.z, k[r][6], x);
                    s[r * kG + g] = fmaf(qb.w, k[r][7], x);
                }
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                const bool up = (sub & o) != 0;
#pragma unroll
                for (int i = 0; i < o; ++i) {
                    const float give = up ? s[i] : s[i + o], keep = up ? s[i + o] : s[i];
                    s[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
            }
            // this lane: head sub % kG of row sub / kG
            const float x = rb + sub / kG < rows ? s[0] * scale : -INFINITY;
            float mx = fmaxf(m, x);
#pragma unroll
            for (int o = kG; o < 16; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (__any_sync(0xffffffffu, mx > m)) {
                const float sc = exp2f(m - mx);
                l *= sc;
#pragma unroll
                for (int g = 0; g < kG; ++g) {
                    const float sg = __shfl_sync(0xffffffffu, sc, g, 16);
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[g][e] *= sg;
                }
                m = mx;
            }
            const float p = exp2f(x - mx);
            l += p;
#pragma unroll
            for (int r = 0; r < kR; ++r)
#pragma unroll
                for (int g = 0; g < kG; ++g) {
                    const float pg = __shfl_sync(0xffffffffu, p, r * kG + g, 16);
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[g][e] = fmaf(pg, v[r][e], acc[g][e]);
                }
        }
    }
    __device__ __forceinline__ void store(float *dst)
    {
        const int lane = threadIdx.x & 31, sub = lane & 15;
        // the two halves of the warp, then the lanes that share a head
        const float mw = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
        const float sc = exp2f(m - mw);
        l *= sc;
#pragma unroll
        for (int o = kG; o < 32; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
#pragma unroll
        for (int g = 0; g < kG; ++g) {
            const float sg = __shfl_sync(0xffffffffu, sc, g, 16);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float x = acc[g][e] * sg;
                x += __shfl_xor_sync(0xffffffffu, x, 16);
                if (lane < 16) dst[g * kDecPart + 4 + (e >> 2) * 64 + 4 * sub + (e & 3)] = x;
            }
        }
        if (lane < kG) {
            dst[lane * kDecPart] = mw;
            dst[lane * kDecPart + 1] = l;
        }
    }
};

// Merges `n` partial results of one unit, part(i, w) = four floats from word w of the i-th
// [G][kDecPart], into `dst` (the output rows, normalised, or a partial result).  All threads of the
// CTA: kDecSplit groups of threads share the parts (four of them requested together), a thread of a group takes four
// outputs; the groups' shares meet in `x` [kDecSplit][G][kDecPart] of shared memory.
constexpr int kDecSplit = 3;
template <int kWarps, typename Part>
__device__ __forceinline__ void decode_merge(int n, int G, Part part, float *x, bool normalise, float *dst,
                                             int dst_stride)
{
    constexpr int kThreads = kWarps * 32, kWidth = kThreads / kDecSplit;
    const int grp = threadIdx.x / kWidth, t = threadIdx.x % kWidth;
    auto fold = [&](int i0, int step, int count, auto get, int g, int d4, float &m, float &l, float4 &o) {
        for (int i = i0; i < count; i += 4 * step) {
            float4 pm[4], po[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                pm[k] = make_float4(kNegBig, 0.f, 0.f, 0.f);
                po[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i + k * step < count) {
                    pm[k] = get(i + k * step, g * kDecPart);
                    po[k] = get(i + k * step, g * kDecPart + 4 + d4 * 4);
                }
            }
            const float mx = fmaxf(fmaxf(fmaxf(m, pm[0].x), fmaxf(pm[1].x, pm[2].x)), pm[3].x);
            const float sc = exp2f(m - mx);
            m = mx;
            l *= sc;
            o.x *= sc; o.y *= sc; o.z *= sc; o.w *= sc;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float w = exp2f(pm[k].x - mx);
                l = fmaf(pm[k].y, w, l);
                o.x = fmaf(po[k].x, w, o.x); o.y = fmaf(po[k].y, w, o.y);
                o.z = fmaf(po[k].z, w, o.z); o.w = fmaf(po[k].w, w, o.w);
            }
        }
    };
    for (int u = t; u < G * 32; u += kWidth) {
        const int g = u >> 5, d4 = u & 31;
        float m = kNegBig, l = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        fold(grp, kDecSplit, n, part, g, d4, m, l, o);
        float *xp = x + (grp * G + g) * kDecPart;
        *reinterpret_cast<float4 *>(xp + 4 + d4 * 4) = o;
        if (d4 == 0) *reinterpret_cast<float4 *>(xp) = make_float4(m, l, 0.f, 0.f);
    }
    __syncthreads();
    auto shared = [&](int i, int w) { return *reinterpret_cast<const float4 *>(x + i * G * kDecPart + w); };
    for (int u = threadIdx.x; u < G * 32; u += kThreads) {
        const int g = u >> 5, d4 = u & 31;
        float m = kNegBig, l = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        fold(0, 1, kDecSplit, shared, g, d4, m, l, o);
        if (normalise) {
            float *p = dst + g * dst_stride + d4 * 4;
            p[0] = o.x / l; p[1] = o.y / l; p[2] = o.z / l; p[3] = o.w / l;
        } else {
            float *p = dst + g * dst_stride;
            *reinterpret_cast<float4 *>(p + 4 + d4 * 4) = o;
            if (d4 == 0) *reinterpret_cast<float4 *>(p) = make_float4(m, l, 0.f, 0.f);
        }
    }
}

// kG: query heads per KV head rounded up to 4 or 8; kWarps 12, or 6 with two CTAs per SM.  grid (splits, units).
template <typename T, int kG, int kWarps>
__global__ void __launch_bounds__(kWarps * 32, kDecWarps / kWarps) decode_kernel(DecodeArgs a, const T *__restrict__ q,
                                                                const T *__restrict__ K,
                                                                const T *__restrict__ V)
{
    constexpr int kThreads = kWarps * 32;
    extern __shared__ __align__(128) uint8_t dec_smem[];         // [kWarps][kDecStages][kDecStage]
    __shared__ __align__(16) float s_x[kDecSplit * kG * kDecPart];
    float *const s_q = s_x;                                      // fp32 rows: the queries [kG][kHeadDim], until the merges
    __shared__ __align__(16) float s_part[kG * kDecPart];
    __shared__ int s_last;
    constexpr int kRows = dec_rows<T>(), kPieces = kHeadDim * (int)sizeof(T) / 16;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, G = a.G, unit = blockIdx.y;
    const int b = unit / a.hkv, h = unit % a.hkv;
    const int nb = a.blocks_per_unit;
    const int b0 = (int)((long long)nb * blockIdx.x / a.splits), b1 = (int)((long long)nb * (blockIdx.x + 1) / a.splits);
    const int n_warps = min(kWarps, b1 - b0);                 // warps with rows
    const float scale = rsqrtf((float)kHeadDim) * kLog2e;
    const T *qu = q + b * a.qs[0] + (long long)(h * G) * a.qs[1];
    const T *Ku = K + b * a.ks[0] + (long long)h * a.ks[1];
    const T *Vu = V + b * a.vs[0] + (long long)h * a.vs[1];
    float *out = a.out + ((long long)b * a.hq + h * G) * kHeadDim;
    uint8_t *ring = dec_smem + warp * (kDecStages * kDecStage);
    const uint32_t ring_s = static_cast<uint32_t>(__cvta_generic_to_shared(ring));
    pdl_wait();
    pdl_launch_dependents();
    if (a.splits > 1 && !a.cluster && tid == kThreads - 1) {
        // this call's tag into the unit's arrival word (nobody waits for it: a word that changes in
        // between has been tagged by another CTA of this call)
        const unsigned long long seen = *reinterpret_cast<volatile unsigned long long *>(a.arrived + unit);
        if ((seen >> 32) != a.call_tag) atomicCAS(a.arrived + unit, seen, (unsigned long long)a.call_tag << 32);
    }
    auto walk = [&](auto &run) {
        run.clear();
        auto request = [&](int i, int stage) {
            if (i < b1) {
                const int r0 = i * kRows;
                const uint32_t st = ring_s + stage * kDecStage;
#pragma unroll
                for (int x = lane; x < kRows * kPieces; x += 32) {
                    const int r = x / kPieces, c = x % kPieces;
                    const bool in = r0 + r < a.rows;
                    const long long row = in ? r0 + r : 0;
                    dec_copy16(st + run.k_at(r, c), Ku + row * a.ks[2] + c * (16 / (int)sizeof(T)), in);
                    dec_copy16(st + kDecHalf + run.v_at(r, c), Vu + row * a.vs[2] + c * (16 / (int)sizeof(T)), in);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        for (int k = 0; k < kDecStages; ++k) request(b0 + warp + k * kWarps, k);
        int stage = 0;
        for (int i = b0 + warp; i < b1; i += kWarps) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kDecStages - 1) : "memory");
            __syncwarp();
            run.block(ring_s + stage * kDecStage, i * kRows, a.rows, scale);
            __syncwarp();
            request(i + kDecStages * kWarps, stage);
            stage = stage + 1 == kDecStages ? 0 : stage + 1;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (warp < n_warps) run.store(reinterpret_cast<float *>(ring));
    };
    if constexpr (sizeof(T) == 2) {
        DecodeTc<kG> run;
        run.load_q(qu, a.qs[1], G);
        walk(run);
    } else {
        for (int i = tid; i < kG * kHeadDim; i += kThreads)
            s_q[i] = i / kHeadDim < G ? qu[(i / kHeadDim) * a.qs[1] + i % kHeadDim] : 0.f;
        __syncthreads();
        DecodeSimt<kG> run;
        run.q = s_q;
        walk(run);
    }
    __syncthreads();
    auto of_warp = [&](int i, int w) {
        return *reinterpret_cast<const float4 *>(dec_smem + i * (kDecStages * kDecStage) + w * 4);
    };
    if (a.splits == 1) {
        decode_merge<kWarps>(n_warps, G, of_warp, s_x, true, out, kHeadDim);
        return;
    }
    if (a.cluster) {
        // the parts stay in shared memory, where the first CTA of the unit's cluster reads them
        namespace cg = cooperative_groups;
        cg::cluster_group cl = cg::this_cluster();
        decode_merge<kWarps>(n_warps, G, of_warp, s_x, false, s_part, kDecPart);
        cl.sync();
        if (blockIdx.x == 0) {
            auto of_peer = [&](int i, int w) { return *reinterpret_cast<const float4 *>(cl.map_shared_rank(s_part, i) + w); };
            decode_merge<kWarps>(a.splits, G, of_peer, s_x, true, out, kHeadDim);
        }
        cl.sync();                                               // nobody leaves while its part is read
        return;
    }
    // this CTA's part goes to memory; the last CTA of the unit to get here merges them
    float *parts = a.part + (long long)unit * a.splits * G * kDecPart;
    decode_merge<kWarps>(n_warps, G, of_warp, s_x, false, parts + (long long)blockIdx.x * G * kDecPart, kDecPart);
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = (uint32_t)atomicAdd(a.arrived + unit, 1ull) + 1u == (uint32_t)a.splits;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        auto of_cta = [&](int i, int w) {
            return __ldcg(reinterpret_cast<const float4 *>(parts + (long long)i * G * kDecPart + w));
        };
        decode_merge<kWarps>(a.splits, G, of_cta, s_x, true, out, kHeadDim);
        // (every CTA of the unit has added, so nobody else touches the word any more)
        if (tid == 0) a.arrived[unit] = 0ull;
    }
}

}  // namespace graphkv
