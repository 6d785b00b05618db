// Step (I), SIMT fp32 path: SnapKV-style window-attention scores for any input dtype.
// Used for fp32 inputs (the tensor-core path takes bf16 only); kD = 64 or 128.  Two sweeps over the
// keys of a head: (1) per-row softmax statistics, (2) the column sums of the normalised probabilities.
//
// Bound: the FMA pipe (G*W*D multiply-adds per key and sweep, about 123 per clock and SM).  Both
// sweeps are a register-tiled product: tiles of 64 keys in shared memory, 64 (or 32) query rows at a
// time, four keys and four (two) rows per thread.  Every dot product keeps four partial sums (terms
// k mod 4), added pairwise at the end.  Measured on one B200 against one row or one key per thread
// (a chunk of 1024 keys per CTA), event-timed: one fp32 head of 544 keys 186 + 45 -> 11 + 13 us,
// eight heads of 4128 keys 315 + 134 -> 50 + 52 us.
#pragma once

#include "common.cuh"

namespace graphkv {

constexpr int kSimtThreads = 256;
constexpr int kSimtKeys = 64;       // keys per tile

// Row tile, key tile (rows of kD floats, four more apart so that 16-byte reads of consecutive rows hit
// different banks) and, for the second sweep, row constants and one partial sum per warp and key.
template <int kD> __host__ __device__ constexpr size_t simt_smem_bytes(int row_tile)
{
    return ((size_t)(row_tile + kSimtKeys) * (kD + 4) + 2 * row_tile + 8 * kSimtKeys) * sizeof(float);
}

// Key tiles [t0, t1) of CTA c of `ctas`.
__device__ __forceinline__ void simt_range(int n_keys, int ctas, int c, int *t0, int *t1)
{
    const int tiles = ceil_div(n_keys, kSimtKeys);
    *t0 = (int)((long long)tiles * c / ctas);
    *t1 = (int)((long long)tiles * (c + 1) / ctas);
}

// Query rows r0 .. r0 + kRT - 1 of the unit, scaled by log2(e) / sqrt(D), zeros past G*W.
template <typename T, int kD, int kRT>
__device__ __forceinline__ void simt_stage_rows(const Dims &d, const T *Q, int b, int h, int r0, float *dst)
{
    const float scale = rsqrtf((float)kD) * kLog2e;
    for (int i = threadIdx.x; i < kRT * (kD / 8); i += kSimtThreads) {
        const int r = i / (kD / 8), c = i % (kD / 8);
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (r0 + r < d.GW) {
            const int g = (r0 + r) / d.W, rw = (r0 + r) % d.W;
            load8(Q + b * d.qs[0] + (long long)(h * d.G + g) * d.qs[1] + rw * d.qs[2] + c * 8, v);
        }
        float4 *o = reinterpret_cast<float4 *>(dst + r * (kD + 4) + c * 8);
        o[0] = make_float4(v[0] * scale, v[1] * scale, v[2] * scale, v[3] * scale);
        o[1] = make_float4(v[4] * scale, v[5] * scale, v[6] * scale, v[7] * scale);
    }
}

// Keys j0 .. j0 + 63 of the head, zeros from `n` on.
template <typename T, int kD>
__device__ __forceinline__ void simt_stage_keys(const T *Kh, long long ks, int j0, int n, float *dst)
{
#pragma unroll 4
    for (int i = threadIdx.x; i < kSimtKeys * (kD / 8); i += kSimtThreads) {
        const int k = i / (kD / 8), c = i % (kD / 8);
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (j0 + k < n) load8(Kh + (long long)(j0 + k) * ks + c * 8, v);
        float4 *o = reinterpret_cast<float4 *>(dst + k * (kD + 4) + c * 8);
        o[0] = make_float4(v[0], v[1], v[2], v[3]);
        o[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
}

// out[i][e] = <row rg + 16 i, key kg + 16 e>.
template <int kD, int kR>
__device__ __forceinline__ void simt_dots(const float *rows, const float *keys, int rg, int kg, float (&out)[kR][4])
{
    float acc[kR][4][4];
#pragma unroll
    for (int i = 0; i < kR; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][e][0] = acc[i][e][1] = acc[i][e][2] = acc[i][e][3] = 0.f;
#pragma unroll 2
    for (int c = 0; c < kD / 4; ++c) {
        float4 q[kR], k[4];
#pragma unroll
        for (int i = 0; i < kR; ++i) q[i] = *reinterpret_cast<const float4 *>(rows + (rg + 16 * i) * (kD + 4) + 4 * c);
#pragma unroll
        for (int e = 0; e < 4; ++e) k[e] = *reinterpret_cast<const float4 *>(keys + (kg + 16 * e) * (kD + 4) + 4 * c);
#pragma unroll
        for (int i = 0; i < kR; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                acc[i][e][0] = fmaf(q[i].x, k[e].x, acc[i][e][0]);
                acc[i][e][1] = fmaf(q[i].y, k[e].y, acc[i][e][1]);
                acc[i][e][2] = fmaf(q[i].z, k[e].z, acc[i][e][2]);
                acc[i][e][3] = fmaf(q[i].w, k[e].w, acc[i][e][3]);
            }
    }
#pragma unroll
    for (int i = 0; i < kR; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) out[i][e] = (acc[i][e][0] + acc[i][e][1]) + (acc[i][e][2] + acc[i][e][3]);
}

// A row spread over a warp, four elements per lane, scaled to unit length.  (Written out in fused multiply-adds: every
// kernel that calls it gets the same bits.)
__device__ __forceinline__ void simt_unit_row(float (&v)[4])
{
    const float n2 = warp_sum(fmaf(v[3], v[3], fmaf(v[2], v[2], fmaf(v[1], v[1], v[0] * v[0]))));
    const float inv = 1.0f / fmaxf(sqrtf(n2), kNormEps);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] *= inv;
}

// Row statistics of the softmax, in the log2 domain: for query row r and the keys of one chunk,
// mx = max_j l2[r][j], z = sum_j 2^(l2[r][j] - mx), l2 = (q.k / sqrt(D)) * log2(e), over the keys
// row r may see (prefix keys and window keys N + r' with r' <= r).
// grid (n_chunks, units, row tiles), block kSimtThreads.  part [units][n_chunks][GW][2].
template <typename T, int kD, int kRT>
__global__ void __launch_bounds__(kSimtThreads) score_stats_simt(Dims d, const T *__restrict__ Q,
                                                                 const T *__restrict__ K,
                                                                 float *__restrict__ part, int n_chunks,
                                                                 int *status_word)
{
    extern __shared__ __align__(16) float sm[];
    constexpr int kR = kRT / 16;
    float *rows = sm, *keys = sm + kRT * (kD + 4);
    const int unit = blockIdx.y, b = unit / d.hkv, h = unit % d.hkv, r0 = blockIdx.z * kRT;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, kg = lane & 15, rg = warp * 2 + (lane >> 4);
    const T *Kh = K + b * d.ks[0] + (long long)h * d.ks[1];
    int t0, t1;
    simt_range(d.L, n_chunks, blockIdx.x, &t0, &t1);
    pdl_wait();
    pdl_launch_dependents();
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) *status_word = 0;
    simt_stage_rows<T, kD, kRT>(d, Q, b, h, r0, rows);
    float mx[kR], z[kR];
#pragma unroll
    for (int i = 0; i < kR; ++i) mx[i] = kNegBig, z[i] = 0.f;
    for (int t = t0; t < t1; ++t) {
        __syncthreads();
        simt_stage_keys<T, kD>(Kh, d.ks[2], t * kSimtKeys, d.L, keys);
        __syncthreads();
        float l2[kR][4];
        simt_dots<kD, kR>(rows, keys, rg, kg, l2);
#pragma unroll
        for (int i = 0; i < kR; ++i) {
            const int last = d.N + (r0 + rg + 16 * i) % d.W;          // last visible key of the row
            float m = mx[i];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (t * kSimtKeys + kg + 16 * e > last) l2[i][e] = -INFINITY;
                m = fmaxf(m, l2[i][e]);
            }
            z[i] *= exp2f(mx[i] - m);
            mx[i] = m;
#pragma unroll
            for (int e = 0; e < 4; ++e) z[i] += exp2f(l2[i][e] - m);
        }
    }
    // the 16 lanes that share a row
#pragma unroll
    for (int i = 0; i < kR; ++i) {
        float m = mx[i];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        float s = z[i] * exp2f(mx[i] - m);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const int r = r0 + rg + 16 * i;
        if (kg == 0 && r < d.GW)
            reinterpret_cast<float2 *>(part)[((long long)unit * n_chunks + blockIdx.x) * d.GW + r] = make_float2(m, s);
    }
}

// Second sweep: a[j] = sum_r 2^(l2[r][j] - mx_r) / Z_r for the prefix keys j of one head.
// grid (CTAs per unit, units), block kSimtThreads; n_chunks: chunks of the first sweep.
template <typename T, int kD, int kRT>
__global__ void __launch_bounds__(kSimtThreads) score_emit_simt(Dims d, const T *__restrict__ Q,
                                                                const T *__restrict__ K,
                                                                const float *__restrict__ part, int n_chunks,
                                                                float *__restrict__ a_out)
{
    extern __shared__ __align__(16) float sm[];
    constexpr int kR = kRT / 16;
    float *rows = sm, *keys = sm + kRT * (kD + 4);
    float *row_mx = keys + kSimtKeys * (kD + 4);         // [kRT]
    float *row_w = row_mx + kRT;                         // [kRT] 1 / Z_r, 0 past G*W
    float *sums = row_w + kRT;                           // [8 warps][kSimtKeys]
    const int unit = blockIdx.y, b = unit / d.hkv, h = unit % d.hkv;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, kg = lane & 15, rg = warp * 2 + (lane >> 4);
    const T *Kh = K + b * d.ks[0] + (long long)h * d.ks[1];
    const float2 *pu = reinterpret_cast<const float2 *>(part) + (long long)unit * n_chunks * d.GW;
    int t0, t1;
    simt_range(d.N, gridDim.x, blockIdx.x, &t0, &t1);
    const int row_tiles = ceil_div(d.GW, kRT);
    for (int t = t0; t < t1; ++t) {
        if (t > t0) __syncthreads();
        simt_stage_keys<T, kD>(Kh, d.ks[2], t * kSimtKeys, d.N, keys);
        if (t == t0) {                                   // (keys and queries are inputs of the call)
            pdl_wait();
            pdl_launch_dependents();
        }
        float a[4] = {0.f, 0.f, 0.f, 0.f};
        for (int rt = 0; rt < row_tiles; ++rt) {
            if (rt > 0) __syncthreads();
            if (row_tiles > 1 || t == t0) {
                simt_stage_rows<T, kD, kRT>(d, Q, b, h, rt * kRT, rows);
                // four threads merge a row's chunks
                constexpr int kTpr = 4;
                const int rl = threadIdx.x / kTpr, r = rt * kRT + rl, sub = threadIdx.x % kTpr;
                if (rl < kRT) {
                    float mx = kNegBig, z = 0.f;
                    for (int q0 = sub; q0 < n_chunks; q0 += 8 * kTpr) {
                        float2 v[8];
                        float mn = mx;
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            v[k] = q0 + k * kTpr < n_chunks && r < d.GW ? pu[(long long)(q0 + k * kTpr) * d.GW + r]
                                                                        : make_float2(kNegBig, 0.f);
                            mn = fmaxf(mn, v[k].x);
                        }
                        z *= exp2f(mx - mn);
#pragma unroll
                        for (int k = 0; k < 8; ++k) z = fmaf(v[k].y, exp2f(v[k].x - mn), z);
                        mx = mn;
                    }
                    float m = mx;
                    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
                    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
                    z *= exp2f(mx - m);
                    z += __shfl_xor_sync(0xffffffffu, z, 1);
                    z += __shfl_xor_sync(0xffffffffu, z, 2);
                    if (sub == 0) {
                        row_mx[rl] = r < d.GW ? m : 0.f;
                        row_w[rl] = r < d.GW ? 1.0f / z : 0.f;
                    }
                }
            }
            __syncthreads();
            float l2[kR][4];
            simt_dots<kD, kR>(rows, keys, rg, kg, l2);
#pragma unroll
            for (int i = 0; i < kR; ++i) {
                const float m = row_mx[rg + 16 * i], w = row_w[rg + 16 * i];
#pragma unroll
                for (int e = 0; e < 4; ++e) a[e] = fmaf(exp2f(l2[i][e] - m), w, a[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            a[e] += __shfl_xor_sync(0xffffffffu, a[e], 16);
            if (lane < 16) sums[warp * kSimtKeys + kg + 16 * e] = a[e];
        }
        __syncthreads();
        const int j = t * kSimtKeys + threadIdx.x;
        if (threadIdx.x < kSimtKeys && j < d.N) {
            float x = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) x += sums[w * kSimtKeys + threadIdx.x];
            a_out[(long long)unit * d.N + j] = x;
        }
    }
}

// 1-D pooling, stride 1, same length: the maximum over the positions inside [0,N), or (avg) the
// sum over them divided by kp (zeros outside the row).  grid (ceil(N/256), units), block 256.
__global__ void pool_max_kernel(int N, int kp, int avg, const float *__restrict__ a,
                                float *__restrict__ s)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    const float *row = a + (long long)blockIdx.y * N;
    const int half = (kp - 1) / 2;
    const int lo = max(j - half, 0), hi = min(j + half, N - 1);
    float best = row[lo];
    if (avg) {
        for (int t = lo + 1; t <= hi; ++t) best += row[t];
        best /= (float)kp;
    } else {
        for (int t = lo + 1; t <= hi; ++t) best = fmaxf(best, row[t]);
    }
    s[(long long)blockIdx.y * N + j] = best;
}

}  // namespace graphkv
