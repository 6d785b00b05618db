// Steps (II)+(III): edges of the source nodes (Eq. 1, Algorithm 1) and the decay rounds
// (Eq. 3-5, Algorithm 2).  SIMT fp32 similarity path for any input dtype.
#pragma once

#include "score_simt.cuh"

namespace graphkv {

constexpr int kSimRows = 16;       // sources per pass over a key tile

// e[a][j] = <k_src[a], k_j> / (max(|k_src[a]|, eps) * max(|k_j|, eps)), clipped to [-1, 1],
// for all sources a of the head and every prefix key j.  Entry j = src[a] is written too; the
// neighbour selection excludes it by index.
// grid (ceil(N / kSimtKeys), units), block kSimtThreads.  sims [units][K_src][N].
// The sources' vectors come from tensor S (strides ss), the swept vectors from tensor K (strides
// ks): the same tensor for Eq. 1, keys and values for the other edge kinds.
// A tile of 64 keys per CTA in shared memory, 16 sources at a time against it, four keys of one
// source per thread (one fp32 head of 512 keys, 8 sources, event-timed on one B200: 25 -> 11 us against a
// whole key in each thread's registers).
struct Strides3 {
    long long v[3];
};

template <int kD> __host__ __device__ constexpr size_t sim_simt_smem_bytes()
{
    return ((size_t)(kSimRows + kSimtKeys) * (kD + 4) + kSimtKeys) * sizeof(float);
}

template <typename T, int kD>
__global__ void __launch_bounds__(kSimtThreads) similarity_simt(Dims d, const T *__restrict__ S, Strides3 ss,
                                                              const T *__restrict__ K, Strides3 ks,
                                                              const int *__restrict__ src,
                                                              float *__restrict__ sims)
{
    extern __shared__ __align__(16) float sm[];
    float *rows = sm;                                    // [kSimRows][kD + 4] unit-norm source keys
    float *keys = rows + kSimRows * (kD + 4);            // [kSimtKeys][kD + 4]
    float *inv_norm = keys + kSimtKeys * (kD + 4);       // [kSimtKeys]
    const int unit = blockIdx.y, b = unit / d.hkv, h = unit % d.hkv;
    const T *Kh = K + b * ks.v[0] + (long long)h * ks.v[1];
    const T *Sh = S + b * ss.v[0] + (long long)h * ss.v[1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, kg = lane & 15, rg = warp * 2 + (lane >> 4);
    const int j0 = blockIdx.x * kSimtKeys;
    simt_stage_keys<T, kD>(Kh, ks.v[2], j0, d.N, keys);      // (inputs of the call)
    pdl_wait();
    pdl_launch_dependents();
    for (int a0 = 0; a0 < d.K_src; a0 += kSimRows) {
        const int na = min(kSimRows, d.K_src - a0);
        if (a0 > 0) __syncthreads();
        // one warp per source row: load, normalise, store
        for (int a = warp; a < kSimRows; a += kSimtThreads / 32) {
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (a < na && lane * 4 < kD) {               // (a row of 64 elements takes the first 16 lanes)
                const int i = src[(long long)unit * d.K_src + a0 + a];
                const T *kp = Sh + (long long)i * ss.v[2] + lane * 4;
                if constexpr (sizeof(T) == 2) {
                    const uint2 raw = *reinterpret_cast<const uint2 *>(kp);
                    v[0] = __uint_as_float(raw.x << 16); v[1] = __uint_as_float(raw.x & 0xffff0000u);
                    v[2] = __uint_as_float(raw.y << 16); v[3] = __uint_as_float(raw.y & 0xffff0000u);
                } else {
                    const float4 raw = *reinterpret_cast<const float4 *>(kp);
                    v[0] = raw.x; v[1] = raw.y; v[2] = raw.z; v[3] = raw.w;
                }
            }
            simt_unit_row(v);
            if (lane * 4 < kD) *reinterpret_cast<float4 *>(rows + a * (kD + 4) + lane * 4) = make_float4(v[0], v[1], v[2], v[3]);
        }
        __syncthreads();
        if (a0 == 0) {
            if (threadIdx.x < kSimtKeys) {
                const float4 *k4 = reinterpret_cast<const float4 *>(keys + threadIdx.x * (kD + 4));
                float n2 = 0.f;
#pragma unroll 8
                for (int c = 0; c < kD / 4; ++c) {
                    const float4 v = k4[c];
                    n2 = fmaf(v.x, v.x, n2); n2 = fmaf(v.y, v.y, n2); n2 = fmaf(v.z, v.z, n2); n2 = fmaf(v.w, v.w, n2);
                }
                inv_norm[threadIdx.x] = 1.0f / fmaxf(sqrtf(n2), kNormEps);
            }
            __syncthreads();
        }
        float dot[1][4];
        simt_dots<kD, 1>(rows, keys, rg, kg, dot);
        if (rg < na) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int k = kg + 16 * e;
                const float c = fminf(fmaxf(dot[0][e] * inv_norm[k], -1.0f), 1.0f);
                if (j0 + k < d.N) sims[((long long)unit * d.K_src + a0 + rg) * d.N + j0 + k] = c;
            }
        }
    }
}

// T rounds of s_j <- s_j * (1 - lambda * max(e_ij, 0)) over the fixed neighbour lists.
// Sources are applied one after another (threads span one source's m distinct neighbours), so
// overlapping neighbourhoods multiply deterministically.  grid units, block 256.
// nbr_idx / nbr_e [units][K_src][m].
__global__ void decay_rounds_kernel(Dims d, const int *__restrict__ nbr_idx,
                                    const float *__restrict__ nbr_e, float *__restrict__ scores)
{
    const int unit = blockIdx.x;
    float *s = scores + (long long)unit * d.N;
    const int *ni = nbr_idx + (long long)unit * d.K_src * d.m;
    const float *ne = nbr_e + (long long)unit * d.K_src * d.m;
    for (int t = 0; t < d.T; ++t) {
        for (int a = 0; a < d.K_src; ++a) {
            for (int u = threadIdx.x; u < d.m; u += blockDim.x) {
                const int j = ni[a * d.m + u];
                s[j] = d.signal == GRAPHKV_SIGNAL_EVICT ? -INFINITY
                                                        : s[j] * signal_factor(ne[a * d.m + u], d.lambda, 1, d.signal);
            }
            __syncthreads();
        }
    }
}

}  // namespace graphkv
