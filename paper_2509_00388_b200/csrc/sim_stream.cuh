// Steps (II)+(III), first half, for many sources or long rows: the edges of all sources of a head with a chunk of its
// keys in one sweep, compared with bounds as they come out of tensor memory.
//
// similarity_tc keeps a chunk's whole edge block in tensor memory until bounds for the chunk are known, so its loads stop
// for half of its time, and a head with more than 64 sources is swept several times.  Here the bounds come first: a
// sample of the row's tiles (similarity_tc in its sampling form, a cluster of CTAs per 32 sources) gives per source a
// value that at least m of its edges reach.  With 1/8 of the row sampled about 9 m edges of the row reach it.  The sweep
// then streams: up to 256 sources are the columns of one product per key tile, two to four accumulators rotate, eight warps take
// the keys' norms, and 16 epilogue warps (thread = key) push the edges that reach their source's bound into queues of
// their own, with predicated stores and no branch, and list them from there, by source and chunk.
// A source with more than kCandCap such edges in a chunk (a run of near-duplicates that the sample missed, ties) is swept once more
// with the chunk's edges resident and searched exactly (rework below).
//
// Bound: the comparisons.  128 keys x 160 sources take 1.8 us per SM, of which the products are 0.35 and the arrival of the tile
// 0.4; per 32 sources a warp spends about 400 issue slots on the comparisons of its 32 keys and on the edges found.  At 32
// sources a tile takes 0.9 us, near the 0.72 at which HBM delivers it.  154 sources at 32K x 8 heads: 94.5 us in five
// sweeps of similarity_tc -> 23 for the bounds and 43 here; 32 sources at 128K x 32 heads 308 -> 27 and 212.  Tried: setp and a predicated
// store per edge instead of the sums of bits (the same time), queues listed at four instead of nine edges (2 us more), four
// warps for the norms (they held up the sweep of 32 sources).
//
// The lists have the form similarity_tc leaves, and together hold every member of the head-wide top-m.
//
#pragma once

#include "sim_tc.cuh"

namespace graphkv {
namespace tc {

constexpr int kStreamThreads = 64 + 256 + 512;          // producer, MMA, 8 norm warps, 16 epilogue warps
constexpr int kStreamMaxSources = 256;
constexpr int kStreamMaxTiles = 32;                     // tiles per chunk: rework holds 16 sources' edges with them
// Edges per thread's queue, and how many make it be listed: a listing takes four edges of each thread at a time, so the
// fuller the queues the better.
__host__ __device__ inline int stream_queue(int np) { return np <= 160 ? 12 : 8; }

struct SimStreamArgs {
    Dims d;
    const __nv_bfloat16 *S;   // tensor the sources' vectors are read from, its element strides: batch, head, token
    long long ss[3];
    const int *src;           // [units][K_src] source positions
    const float *tau;         // [units][K_src] values that m edges of the source reach
    Cand *cand;               // [units][K_src][chunks][kCandCap]; unused slots hold e = kCandEmpty
    uint32_t *cand_hist;      // [units][K_src][kCandBins] edges of the row per cosine bin (zeroed before)
    int *status;
    int chunks;               // CTAs per unit
    int n_tiles;              // 128-key tiles per unit
    int np;                   // sources per sweep, padded to a multiple of 32
    int stages;
    int wait_prior;
    long long wait_cycles;
};

// Dynamic shared memory, byte offsets from a 1024-byte aligned base.
struct StreamLayout {
    uint32_t stage, queue, inv_norm, src_pos, src_inv, theta, cnt, flooded, bars, bytes;
};
template <int kD> __host__ __device__ inline StreamLayout stream_layout(int np, int stages)
{
    StreamLayout l;
    l.stage = np * 2 * kD;                               // source keys | key tiles in flight
    l.queue = l.stage + stages * tile_bytes<kD>();       // [stream_queue][512]
    l.inv_norm = l.queue + stream_queue(np) * 512 * 8;   // [kStreamMaxTiles][128]
    l.src_pos = l.inv_norm + kStreamMaxTiles * 128 * 4;
    l.src_inv = l.src_pos + np * 4;
    l.theta = l.src_inv + np * 4;
    l.cnt = l.theta + np * 4;
    l.flooded = l.cnt + np * 4;                          // [np] sources to rework
    l.bars = l.flooded + np * 4;                         // full[8], empty[8], tfull[4], tempty[4], done, words, norms[kStreamMaxTiles]
    l.bytes = l.bars + 28 * 8 + 32 + kStreamMaxTiles * 8 + 1024;
    return l;
}
__host__ __device__ inline int stream_bufs(int np) { return np <= 128 ? 4 : np <= 160 ? 3 : 2; }

// One edge's place in the list of (source, chunk), and the edge into it where there is one.
template <int kN>
__device__ __forceinline__ void stream_list(const int (&c)[kN], const int (&key)[kN], const float (&x)[kN], const int *src_pos, int j0,
                                            int *cnt, Cand *cand, long long source_stride, uint32_t *hist)
{
    int at[kN];
#pragma unroll
    for (int q = 0; q < kN; ++q) {
        at[q] = kCandCap;
        if (c[q] >= 0 && j0 + key[q] != src_pos[c[q]] && !list_overflowed(cnt, c[q])) at[q] = atomicAdd(cnt + c[q], 1);
    }
#pragma unroll
    for (int q = 0; q < kN; ++q)
        if (at[q] < kCandCap) {
            const float e = clamped_edge(x[q]);
            cand[c[q] * source_stride + at[q]] = Cand{e, j0 + key[q]};
            atomicAdd(hist + c[q] * kCandBins + cand_bin(e), 1u);
        }
}

// grid (chunks, units, sweeps of np sources).
template <int kD>
__global__ void __launch_bounds__(kStreamThreads, 1)
sim_stream_tc(const __grid_constant__ CUtensorMap tmK, SimStreamArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const Dims &d = a.d;
    const long long lim = a.wait_cycles;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base - smem_u32(smem_raw));
    const int np = a.np, S = a.stages, bufs = stream_bufs(np), n_slices = np / 32;
    const StreamLayout l = stream_layout<kD>(np, S);
    float *inv_norm = reinterpret_cast<float *>(gen + l.inv_norm);
    int *src_pos = reinterpret_cast<int *>(gen + l.src_pos);
    float *src_inv = reinterpret_cast<float *>(gen + l.src_inv), *theta = reinterpret_cast<float *>(gen + l.theta);
    int *cnt = reinterpret_cast<int *>(gen + l.cnt), *flooded = reinterpret_cast<int *>(gen + l.flooded);
    const uint32_t s_full0 = base + l.bars, s_empty0 = s_full0 + 64, s_tfull0 = s_empty0 + 64, s_tempty0 = s_tfull0 + 32,
                   s_done = s_tempty0 + 32, s_tmem = s_done + 8, s_norms0 = s_full0 + 28 * 8 + 32;
    int *words = reinterpret_cast<int *>(gen + l.bars + 28 * 8);        // [0] tensor memory's base (s_tmem lies before), [1] failed, [2] flooded sources
    PhaseClock pc(threadIdx.x == 320);
    pc.mark();
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int unit = blockIdx.y, b = unit / d.hkv, h = unit % d.hkv, chunk = blockIdx.x;
    int t0, t1;
    tile_range(a.n_tiles, a.chunks, chunk, &t0, &t1);
    const int n_local = t1 - t0, j0 = t0 * kTileKeys;
    const __nv_bfloat16 *src_rows = a.S + b * a.ss[0] + (long long)h * a.ss[1];
    const int src0 = blockIdx.z * np, n_src = min(np, d.K_src - src0);
    const long long source0 = (long long)unit * d.K_src + src0, source_stride = (long long)a.chunks * kCandCap;
    Cand *cand = a.cand + (source0 * a.chunks + chunk) * kCandCap;      // source c's list of this chunk at c * source_stride
    uint32_t *hist = a.cand_hist + source0 * kCandBins;

    int n_ahead = 0;
    if (threadIdx.x == 0) {
        for (int i = 0; i < S; ++i) {
            mbar_init(s_full0 + 8 * i, 1);
            mbar_init(s_empty0 + 8 * i, 1 + 4);                         // the MMA's commit and the norm warps
        }
        for (int i = 0; i < bufs; ++i) {
            mbar_init(s_tfull0 + 8 * i, 1);
            mbar_init(s_tempty0 + 8 * i, 4 * n_slices);                 // a warp per slice of 32 sources and lane quarter
        }
        for (int i = 0; i < n_local; ++i) mbar_init(s_norms0 + 8 * i, 4);
        mbar_init(s_done, 1);
        words[1] = words[2] = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmK);
        // (keys are an input of the call: no wait for the kernels before)
        n_ahead = min(S, n_local);
        for (int i = 0; i < n_ahead; ++i)
            tma_load_tile<kD>(base + l.stage + i * tile_bytes<kD>(), &tmK, s_full0 + 8 * i, (t0 + i) * kTileKeys, h, b);
    }
    if (warp == 1) {
        tmem_alloc(s_tmem, 512);
        tmem_relinquish();
    }
    pc.mark();
    if (a.wait_prior) pdl_wait();
    pdl_launch_dependents();
    pc.mark();
    // rows of sources -> swizzled operand of n rows, `of(r)`: the source of row r or -1
    constexpr int kPieces = kD / 8;
    auto stage_sources = [&](int n, auto of, auto put) {
        constexpr int kU = 3;                            // pieces in flight per thread: a position, then the row's piece
        for (int i0 = threadIdx.x; i0 - (int)threadIdx.x < n * kPieces; i0 += kU * kStreamThreads) {
            int pos[kU];
            uint4 v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int i = i0 + u * kStreamThreads, c = i < n * kPieces ? of(i / kPieces) : -1;
                pos[u] = c >= 0 ? a.src[source0 + c] : -1;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                v[u] = make_uint4(0, 0, 0, 0);
                if (pos[u] >= 0) v[u] = *reinterpret_cast<const uint4 *>(src_rows + (long long)pos[u] * a.ss[2] + (i0 + u * kStreamThreads) % kPieces * 8);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int i = i0 + u * kStreamThreads, r = i / kPieces, c16 = i % kPieces;
                const bool in = i < n * kPieces;
                if (in) *reinterpret_cast<uint4 *>(gen + sw128_offset(n, r, c16)) = v[u];
                const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
                float n2 = 0.f;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float lo = __uint_as_float(w[q] << 16), hi = __uint_as_float(w[q] & 0xffff0000u);
                    n2 = fmaf(lo, lo, fmaf(hi, hi, n2));
                }
#pragma unroll
                for (int o = kPieces / 2; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
                if (in && c16 == 0) put(r, pos[u], n2);
            }
        }
    };
    stage_sources(np, [&](int r) { return r < n_src ? r : -1; }, [&](int r, int pos, float n2) {
        const float norm = fmaxf(sqrtf(n2), kNormEps);
        src_pos[r] = pos;
        src_inv[r] = 1.0f / norm;
        cnt[r] = 0;
        // the bound brought to the scale of dot / |k_j|, lowered so that no edge whose cosine rounds up to it is missed
        // (kept negated; an infinite bound would make a difference of infinities)
        const float q = r < n_src ? (fmaxf(__ldcg(a.tau + source0 + r), -2.0f) - 2.4e-7f) * norm : 3.0e38f;
        theta[r] = -(q - fabsf(q) * 3.6e-7f - 1e-30f);
    });
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(gen + (s_tmem - base)), 0);
    bool ok = true;
    pc.mark();

    const int ew = warp - 10, quad = warp & 3, et = (int)threadIdx.x - 320;
    const int key_lane = quad * 32 + lane;
    if (warp == 0) {
        if (lane == 0) {
            int issued = n_ahead;
            for (int i = n_ahead; i < n_local; ++i) {
                const int st = i % S, ph = (i / S) & 1;
                if (!mbar_wait(s_empty0 + 8 * st, ph ^ 1, lim)) { ok = false; break; }
                tma_load_tile<kD>(base + l.stage + st * tile_bytes<kD>(), &tmK, s_full0 + 8 * st, (t0 + i) * kTileKeys, h, b);
                ++issued;
            }
            // the last copies have landed before the ring's place is used again or the CTA exits
            for (int i = max(0, issued - S); i < issued; ++i) ok = mbar_wait(s_full0 + 8 * (i % S), (i / S) & 1, lim) && ok;
        }
    } else if (warp == 1) {
        const uint32_t idesc = umma_idesc_bf16(128, np), src_lo = umma_desc_lo(base), ring_lo = umma_desc_lo(base + l.stage);
        int st = 0, buf = 0;
        uint32_t ph = 0u, bph = 1u;
        for (int i = 0; i < n_local; ++i) {
            ok = mbar_wait(s_tempty0 + 8 * buf, bph, lim) && mbar_wait(s_full0 + 8 * st, ph, lim);
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            tc_fence_after();
            if (elect_one()) {
                umma_tile<kD>(tmem_base + buf * np, ring_lo + st * (tile_bytes<kD>() >> 4), kHalfBytes >> 4, src_lo, np * 128 >> 4, idesc);
                umma_commit(s_empty0 + 8 * st);
                umma_commit(s_tfull0 + 8 * buf);
            }
            __syncwarp();
            if (++st == S) st = 0, ph ^= 1u;
            if (++buf == bufs) buf = 0, bph ^= 1u;
        }
    } else if (warp < 10) {
        // ---- norms of the keys, four warps a tile ----
        for (int i = (warp - 2) >> 2; i < n_local && ok; i += 2) {
            const int st = i % S;
            // (The norms of the tile before in this stage first: with S odd the other group took it, so this group's view of
            // the stage's barrier skips phases, and the parity of the phase it waits for could be an older one's.)
            ok = __all_sync(0xffffffffu, (i < S || mbar_wait(s_norms0 + 8 * (i - S), 0, lim)) && mbar_wait(s_full0 + 8 * st, (i / S) & 1, lim));
            if (!ok) break;
            const uint8_t *tile = gen + l.stage + st * tile_bytes<kD>();
            uint64_t n2 = 0ull;                                         // (the same two sums as elsewhere, packed)
#pragma unroll
            for (int c16 = 0; c16 < kPieces; ++c16) {
                const uint4 piece = *reinterpret_cast<const uint4 *>(tile + sw128_offset(128, key_lane, c16));
                const uint32_t w[4] = {piece.x, piece.y, piece.z, piece.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint64_t v = pack2(__uint_as_float(w[q] << 16), __uint_as_float(w[q] & 0xffff0000u));
                    n2 = fma2(v, v, n2);
                }
            }
            float n0, n1;
            unpack2(n2, n0, n1);
            // (a key past the end of the row: NaN, which no comparison takes)
            inv_norm[i * kTileKeys + key_lane] =
                j0 + i * kTileKeys + key_lane < d.N ? 1.0f / fmaxf(sqrtf(n0 + n1), kNormEps) : __int_as_float(0x7fc00000);
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(s_empty0 + 8 * st);
                mbar_arrive(s_norms0 + 8 * i);
            }
        }
    } else {
        // ---- epilogue: thread = key; the sets of four warps take the slices of 32 sources of all tiles in turn ----
        const int set = ew >> 2;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16);
        uint2 *const q0 = reinterpret_cast<uint2 *>(gen + l.queue) + et;
        constexpr uint32_t kStep = 512 * sizeof(uint2);
        const int queue = stream_queue(np);
        const uint32_t q_first = smem_u32(q0), q_last = q_first + (queue - 1) * kStep;
        uint32_t qa = q_first;
        auto flush = [&]() {
            const int queued = static_cast<int>((qa - q_first) / kStep);
#pragma unroll 1
            for (int k = 0; k < queued; k += 4) {
                int c[4], key[4];
                float x[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint2 en = q0[min(k + q, queue - 1) * 512];
                    const bool in = k + q < queued;
                    c[q] = in ? (int)(en.y >> 16) : -1;
                    key[q] = (int)(en.y & 0xffffu);
                    x[q] = __uint_as_float(en.x) * src_inv[max(c[q], 0)];
                }
                stream_list<4>(c, key, x, src_pos, j0, cnt, cand, source_stride, hist);
            }
            qa = q_first;
            __syncwarp();
        };
        int i = set / n_slices, sl = set % n_slices;
        while (i < n_local) {
            const int buf = i % bufs, col0 = sl * 32;
            ok = __all_sync(0xffffffffu, mbar_wait(s_tfull0 + 8 * buf, (i / bufs) & 1, lim));
            if (!ok) break;
            tc_fence_after();
            uint32_t raw[32];
            tmem_ld32_issue(lane_addr + buf * np + col0, raw);
            ok = __all_sync(0xffffffffu, mbar_wait(s_norms0 + 8 * i, 0, lim));
            const int key = i * kTileKeys + key_lane;
            const float inv = inv_norm[key];
            const uint64_t inv2 = pack2(inv, inv);
            const uint32_t id0 = ((uint32_t)col0 << 16) | (uint32_t)key;
            tmem_ld_fence(raw);
            if (!ok) break;
            const uint32_t before = qa;
            // The slice's edges that reach their bounds, a bit each.  All on the FMA pipe (the others take twice as long per
            // instruction): t = x - theta, s = 1 where t > 0 (saturated after scaling, 0 for NaN), and the sum of s 2^c
            // on top of 2^23 has the bits where an integer would have them.
            uint32_t mask = 0u;
#pragma unroll
            for (int c16 = 0; c16 < 32; c16 += 16) {
                float bits = 8388608.0f;
#pragma unroll
                for (int c4 = c16; c4 < c16 + 16; c4 += 4) {
                    const ulonglong2 th = *reinterpret_cast<const ulonglong2 *>(theta + col0 + c4);       // -theta
                    const uint64_t t01 = fma2(pack2(__uint_as_float(raw[c4]), __uint_as_float(raw[c4 + 1])), inv2, th.x);
                    const uint64_t t23 = fma2(pack2(__uint_as_float(raw[c4 + 2]), __uint_as_float(raw[c4 + 3])), inv2, th.y);
                    float t[4];
                    unpack2(t01, t[0], t[1]);
                    unpack2(t23, t[2], t[3]);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float one;
                        asm("mul.rn.ftz.sat.f32 %0, %1, %2;" : "=f"(one) : "f"(t[q]), "f"(8.50705917e37f));       // 2^126
                        bits = fmaf(one, (float)(1u << (c4 - c16 + q)), bits);
                    }
                }
                mask |= (__float_as_uint(bits) & 0xffffu) << c16;
            }
            const uint32_t some = __reduce_or_sync(0xffffffffu, mask);
#pragma unroll
            for (int c4 = 0; c4 < 32; c4 += 4) {
                if (!(some >> c4 & 0xfu)) continue;
#pragma unroll
                for (int q = c4; q < c4 + 4; ++q)
                    // (the store and the count under one predicate; the last place takes what does not fit)
                    asm volatile(
                        "{\n\t.reg .pred p;\n\t.reg .u32 a;\n\t"
                        "setp.ne.u32 p, %3, 0;\n\t"
                        "min.u32 a, %0, %4;\n\t"
                        "@p st.shared.v2.b32 [a], {%1, %2};\n\t"
                        "@p add.u32 %0, %0, %5;\n\t}"
                        : "+r"(qa)
                        : "f"(__uint_as_float(raw[q]) * inv), "r"(id0 + ((uint32_t)q << 16)), "r"(mask & (1u << q)), "r"(q_last), "r"(kStep)
                        : "memory");
            }
            const uint32_t fill = __reduce_max_sync(0xffffffffu, qa - q_first);
            if (fill > queue * kStep) {
                // a key close to many sources: what the queues held before this slice, then the slice without queues
                qa = before;
                flush();
#pragma unroll 1
                for (int c0 = col0; c0 < col0 + 32 && c0 < n_src; c0 += 8) {
                    uint32_t r[8];
                    __syncwarp();
                    tmem_ld8_issue(lane_addr + buf * np + c0, r);
                    tmem_ld_fence(r);
                    int c[8], keys[8];
                    float x[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float v = __uint_as_float(r[q]) * inv;
                        c[q] = fmaf(__uint_as_float(r[q]), inv, theta[c0 + q]) > 0.f ? c0 + q : -1;
                        keys[q] = key;
                        x[q] = v * src_inv[c0 + q];
                    }
                    stream_list<8>(c, keys, x, src_pos, j0, cnt, cand, source_stride, hist);
                }
                __syncwarp();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(s_tempty0 + 8 * buf);
            if (fill > (queue - 4) * kStep && fill <= queue * kStep) flush();
            for (sl += 4; sl >= n_slices; sl -= n_slices) ++i;
        }
        flush();
        pc.mark();
    }
    if (!ok && lane == 0) words[1] = 1;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const bool all_ok = *reinterpret_cast<volatile int *>(words + 1) == 0;
    pc.mark();

    // ---- unused slots marked empty; the sources with more edges than slots gathered ----
    for (int idx = threadIdx.x; idx < n_src * kCandCap; idx += kStreamThreads) {
        const int c = idx / kCandCap, q = idx % kCandCap, n = cnt[c];
        if (q >= n || !all_ok) cand[c * source_stride + q] = Cand{kCandEmpty, -1};
        if (q == 0 && n > kCandCap && all_ok) flooded[atomicAdd(words + 2, 1)] = c;
    }
    __syncthreads();
    const int n_flooded = *reinterpret_cast<volatile int *>(words + 2);
    // ---- rework: sixteen such sources at a time, the chunk's edges resident, each source searched exactly by a warp ----
    // (thread 0 alone copies and multiplies, tile after tile; uses of a barrier are counted on from the sweep's)
    bool alive = true;
    for (int f0 = 0; f0 < n_flooded && alive; f0 += 16) {
        const int nf = min(16, n_flooded - f0);
        stage_sources(16, [&](int r) { return r < nf ? flooded[f0 + r] : -1; }, [](int, int, float) {});
        fence_proxy_async();
        __syncthreads();
        if (threadIdx.x == 0) {
            // stage 0 of the ring, one tile at a time: slow and simple
            int use = (n_local + S - 1) / S + (f0 / 16) * n_local;      // fills of stage 0 so far
            const uint32_t idesc = umma_idesc_bf16(128, 16);
            for (int i = 0; i < n_local && ok; ++i, ++use) {
                tma_load_tile<kD>(base + l.stage, &tmK, s_full0, (t0 + i) * kTileKeys, h, b);
                ok = mbar_wait(s_full0, use & 1, lim);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < kD / 16; ++k)
                    umma_bf16(tmem_base + i * 16, umma_desc_sw128(base + l.stage + (k >> 2) * kHalfBytes + (k & 3) * 32),
                              umma_desc_sw128(base + (k >> 2) * (16 * 128) + (k & 3) * 32), idesc, k > 0);
                umma_commit(s_done);
                ok = mbar_wait(s_done, ((f0 / 16) * n_local + i) & 1, lim);
            }
        }
        tc_fence_before();
        alive = __syncthreads_and(ok ? 1 : 0) != 0;
        tc_fence_after();
        if (!alive) break;
        // cosines in the place of the ring, eight sources at a time
        float *cosines = reinterpret_cast<float *>(gen + l.stage);      // [round][keys]
        const int keys = n_local * kTileKeys;
        const int round = 8 * keys * 4 <= S * tile_bytes<kD>() ? 8 : 4;
        for (int g0 = 0; g0 < nf; g0 += round) {
            if (ew >= 0)
                for (int i = ew >> 2; i < n_local; i += 4) {
                    uint32_t r[8];
                    __syncwarp();
                    tmem_ld8_issue(tmem_base + ((uint32_t)(quad * 32) << 16) + i * 16 + (g0 & ~7), r);
                    tmem_ld_fence(r);
                    const int key = i * kTileKeys + key_lane;
                    const float inv = inv_norm[key];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int g = (g0 & ~7) + q;
                        if (g >= g0 && g < min(nf, g0 + round)) {
                            const int c = flooded[f0 + g];
                            const float e = clamped_edge(__uint_as_float(r[q]) * inv * src_inv[c]);
                            cosines[(g - g0) * keys + key] = j0 + key == src_pos[c] ? kCandEmpty : e;
                        }
                    }
                }
            __syncthreads();
            if (ew >= 0 && ew < round && g0 + ew < nf) {
                const int c = flooded[f0 + g0 + ew];
                const float *x = cosines + ew * keys;
                float bound;
                const int n = warp_list_top(keys, d.m, -1.0f, [&](int i) { return x[i]; },
                                            [&](int at, float e, int i) { cand[c * source_stride + at] = Cand{e, j0 + i}; }, &bound);
                for (int q = n + lane; q < kCandCap; q += 32) cand[c * source_stride + q] = Cand{kCandEmpty, -1};
            }
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
        }
    }
    if (!ok && a.status) atomicExch(a.status, (int)GRAPHKV_ERR_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    pc.mark();
    pc.flush(0);
}

}  // namespace tc
}  // namespace graphkv
