// Steps (II)+(III), first half, for many sources or long rows: the edges of all sources of a head with a chunk of its
// keys in one sweep, compared with bounds as they come out of tensor memory.
//
// similarity_tc keeps a chunk's whole edge block in tensor memory until bounds for the chunk are known, so its loads stop
// for half of its time, and a head with more than 64 sources is swept several times.  Here the bounds come first: a
// sample of the row (similarity_tc in its sampling form, a cluster of CTAs per 32 sources) gives per source a
// value that at least m of its edges reach; with a fifth of the row sampled about 7 m edges of the row reach it.  The sweep
// then streams: up to 192 sources are the columns of one product per key tile, two to four accumulators rotate, eight warps take
// the keys' norms, and 16 epilogue warps (thread = key) push the edges that reach their source's bound into queues of
// their own, with predicated stores and no branch, and list them from there, by source and chunk.
//
// In a text, keys that are alike stand together, so most of a source's 7 m edges can fall to few tiles.  So the sample is slices
// of eight keys all along the row, a chunk's tiles are spread over the row, and a list that is full (kCandCap) spills: the
// CTA keeps up to kStreamSpill more edges in memory, and a warp picks from those of a source when the sweep is done.  What does
// not fit there either is counted in bins, and the sources concerned are swept again with the bound that the bins give.  Where
// more edges tie than a list holds, the chunk's edges of the source are searched exactly.
//
// Bound: the comparisons.  128 keys x 160 sources take 1.8 us per SM, of which the products are 0.35 and the arrival of the tile
// 0.4; per 32 sources a warp spends about 400 issue slots on the comparisons of its 32 keys and on the edges found.  At 32
// sources a tile takes 0.8 us, near the 0.72 at which HBM delivers it.  Whole calls, with similarity_tc and with this (keys drawn
// independently; topics that last 64 tokens; 512): 154 sources at 32K x 8 heads 189 -> 154, 195 -> 183, 214 -> 173 us; 100 sources
// at 128K x 32 heads 1692 -> 1001, 1703 -> 1111, 1703 -> 1118; 32 sources there 822 -> 780, 822 -> 765, 854 -> 780; 100 at 16K x 128
// 878 -> 705, 901 -> 805, 904 -> 754.  A sample of whole tiles, chunks of adjacent tiles and lists without spill took, in place of
// 154, 183 and 173, 152, 326 and 463.  Tried: setp and a predicated store per edge instead of the sums of bits (the same time),
// queues listed at four instead of nine edges (2 us more), four warps for the norms (they held up the sweep of 32 sources),
// another sweep in place of the spilled edges (topics of 256 tokens: 20 to 60 us more), spilled edges without the bins (where they
// do not suffice, up to ten times the time).
//
// The lists have the form similarity_tc leaves, and together hold every member of the head-wide top-m.
//
#pragma once

#include "block_select.cuh"
#include "sim_tc.cuh"

namespace graphkv {
namespace tc {

constexpr int kStreamThreads = 64 + 256 + 512;          // producer, MMA, 8 norm warps, 16 epilogue warps
constexpr int kStreamMaxSources = 192;
constexpr int kStreamMaxTiles = 32;                     // tiles per chunk: the exact search holds 16 sources' edges with them
constexpr int kStreamSpill = 4096;                      // edges that full lists do not take, kept by a CTA
constexpr int kStreamBins = 64;                         // per source, in which those beyond are counted
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
    uint2 *spill;             // [sweeps][units][chunks][kStreamSpill] edges that a CTA keeps beside the lists
    int *status;
    int chunks;               // CTAs per unit
    int n_tiles;              // 128-key tiles per unit
    int np;                   // sources per sweep, padded to a multiple of 32
    int stages;
    int wait_prior;
    long long wait_cycles;
    int withhold_commit;      // test hook: the first accumulator is never announced
};

// Dynamic shared memory, byte offsets from a 1024-byte aligned base.
struct StreamLayout {
    uint32_t stage, queue, inv_norm, own_key, src_inv, theta, cnt, lo, scale, col, exact, hist, bars, bytes;
};
template <int kD> __host__ __device__ inline StreamLayout stream_layout(int np, int stages)
{
    StreamLayout l;
    l.stage = np * 2 * kD;                               // source keys | key tiles in flight
    l.queue = l.stage + stages * tile_bytes<kD>();       // [stream_queue][512]; between sweeps the next one's columns [3][np]
    l.inv_norm = l.queue + stream_queue(np) * 512 * 8;   // [kStreamMaxTiles][128]
    l.own_key = l.inv_norm + kStreamMaxTiles * 128 * 4;  // per column of the sweep: own key, 1 / norm, bound (negated), edges
    l.src_inv = l.own_key + np * 4;                      // found, source
    l.theta = l.src_inv + np * 4;
    l.cnt = l.theta + np * 4;
    l.lo = l.cnt + np * 4;                               // bound, and bins per unit above it, of the histogram
    l.scale = l.lo + np * 4;
    l.col = l.scale + np * 4;
    l.exact = l.col + np * 4;                            // [np] sources to be searched exactly
    l.hist = l.exact + np * 4;                           // [np][kStreamBins] 16-bit counts
    l.bars = l.hist + np * kStreamBins * 2;              // full[8], empty[8], tfull[4], tempty[4], tensor memory's base, words, norms[kStreamMaxTiles]
    l.bytes = l.bars + 28 * 8 + 32 + kStreamMaxTiles * 8 + 1024;
    return l;
}
__host__ __device__ inline int stream_bufs(int np) { return np <= 128 ? 4 : np <= 160 ? 3 : 2; }

// What the listing of edges needs.  (Put together where edges are listed, from the arguments: kept through the sweep, its
// registers cost 2 us of a call of 154 sources.)
struct StreamColumns {
    int chunk, chunks, again;
    const int *own_key, *col;    // per column of the sweep: the source's own key of the chunk or -1, the source (the first sweep's: itself)
    int *cnt;                    // edges found
    Cand *cand;                  // source c's list of this chunk at c * source_stride
    long long source_stride;
    uint32_t *row_hist;          // the row's listed edges
    uint2 *spill;                // [kStreamSpill] edges that full lists did not take: cosine, (column, key)
    int *spilled;                // their number, kept or not
    const float *lo, *scale;     // the bins: the bound, bins per unit above it
    uint32_t *hist;              // [np][kStreamBins] 16-bit counts of those not kept
    __device__ __forceinline__ int position(int key) const { return ((key >> 7) * chunks + chunk) * kTileKeys + (key & 127); }
    __device__ __forceinline__ int key_of(int pos) const
    {
        const int tile = pos >> 7;
        return tile % chunks == chunk ? tile / chunks * kTileKeys + (pos & 127) : -1;
    }
    __device__ __forceinline__ void count(int c, float e) const
    {
        const int b = min(max(static_cast<int>((e - lo[c]) * scale[c]), 0), kStreamBins - 1);
        atomicAdd(hist + c * (kStreamBins / 2) + (b >> 1), 1u << (16 * (b & 1)));
    }
    // edge `at` of the column, below kCandCap
    __device__ __forceinline__ void list(int c, int at, int key, float x) const
    {
        const float e = clamped_edge(x);
        const int src = again ? col[c] : c;
        cand[src * source_stride + at] = Cand{e, position(key)};
        atomicAdd(row_hist + src * kCandBins + cand_bin(e), 1u);
    }
    // an edge beyond the list, the place-th of the chunk
    __device__ __forceinline__ void put_aside(int c, int place, int key, float x) const
    {
        const float e = clamped_edge(x);
        if (place < kStreamSpill) spill[place] = make_uint2(__float_as_uint(e), (uint32_t)c << 16 | (uint32_t)key);
        else count(c, e);
    }
};

// Edges (column c, key of the chunk, cosine before clamping x; c < 0: none) into the lists of their sources.  (Their number is
// small, but a warp goes through this for whichever lane has one: 30 instructions more took 3 us of a call of 154 sources.)
template <int kN>
__device__ __forceinline__ void stream_list(const int (&c)[kN], const int (&key)[kN], const float (&x)[kN], const StreamColumns &s)
{
    int at[kN];
#pragma unroll
    for (int q = 0; q < kN; ++q) {
        at[q] = -1;
        if (c[q] >= 0 && key[q] != s.own_key[c[q]]) at[q] = atomicAdd(s.cnt + c[q], 1);
    }
    bool beyond = false;
#pragma unroll
    for (int q = 0; q < kN; ++q) {
        if ((uint32_t)at[q] < (uint32_t)kCandCap) s.list(c[q], at[q], key[q], x[q]);
        beyond |= at[q] >= kCandCap;
    }
    if (beyond) {
#pragma unroll
        for (int q = 0; q < kN; ++q)
            if (at[q] >= kCandCap) s.put_aside(c[q], atomicAdd(s.spilled, 1), key[q], x[q]);
    }
}

// One column's edges of a warp's keys (in: the edge reaches the bound), counted together.
__device__ __forceinline__ void stream_list_column(int c, int key, bool in, float x, const StreamColumns &s)
{
    const int lane = threadIdx.x & 31;
    in = in && key != s.own_key[c];
    const unsigned all = __ballot_sync(0xffffffffu, in);
    if (all == 0u) return;
    const int n = __popc(all), rank = __popc(all & ((1u << lane) - 1u));
    int first = 0, place = 0;
    if (lane == 0) {
        first = atomicAdd(s.cnt + c, n);
        if (first + n > kCandCap) place = atomicAdd(s.spilled, min(n, first + n - kCandCap));
    }
    first = __shfl_sync(0xffffffffu, first, 0);
    place = __shfl_sync(0xffffffffu, place, 0);
    if (in && first + rank < kCandCap) s.list(c, first + rank, key, x);
    else if (in) s.put_aside(c, place + rank - max(kCandCap - first, 0), key, x);
}

template <int kD>
__device__ __forceinline__ StreamColumns stream_columns(const SimStreamArgs &a, uint8_t *gen, int again)
{
    const StreamLayout l = stream_layout<kD>(a.np, a.stages);
    const int unit = blockIdx.y, chunk = blockIdx.x;
    const long long source0 = (long long)unit * a.d.K_src + blockIdx.z * a.np;
    return StreamColumns{chunk, a.chunks, again, reinterpret_cast<int *>(gen + l.own_key), reinterpret_cast<int *>(gen + l.col),
                         reinterpret_cast<int *>(gen + l.cnt), a.cand + (source0 * a.chunks + chunk) * kCandCap, (long long)a.chunks * kCandCap,
                         a.cand_hist + source0 * kCandBins,
                         a.spill + ((long long)(blockIdx.z * gridDim.y + unit) * a.chunks + chunk) * kStreamSpill,
                         reinterpret_cast<int *>(gen + l.bars + 28 * 8) + 3, reinterpret_cast<float *>(gen + l.lo),
                         reinterpret_cast<float *>(gen + l.scale), reinterpret_cast<uint32_t *>(gen + l.hist)};
}

// The edges of this thread's queue listed.
template <int kD>
__device__ __forceinline__ void stream_flush(const SimStreamArgs &a, uint8_t *gen, int queued, int again)
{
    const StreamLayout l = stream_layout<kD>(a.np, a.stages);
    const StreamColumns columns = stream_columns<kD>(a, gen, again);
    const float *src_inv = reinterpret_cast<const float *>(gen + l.src_inv);
    const uint2 *q0 = reinterpret_cast<const uint2 *>(gen + l.queue) + ((int)threadIdx.x - 320);
    const int queue = stream_queue(a.np);
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
        stream_list<4>(c, key, x, columns);
    }
    __syncwarp();
}

// The edges of a slice that are more than the queues take, listed from tensor memory.
template <int kD>
__device__ __forceinline__ void stream_slice(const SimStreamArgs &a, uint8_t *gen, uint32_t taddr, int col0, int n_col, int key, float inv, int again)
{
    const StreamLayout l = stream_layout<kD>(a.np, a.stages);
    const StreamColumns columns = stream_columns<kD>(a, gen, again);
    const float *src_inv = reinterpret_cast<const float *>(gen + l.src_inv), *theta = reinterpret_cast<const float *>(gen + l.theta);
#pragma unroll 1
    for (int c0 = col0; c0 < col0 + 32 && c0 < n_col; c0 += 8) {
        uint32_t r[8];
        __syncwarp();
        tmem_ld8_issue(taddr + c0 - col0, r);
        tmem_ld_fence(r);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            stream_list_column(c0 + q, key, fmaf(__uint_as_float(r[q]), inv, theta[c0 + q]) > 0.f,
                               __uint_as_float(r[q]) * inv * src_inv[c0 + q], columns);
    }
    __syncwarp();
}

// After a sweep in which lists were full: what was spilled, put in order by column (sorted, in the place of the ring; the columns'
// counts behind it), and for every column concerned its list, or its place among those to sweep again (`last`: none) or to
// search exactly.  By all threads; a function of its own, which keeps its registers out of the sweep's.
__device__ __noinline__ void stream_resolve(StreamColumns s, uint2 *sorted, int *next, int *exact, int *words, int np, int n_col, int m, bool last)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_spilled = min(*reinterpret_cast<volatile int *>(words + 3), kStreamSpill);
    float *bound = reinterpret_cast<float *>(next + np), *bins_of = bound + np;
    int *kept = reinterpret_cast<int *>(sorted + kStreamSpill), *end = kept + np;       // [np] a column's edges, and their end
    for (int c = threadIdx.x; c < n_col; c += kStreamThreads) kept[c] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n_spilled; i += kStreamThreads) atomicAdd(kept + (__ldcg(&s.spill[i].y) >> 16), 1);
    __syncthreads();
    if (warp == 0) {
        int run = 0;
        for (int c0 = 0; c0 < n_col; c0 += 32) {
            const int mine = c0 + lane < n_col ? kept[c0 + lane] : 0, incl = (int)bs::incl_scan((uint32_t)mine, lane);
            if (c0 + lane < n_col) end[c0 + lane] = run + incl - mine;
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n_spilled; i += kStreamThreads) {
        const uint2 en = __ldcg(s.spill + i);
        sorted[atomicAdd(end + (en.y >> 16), 1)] = make_uint2(en.x, en.y & 0xffffu);
    }
    __syncthreads();
    // A source with more edges than slots, by a warp: those that reach a bound at which a list holds them.  Where some
    // were not kept, another sweep with a bound from the counts; where too many tie, the exact search.
    for (int c = warp; c < n_col; c += kStreamThreads / 32) {
        const int excess = s.cnt[c] - kCandCap, have = kept[c];
        if (excess <= 0) continue;
        Cand *list = s.cand + s.col[c] * s.source_stride;
        uint32_t *bins = s.row_hist + s.col[c] * kCandBins;
        Cand own[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int2 raw = __ldcg(reinterpret_cast<const int2 *>(list + q * 32 + lane));
            own[q] = Cand{__int_as_float(raw.x), raw.y};
            atomicAdd(bins + cand_bin(own[q].e), 0xffffffffu);          // (counted anew)
        }
        const uint2 *more = sorted + end[c] - have - kCandCap;
        if (have == excess) {
            float reached;
            const int n = warp_list_top<false>(kCandCap + have, m, -1.0f,
                [&](int i) { return i < 32 ? own[0].e : i < 64 ? own[1].e : __uint_as_float(more[i].x); },
                [&](int at, float e, int i) {
                    list[at] = Cand{e, i < 32 ? own[0].j : i < 64 ? own[1].j : s.position((int)more[i].y)};
                    atomicAdd(bins + cand_bin(e), 1u);
                }, &reached);
            if (n >= 0) {
                for (int q = n + lane; q < kCandCap; q += 32) list[q] = Cand{kCandEmpty, -1};
                continue;
            }
        } else if (!last) {
            // all of the column's edges counted, two bins per lane: the highest bin from which on there are m of them
            // (its lower end less what a rounding may be)
            s.count(c, own[0].e);
            s.count(c, own[1].e);
            for (int i = kCandCap + lane; i < kCandCap + have; i += 32) s.count(c, __uint_as_float(more[i].x));
            __syncwarp();
            const uint32_t two = s.hist[c * (kStreamBins / 2) + lane];
            const int from = (int)bs::incl_scan(__shfl_sync(0xffffffffu, (two & 0xffffu) + (two >> 16), 31 - lane), lane);
            const int run = __shfl_sync(0xffffffffu, from, 31 - lane);           // in this lane's bins and above
            const int word = 31 - __clz(__ballot_sync(0xffffffffu, run >= m));
            const int above = __shfl_sync(0xffffffffu, run - (int)(two & 0xffffu), word);
            const int bin = 2 * word + (above >= m ? 1 : 0);
            if (lane == 0) {
                const int at = atomicAdd(words + 2, 1);
                next[at] = s.col[c];
                bound[at] = s.lo[c] + bin / s.scale[c] - (bin > 0 ? 4e-7f : 0.f);
                bins_of[at] = s.scale[c] * kStreamBins;
            }
            continue;
        }
        if (lane == 0) exact[atomicAdd(words + 4, 1)] = s.col[c];
    }
}

// grid (chunks, units, sweeps of np sources).
template <int kD>
__global__ void __launch_bounds__(kStreamThreads, 1)
sim_stream_tc(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ SimStreamArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const Dims &d = a.d;
    const long long lim = a.wait_cycles;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base - smem_u32(smem_raw));
    const int np = a.np, S = a.stages;
    const StreamLayout l = stream_layout<kD>(np, S);
    float *inv_norm = reinterpret_cast<float *>(gen + l.inv_norm);
    int *own_key = reinterpret_cast<int *>(gen + l.own_key), *col = reinterpret_cast<int *>(gen + l.col);
    float *src_inv = reinterpret_cast<float *>(gen + l.src_inv), *theta = reinterpret_cast<float *>(gen + l.theta);
    int *cnt = reinterpret_cast<int *>(gen + l.cnt), *exact = reinterpret_cast<int *>(gen + l.exact);
    int *next = reinterpret_cast<int *>(gen + l.queue);                 // [np] the next sweep's sources,
    float *bound = reinterpret_cast<float *>(next + np), *bins_of = bound + np;                // [np] their bounds and bins per unit
    float *lo = reinterpret_cast<float *>(gen + l.lo), *scale = reinterpret_cast<float *>(gen + l.scale);
    uint32_t *counts = reinterpret_cast<uint32_t *>(gen + l.hist);      // [np][kStreamBins / 2]
    const uint32_t s_full0 = base + l.bars, s_empty0 = s_full0 + 64, s_tfull0 = s_empty0 + 64, s_tempty0 = s_tfull0 + 32,
                   s_tmem = s_tempty0 + 40, s_norms0 = s_full0 + 28 * 8 + 32;
    int *words = reinterpret_cast<int *>(gen + l.bars + 28 * 8);        // [1] failed, [2] sources to sweep again, [3] edges spilled, [4] sources to search
    PhaseClock pc(threadIdx.x == 320);
    pc.mark();
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int unit = blockIdx.y, b = unit / d.hkv, h = unit % d.hkv, chunk = blockIdx.x;
    // (a chunk's tiles are spread over the row, so that a passage of similar keys is spread over the chunks)
    const int n_local = (a.n_tiles - chunk + a.chunks - 1) / a.chunks;
    auto tile_of = [&](int i) { return chunk + i * a.chunks; };
    const __nv_bfloat16 *src_rows = a.S + b * a.ss[0] + (long long)h * a.ss[1];
    const int src0 = blockIdx.z * np, n_src = min(np, d.K_src - src0);
    const long long source0 = (long long)unit * d.K_src + src0, source_stride = (long long)a.chunks * kCandCap;
    Cand *cand = a.cand + (source0 * a.chunks + chunk) * kCandCap;      // source c's list of this chunk at c * source_stride
    uint32_t *hist = a.cand_hist + source0 * kCandBins;

    int n_ahead = 0;
    // barriers for a sweep of n columns (the first: with the keys' norms); those before are at rest
    auto init_barriers = [&](int n, bool first) {
        if (!first) {
            for (int i = 0; i < S; ++i) mbar_inval(s_full0 + 8 * i), mbar_inval(s_empty0 + 8 * i);
            for (int i = 0; i < 4; ++i) mbar_inval(s_tfull0 + 8 * i), mbar_inval(s_tempty0 + 8 * i);
        }
        for (int i = 0; i < S; ++i) {
            mbar_init(s_full0 + 8 * i, 1);
            mbar_init(s_empty0 + 8 * i, first ? 1 + 4 : 1);        // the MMA's commit and the norm warps
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(s_tfull0 + 8 * i, 1);
            mbar_init(s_tempty0 + 8 * i, 4 * (n / 32));                 // a warp per slice of 32 sources and lane quarter
        }
        if (first)
            for (int i = 0; i < n_local; ++i) mbar_init(s_norms0 + 8 * i, 4);
        mbar_fence_init();
    };
    if (threadIdx.x == 0) {
        init_barriers(np, true);
        words[1] = words[2] = words[3] = words[4] = 0;
        tma_prefetch_desc(&tmK);
        // (keys are an input of the call: no wait for the kernels before)
        n_ahead = min(S, n_local);
        for (int i = 0; i < n_ahead; ++i)
            tma_load_tile<kD>(base + l.stage + i * tile_bytes<kD>(), &tmK, s_full0 + 8 * i, tile_of(i) * kTileKeys, h, b);
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
        constexpr int kU = 4;                            // pieces in flight per thread: a position, then the row's piece
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
    bool ok = true, all_ok = true;
    uint32_t tmem_base = 0u;
    const int ew = warp - 10, quad = warp & 3, et = (int)threadIdx.x - 320;
    const int key_lane = quad * 32 + lane;
    // Sweeps: the first of all sources with the sample's bounds; then of those whose edges were not all kept, with bounds from
    // the counts of the first.  (Each with code of its own: in one loop the first took 3 us more.)
    int n_col = n_src;
    auto sweep = [&](auto again) {
        constexpr int pass = decltype(again)::value;
        const int width = pass == 0 ? np : (n_col + 31) & ~31, bufs = stream_bufs(width), n_slices = width / 32;
        stage_sources(width, [&](int r) { return r >= n_col ? -1 : pass == 0 ? r : next[r]; }, [&](int r, int pos, float n2) {
            const float norm = fmaxf(sqrtf(n2), kNormEps);
            const bool in = r < n_col;
            const float least = !in ? 0.f : pass == 0 ? fmaxf(__ldcg(a.tau + source0 + r), -1.0f) : bound[r];
            own_key[r] = pos < 0 ? -1 : StreamColumns{chunk, a.chunks}.key_of(pos);
            src_inv[r] = 1.0f / norm;
            cnt[r] = 0;
            col[r] = !in ? 0 : pass == 0 ? r : next[r];
            lo[r] = least;
            scale[r] = pass == 0 ? kStreamBins / fmaxf(1.0f - least, 1e-6f) : in ? bins_of[r] : 0.f;
            // the bound brought to the scale of dot / |k_j|, lowered so that no edge whose cosine rounds up to it is missed
            // (kept negated; an infinite bound would make a difference of infinities)
            const float q = in ? ((least <= -1.0f ? -2.0f : least) - 2.4e-7f) * norm : 3.0e38f;
            theta[r] = -(q - fabsf(q) * 3.6e-7f - 1e-30f);
        });
        for (int i = threadIdx.x; i < width * (kStreamBins / 2); i += kStreamThreads) counts[i] = 0u;
        fence_proxy_async();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        tmem_base = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(gen + (s_tmem - base)), 0);
        pc.mark();
        if (warp == 0) {
            if (lane == 0) {
                int issued = n_ahead;
                for (int i = n_ahead; i < n_local; ++i) {
                    const int st = i % S, ph = (i / S) & 1;
                    if (!mbar_wait(s_empty0 + 8 * st, ph ^ 1, lim)) { ok = false; break; }
                    tma_load_tile<kD>(base + l.stage + st * tile_bytes<kD>(), &tmK, s_full0 + 8 * st, tile_of(i) * kTileKeys, h, b);
                    ++issued;
                }
                // the last copies have landed, and are used, before the ring's place and its barriers are used again or the CTA exits
                for (int i = max(0, issued - S); i < issued; ++i) {
                    ok = mbar_wait(s_full0 + 8 * (i % S), (i / S) & 1, lim) && ok;
                    ok = ok && mbar_wait(s_empty0 + 8 * (i % S), (i / S) & 1, lim);
                }
            }
        } else if (warp == 1) {
            const uint32_t idesc = umma_idesc_bf16(128, width), src_lo = umma_desc_lo(base), ring_lo = umma_desc_lo(base + l.stage);
            int st = 0, buf = 0;
            uint32_t ph = 0u, bph = 1u;
            for (int i = 0; i < n_local; ++i) {
                ok = mbar_wait(s_tempty0 + 8 * buf, bph, lim) && mbar_wait(s_full0 + 8 * st, ph, lim);
                if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
                tc_fence_after();
                if (elect_one()) {
                    umma_tile<kD>(tmem_base + buf * width, ring_lo + st * (tile_bytes<kD>() >> 4), kHalfBytes >> 4, src_lo, width * 128 >> 4, idesc);
                    umma_commit(s_empty0 + 8 * st);
                    if (!(a.withhold_commit && i == 0)) umma_commit(s_tfull0 + 8 * buf);
                }
                __syncwarp();
                if (++st == S) st = 0, ph ^= 1u;
                if (++buf == bufs) buf = 0, bph ^= 1u;
            }
        } else if (warp < 10) {
            // ---- norms of the keys, four warps a tile ----
            for (int i = (warp - 2) >> 2; i < n_local && ok && pass == 0; i += 2) {
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
                    tile_of(i) * kTileKeys + key_lane < d.N ? 1.0f / fmaxf(sqrtf(n0 + n1), kNormEps) : __int_as_float(0x7fc00000);
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
                stream_flush<kD>(a, gen, static_cast<int>((qa - q_first) / kStep), pass);
                qa = q_first;
            };
            int i = set / n_slices, sl = set % n_slices;
            while (i < n_local) {
                const int buf = i % bufs, col0 = sl * 32;
                ok = __all_sync(0xffffffffu, mbar_wait(s_tfull0 + 8 * buf, (i / bufs) & 1, lim));
                if (!ok) break;
                tc_fence_after();
                uint32_t raw[32];
                tmem_ld32_issue(lane_addr + buf * width + col0, raw);
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
                    stream_slice<kD>(a, gen, lane_addr + buf * width + col0, col0, n_col, key, inv, pass);
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
        all_ok = *reinterpret_cast<volatile int *>(words + 1) == 0;
        pc.mark();

        // ---- unused slots marked empty; what was spilled into order by column, in the place of the ring ----
        for (int idx = threadIdx.x; idx < n_col * kCandCap; idx += kStreamThreads) {
            const int c = idx / kCandCap, q = idx % kCandCap, n = cnt[c];
            if (q >= n || !all_ok) cand[col[c] * source_stride + q] = Cand{kCandEmpty, -1};
        }
        const int n_spilled = min(*reinterpret_cast<volatile int *>(words + 3), kStreamSpill);
        if (n_spilled > 0 && all_ok) {
            stream_resolve(stream_columns<kD>(a, gen, pass), reinterpret_cast<uint2 *>(gen + l.stage), next, exact, words, np, n_col, d.m, pass == 1);
        }
        __syncthreads();
        n_col = *reinterpret_cast<volatile int *>(words + 2);
    };
    sweep(std::integral_constant<int, 0>{});
    if (n_col > 0) {
        n_ahead = 0;
        __syncthreads();
        if (threadIdx.x == 0) {
            words[2] = words[3] = 0;
            init_barriers((n_col + 31) & ~31, false);
        }
        sweep(std::integral_constant<int, 1>{});
    }
    const int n_exact = *reinterpret_cast<volatile int *>(words + 4);
    if (n_exact > 0) {
        __syncthreads();
        if (threadIdx.x == 0) init_barriers(32, false);
        __syncthreads();
    }
    // ---- sixteen such sources at a time, the chunk's edges resident, each source searched exactly by a warp ----
    // (thread 0 alone copies and multiplies)
    bool alive = true;
    for (int f0 = 0; f0 < n_exact && alive; f0 += 16) {
        const int nf = min(16, n_exact - f0);
        stage_sources(16, [&](int r) { return r < nf ? exact[f0 + r] : -1; }, [&](int r, int pos, float n2) {
            own_key[r] = pos;                       // (here its position)
            src_inv[r] = 1.0f / fmaxf(sqrtf(n2), kNormEps);
        });
        fence_proxy_async();
        __syncthreads();
        if (threadIdx.x == 0) {
            const uint32_t idesc = umma_idesc_bf16(128, 16);
            const int use0 = (f0 / 16) * n_local;                       // fills and uses of the ring go on from group to group
            auto load = [&](int i) {
                const int st = (use0 + i) % S;
                tma_load_tile<kD>(base + l.stage + st * tile_bytes<kD>(), &tmK, s_full0 + 8 * st, tile_of(i) * kTileKeys, h, b);
            };
            int issued = 0;
            for (; issued < min(S, n_local); ++issued) load(issued);
            for (int i = 0; i < n_local && ok; ++i) {
                const int st = (use0 + i) % S, ph = (use0 + i) / S & 1;
                ok = mbar_wait(s_full0 + 8 * st, ph, lim);
                if (!ok) break;
                tc_fence_after();
                const uint32_t tile = base + l.stage + st * tile_bytes<kD>();
#pragma unroll
                for (int k = 0; k < kD / 16; ++k)
                    umma_bf16(tmem_base + i * 16, umma_desc_sw128(tile + (k >> 2) * kHalfBytes + (k & 3) * 32),
                              umma_desc_sw128(base + (k >> 2) * (16 * 128) + (k & 3) * 32), idesc, k > 0);
                umma_commit(s_empty0 + 8 * st);
                // the product before this one has left its tile
                if (i > 0) ok = mbar_wait(s_empty0 + 8 * ((use0 + i - 1) % S), (use0 + i - 1) / S & 1, lim);
                if (ok && i > 0 && issued < n_local) load(issued++);
            }
            if (ok) ok = mbar_wait(s_empty0 + 8 * ((use0 + n_local - 1) % S), (use0 + n_local - 1) / S & 1, lim);
            else        // gave up: the copies in flight land before the CTA exits
                for (int i = max(0, issued - S); i < issued; ++i) mbar_wait(s_full0 + 8 * ((use0 + i) % S), (use0 + i) / S & 1, lim);
        }
        tc_fence_before();
        alive = __syncthreads_and(ok ? 1 : 0) != 0;
        tc_fence_after();
        if (!alive) break;
        // cosines in the place of the ring, sixteen, eight or four sources at a time
        float *cosines = reinterpret_cast<float *>(gen + l.stage);      // [round][keys]
        const int keys = n_local * kTileKeys;
        int round = 16;
        while (round * keys * 4 > S * tile_bytes<kD>()) round /= 2;
        for (int g0 = 0; g0 < nf; g0 += round) {
            if (ew >= 0)
                for (int i = ew >> 2; i < n_local; i += 4)
                    for (int h0 = g0 & ~7; h0 < min(nf, g0 + round); h0 += 8) {
                        uint32_t r[8];
                        __syncwarp();
                        tmem_ld8_issue(tmem_base + ((uint32_t)(quad * 32) << 16) + i * 16 + h0, r);
                        tmem_ld_fence(r);
                        const int key = i * kTileKeys + key_lane;
                        const float inv = inv_norm[key];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const int g = h0 + q;
                            if (g >= g0 && g < min(nf, g0 + round)) {
                                const float e = clamped_edge(__uint_as_float(r[q]) * inv * src_inv[g]);
                                cosines[(g - g0) * keys + key] = tile_of(i) * kTileKeys + key_lane == own_key[g] ? kCandEmpty : e;
                            }
                        }
                    }
            __syncthreads();
            if (ew >= 0 && ew < round && g0 + ew < nf) {
                const int c = exact[f0 + g0 + ew];
                const float *x = cosines + ew * keys;
                Cand *list = cand + c * source_stride;
                float reached;
                const int n = warp_list_top(keys, d.m, -1.0f, [&](int i) { return x[i]; },
                                            [&](int at, float e, int i) {
                                                list[at] = Cand{e, tile_of(i >> 7) * kTileKeys + (i & 127)};
                                                atomicAdd(hist + c * kCandBins + cand_bin(e), 1u);
                                            }, &reached);
                for (int q = n + lane; q < kCandCap; q += 32) list[q] = Cand{kCandEmpty, -1};
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
    pc.flush(8);
}

}  // namespace tc
}  // namespace graphkv
