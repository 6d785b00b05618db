// Steps (II)+(III), first half, on the tensor cores (bf16 inputs): the edges e_ij of Eq. 1 between
// the source nodes of a head and every prefix key, and per key chunk the candidates for each
// source's top-m neighbourhood (Eq. 3).  The edge matrix never leaves the SM.
//
// One CTA owns a chunk of at most 512 / NP key tiles of one head (NP = source count padded to
// 16, 32 or 64; a head with more sources is swept once per NP of them, by CTAs of their own).  Each
// 128-key tile arrives by TMA, one tcgen05.mma block computes its 128 x NP dot products against the
// source keys into its own TMEM columns, and epilogue threads (thread = key) take the key's norm from the
// staged tile and, per source, the maximum of dot / |k_j| over their keys.  When the sweep is over the
// chunk's whole edge block still sits in TMEM, and
//   1. a warp per source bounds the chunk's m-th largest edge from below by those maxima (edge_search.cuh);
//   2. every thread reads its part of the block again and queues the edges that reach the bound, with
//      predicated stores and no branch;
//   3. the queued edges are turned into cosines and listed by source; where a queue runs over (a key close to every
//      source of a cluster), all edges that reach the bounds are listed anew, without queues;
//   4. sources with too many (ties) are searched exactly, from cosines in the ring's memory.
// The lists of all chunks hold every member of the head-wide top-m.  Each listed edge is also counted in a
// per-source histogram over the cosine, from which the finishing kernel takes a bound that leaves it a few
// dozen edges to rank.
//
// Bound: the sweep by HBM or L2 (about 0.6 us per 32 KB tile and SM); what follows it is latency: 6.5 us for
// 14 tiles and 16 sources, 9.5 us for 32 (of them the bounds 2 and 3.5, the second pass 2 and 3, the lists 1:
// 1.7 with one edge after the other).  Sources of one cluster (32 of them, 512 keys close to each, 32768 keys in
// all) 39 us instead of 27; when a queue that ran over sent every source to step 4 it was 55.  With
// eight epilogue warps, maxima turned into bins of bytes and a threshold bin bisected, it was 9 and 13.5 us;
// with the cosines of 16 sources staged in shared memory and searched there, 9 and 17.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "edge_search.cuh"
#include "tc_common.cuh"

namespace graphkv {
namespace tc {

constexpr int kSimEpiThreads = 512;
constexpr int kSimThreads = 64 + kSimEpiThreads;        // producer warp, MMA warp, 16 epilogue warps
constexpr int kSimMaxNeighbors = 32;    // m this path handles
constexpr int kSimMaxTiles = 32;        // tiles per CTA at NP = 16 (512 TMEM columns)

struct SimTcArgs {
    Dims d;
    const __nv_bfloat16 *S;   // tensor the source nodes' vectors are read from (the swept tensor comes
                              // through the tensor map)
    long long ss[3];          // its element strides: batch, head, token
    const int *src;        // [units][K_src] source positions
    Cand *cand;            // [units][K_src][chunks][kCandCap]; unused slots hold e = kCandEmpty
    uint32_t *cand_hist;   // [units][K_src][kCandBins] listed edges per cosine bin (zeroed before)
    int *status;
    int unit0;
    int chunks;            // CTAs per unit
    int n_tiles;           // 128-key tiles per unit
    int stages;
    int wait_prior;        // launched with programmatic stream serialization
    long long wait_cycles; // limit of every wait of the kernel, in clocks
    int slice_step;        // sampling form: n_tiles tiles shared by the `chunks` CTAs of a cluster, each of kSlices slices of the
                           // row's, one every slice_step keys (a passage of few similar keys has its share of the sample)
    float *tau;            // sampling form: [units][K_src] per source, a value that at least m of its edges reach
    int withhold_commit;   // test hook: the first product is never announced
};

constexpr int kSliceKeys = 8, kSlices = kTileKeys / kSliceKeys;

template <int NP> __host__ __device__ constexpr int sim_tiles_cap() { return 512 / NP; }
// Bytes of the ring's place: the tiles in flight; then maxima [NP][512 or 256]; then, with the bounds taken,
// queues; then, where a source is searched exactly, cosines of a round of 8 or 16 sources (8 x 4096 or 16 x 2048
// keys).
constexpr int kSimQueue = 40;           // edges per thread's queue
constexpr int kSimRing = 163840;
template <int NP> __host__ __device__ constexpr int sim_parts() { return NP == 64 ? 256 : 512; }
static_assert(16 * 2048 * 4 <= kSimRing && 8 * 4096 * 4 <= kSimRing, "cosines of a round");
static_assert(64 * 256 * 4 <= kSimRing && 32 * 512 * 4 <= kSimRing, "maxima");
static_assert(kSimQueue * kSimEpiThreads * 8 <= kSimRing, "queues");

// Dynamic shared memory, byte offsets from a 1024-byte aligned base: source keys (K-major, 128-byte swizzle) | key
// tiles in flight, then what kSimRing lists | barriers | inverse norms of the chunk's keys [tile][128] | per source
// [NP]: position, 1 / norm, max(|k_c|, eps), bound of the chunk's m-th edge, count of listed edges | lists [NP][kCandCap]
template <int NP, int kD> struct SimShared {
    static constexpr uint32_t stage = NP * 2 * kD, full = stage + kSimRing, empty = full + 64, done = empty + 64,
                              tmem = done + kSimMaxTiles * 8, inv_norm = tmem + 16, src_pos = inv_norm + sim_tiles_cap<NP>() * 128 * 4,
                              src_inv = src_pos + NP * 4, src_norm = src_inv + NP * 4, tau = src_norm + NP * 4, cnt = tau + NP * 4,
                              list = cnt + NP * 4, bytes = list + NP * kCandCap * 8;
};
template <int NP, int kD> __host__ __device__ constexpr size_t sim_smem_bytes() { return 1024 + SimShared<NP, kD>::bytes + 64; }

__device__ __forceinline__ bool list_overflowed(const int *cnt, int c) { return *reinterpret_cast<const volatile int *>(cnt + c) > kCandCap; }

// Several edges (source c, key j of the chunk, cosine before clamping x; c < 0: none) into the lists, their latencies
// overlapped.  The order within a list carries no meaning; the source itself is no neighbour of its own; a list that has
// overflowed is not counted on (additions to one word take turns).
template <int kN>
__device__ __forceinline__ void list_edges(const int (&c)[kN], const int (&j)[kN], const float (&x)[kN], const int *src_pos, int j0,
                                           int *cnt, Cand *list)
{
    const uint32_t cnt_s = smem_u32(cnt);
    int at[kN];
#pragma unroll
    for (int q = 0; q < kN; ++q) {
        const int cc = max(c[q], 0);
        at[q] = (c[q] >= 0) & (j0 + j[q] != src_pos[cc]) & !list_overflowed(cnt, cc);
    }
#pragma unroll
    for (int q = 0; q < kN; ++q)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %0, 0;\n\tmov.s32 %0, %2;\n\t"
                     "@p atom.shared.add.u32 %0, [%1], 1;\n\t}"
                     : "+r"(at[q]) : "r"(cnt_s + 4 * max(c[q], 0)), "n"(kCandCap) : "memory");
#pragma unroll
    for (int q = 0; q < kN; ++q)
        if (at[q] < kCandCap) list[c[q] * kCandCap + at[q]] = Cand{clamped_edge(x[q]), j0 + j[q]};
}

// The lists of a chunk anew, without queues, by a warp over its part of the edge block (cnt at zero before).  A function
// of its own: in the kernel's body it cost a CTA of 14 tiles and 16 sources 0.6 us of 23.3 (registers and schedule), called
// or not.  Everything it needs is in shared memory (gen: its aligned base) or follows from the thread's number.
template <int NP, int kD>
__device__ __noinline__ void list_anew(uint8_t *gen, uint32_t tmem_base, int n_local, int n_src, int j0)
{
    using Sh = SimShared<NP, kD>;
    constexpr int kCols = NP < 32 ? NP : 32, kColSets = NP / kCols, kTileSets = 4 / kColSets;
    const int lane = threadIdx.x & 31, quad = (threadIdx.x >> 5) & 3, set = ((threadIdx.x >> 5) - 2) >> 2;
    const int col0 = (set % kColSets) * kCols;
    const float *inv_norm = reinterpret_cast<const float *>(gen + Sh::inv_norm), *tau = reinterpret_cast<const float *>(gen + Sh::tau);
    const float *src_inv = reinterpret_cast<const float *>(gen + Sh::src_inv);
    int *cnt = reinterpret_cast<int *>(gen + Sh::cnt);
#pragma unroll 1
    for (int i = set / kColSets; i < n_local; i += kTileSets) {
        const int key = i * kTileKeys + quad * 32 + lane;
        const float inv = inv_norm[key];
        // (no list left to add to: on to the exact search of all sources)
        if (__all_sync(0xffffffffu, (lane >= n_src || list_overflowed(cnt, lane)) &&
                                        (NP < 64 || lane + 32 >= n_src || list_overflowed(cnt, lane + 32))))
            break;
#pragma unroll 1
        for (int c0 = col0; c0 < col0 + kCols && c0 < n_src; c0 += 8) {
            uint32_t r[8];
            __syncwarp();
            tmem_ld8_issue(tmem_base + ((uint32_t)(quad * 32) << 16) + i * NP + c0, r);
            tmem_ld_fence(r);
            int c[8], j[8];
            float x[8];
            bool some = false;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int at = min(c0 + q, n_src - 1);
                x[q] = __uint_as_float(r[q]) * inv * src_inv[at];
                j[q] = key;
                const bool in = c0 + q < n_src && x[q] >= tau[at] - 2.4e-7f;
                c[q] = in ? at : -1;
                some |= in;
            }
            if (some) list_edges<8>(c, j, x, reinterpret_cast<const int *>(gen + Sh::src_pos), j0, cnt, reinterpret_cast<Cand *>(gen + Sh::list));
        }
    }
    __syncwarp();
}

// kSample: bounds only, of a sample of the row: the CTAs of a cluster (one unit and NP sources) take sample tiles in turn
// and combine their maxima, each for its share of the sources.
template <int NP, int kD, bool kSample = false>
__global__ void __launch_bounds__(kSimThreads, 1)
similarity_tc(const __grid_constant__ CUtensorMap tmK, SimTcArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const Dims &d = a.d;
    const long long lim = a.wait_cycles;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base - smem_u32(smem_raw));
    using Sh = SimShared<NP, kD>;
    const uint32_t s_stage0 = base + Sh::stage, s_full0 = base + Sh::full, s_empty0 = base + Sh::empty, s_done0 = base + Sh::done;
    const uint32_t s_tmem = base + Sh::tmem;
    float *inv_norm = reinterpret_cast<float *>(gen + Sh::inv_norm);
    int *src_pos = reinterpret_cast<int *>(gen + Sh::src_pos);
    float *src_inv = reinterpret_cast<float *>(gen + Sh::src_inv);
    float *src_norm = reinterpret_cast<float *>(gen + Sh::src_norm);
    float *tau = reinterpret_cast<float *>(gen + Sh::tau);
    int *cnt = reinterpret_cast<int *>(gen + Sh::cnt);
    Cand *list = reinterpret_cast<Cand *>(gen + Sh::list);
    constexpr int kParts = sim_parts<NP>();
    // Tiles whose edges tensor memory holds.  The sampling form, which keeps maxima only, goes round: tile i's place is free once the
    // same warps have given back tile i - 8, that is before tile i is copied (up to eight stages).
    constexpr int kHeld = sim_tiles_cap<NP>();
    static_assert(!kSample || (kHeld % 8 == 0 && NP == 32), "four sets of warps take the tiles in turn");
    float *maxima = reinterpret_cast<float *>(gen + Sh::stage);                 // [NP][kParts] after the sweep
    uint2 *queue = reinterpret_cast<uint2 *>(maxima);                           // [kSimQueue][kSimEpiThreads] after the bounds
    int *failed = reinterpret_cast<int *>(gen + Sh::tmem) + 1;

    PhaseClock pc(threadIdx.x == 64);
    pc.mark();
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int unit = a.unit0 + blockIdx.y, b = unit / d.hkv, h = unit % d.hkv;
    const int chunk = blockIdx.x;
    const int per = a.n_tiles / a.chunks, rem = a.n_tiles % a.chunks;
    const int t0 = chunk * per + min(chunk, rem);
    const int n_local = per + (chunk < rem ? 1 : 0);
    // the sample's tile i, a tile of the chunk
    auto load_tile = [&](int i, int st) {
        const uint32_t dst = s_stage0 + st * tile_bytes<kD>(), bar = s_full0 + 8 * st;
        if constexpr (kSample) {
            mbar_expect_tx(bar, tile_bytes<kD>());
#pragma unroll
            for (int half = 0; half < kD / 64; ++half)
                tma_load_5d(dst + half * kHalfBytes, &tmK, bar, half * 64, 0, (chunk + i * a.chunks) * kSlices, h, b);
        } else {
            tma_load_tile<kD>(dst, &tmK, bar, (t0 + i) * kTileKeys, h, b);
        }
    };
    const __nv_bfloat16 *src_rows = a.S + b * a.ss[0] + (long long)h * a.ss[1];
    // a head with more than NP sources is swept once per NP of them: grid.z counts those sweeps
    const int src0 = blockIdx.z * NP;
    const int *src = a.src + (long long)unit * d.K_src + src0;
    const int n_src = min(NP, d.K_src - src0);               // sources of this CTA

    int n_ahead = 0;                 // tiles thread 0 has requested before the roles split
    if (threadIdx.x == 0) {
        for (int i = 0; i < a.stages; ++i) {
            mbar_init(s_full0 + 8 * i, 1);
            mbar_init(s_empty0 + 8 * i, 1 + (NP == 64 ? 8 : 4));       // MMA commit + the epilogue warps of a tile
        }
        for (int i = 0; i < min(n_local, kHeld); ++i) mbar_init(s_done0 + 8 * i, 1);
        *failed = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmK);
        // the first ring-full of key tiles is under way while the sources are gathered (keys are an
        // input of the call: no wait for the kernels before)
        n_ahead = min(a.stages, n_local);
        for (int i = 0; i < n_ahead; ++i) load_tile(i, i);
    }
    if (warp == 1) {
        tmem_alloc(s_tmem, 512);
        tmem_relinquish();
    }
    pc.mark();
    if (a.wait_prior) pdl_wait();
    pdl_launch_dependents();
    pc.mark();
    // source keys -> swizzled operand rows (rows >= K_src are zero), their positions and norms
    // (kPieces consecutive threads share a row: the row's squared norm is reduced among them)
    constexpr int kPieces = kD / 8;
    for (int i0 = 0; i0 < NP * kPieces; i0 += kSimThreads) {
        const int i = i0 + threadIdx.x;
        const int r = i / kPieces, c16 = i % kPieces;
        const bool in = i < NP * kPieces;
        uint4 v = make_uint4(0, 0, 0, 0);
        int pos = -1;
        if (in && r < n_src) {
            pos = src[r];
            v = *reinterpret_cast<const uint4 *>(src_rows + (long long)pos * a.ss[2] + c16 * 8);
        }
        if (in) *reinterpret_cast<uint4 *>(gen + sw128_offset(NP, r, c16)) = v;
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        float n2 = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float lo = __uint_as_float(w[q] << 16), hi = __uint_as_float(w[q] & 0xffff0000u);
            n2 = fmaf(lo, lo, fmaf(hi, hi, n2));
        }
#pragma unroll
        for (int o = kPieces / 2; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        if (in && c16 == 0) {
            src_pos[r] = pos;
            src_norm[r] = fmaxf(sqrtf(n2), kNormEps);
            src_inv[r] = 1.0f / fmaxf(sqrtf(n2), kNormEps);
            cnt[r] = 0;
        }
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(gen + Sh::tmem), 0);
    bool ok = true;
    pc.mark();

    if (warp == 0) {
        if (lane == 0) {
            int issued = n_ahead;
            for (int i = n_ahead; i < n_local; ++i) {
                const int st = i % a.stages, ph = (i / a.stages) & 1;
                if (!mbar_wait(s_empty0 + 8 * st, ph ^ 1, lim)) { ok = false; break; }
                load_tile(i, st);
                ++issued;
            }
            if (!ok)        // gave up: let the copies already in flight land before the CTA exits
                for (int i = max(0, issued - a.stages); i < issued; ++i)
                    mbar_wait(s_full0 + 8 * (i % a.stages), (i / a.stages) & 1, lim);
        }
    } else if (warp == 1) {
        // (all lanes: see umma_tile)
        constexpr uint32_t idesc = umma_idesc_bf16(128, NP);
        const uint32_t src_lo = umma_desc_lo(base), ring_lo = umma_desc_lo(s_stage0);
        int st = 0;
        uint32_t ph = 0u;
        for (int i = 0; i < n_local; ++i) {
            ok = mbar_wait(s_full0 + 8 * st, ph, lim);
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            tc_fence_after();
            if (elect_one()) {
                umma_tile<kD>(tmem_base + i % kHeld * NP, ring_lo + st * (tile_bytes<kD>() >> 4), kHalfBytes >> 4, src_lo, NP * 128 >> 4, idesc);
                umma_commit(s_empty0 + 8 * st);
                if (!(a.withhold_commit && i == 0)) umma_commit(s_done0 + 8 * (i % kHeld));
            }
            __syncwarp();
            if (++st == a.stages) st = 0, ph ^= 1u;
        }
    } else {
        // ---- epilogue: thread = key (TMEM lane), four sets of four warps.  With 64 sources a set takes 32 of
        // the columns of every second tile, else all columns of every fourth. ----
        constexpr int kCols = NP < 32 ? NP : 32, kColSets = NP / kCols, kTileSets = 4 / kColSets;
        const int quad = warp & 3, set = (warp - 2) >> 2, ew = warp - 2;
        const int key_lane = quad * 32 + lane, et = threadIdx.x - 64;
        const int tile0 = set / kColSets, col0 = (set % kColSets) * kCols;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + col0;
        auto load = [&](int i, uint32_t (&r)[kCols]) {
            if constexpr (kCols == 16) tmem_ld16_issue(lane_addr + i * NP, r);
            else tmem_ld32_issue(lane_addr + i * NP, r);
        };
        {
            float best[kCols];                  // per source: max over this thread's keys of dot / |k_j|
#pragma unroll
            for (int c = 0; c < kCols; ++c) best[c] = -INFINITY;
            for (int i = tile0; i < n_local && ok; i += kTileSets) {
                const int st = i % a.stages, ph = (i / a.stages) & 1;
                // (The MMA of the tile first, on a barrier of its own: a set sees only some of the tiles, so its view
                // of a stage's barrier skips phases, and the parity of a phase it waits for could be an older one's.)
                ok = __all_sync(0xffffffffu, mbar_wait(s_done0 + 8 * (i % kHeld), (i / kHeld) & 1, lim) && mbar_wait(s_full0 + 8 * st, ph, lim));
                if (!ok) break;
                tc_fence_after();
                uint32_t raw[kCols];
                load(i % kHeld, raw);
                // squared norm of this thread's key from the staged tile
                const uint8_t *tile = gen + Sh::stage + st * tile_bytes<kD>();
                float n0 = 0.f, n1 = 0.f;
#pragma unroll
                for (int c16 = 0; c16 < kPieces; ++c16) {
                    const uint4 piece = *reinterpret_cast<const uint4 *>(tile + sw128_offset(128, key_lane, c16));
                    const uint32_t w[4] = {piece.x, piece.y, piece.z, piece.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float lo = __uint_as_float(w[q] << 16), hi = __uint_as_float(w[q] & 0xffff0000u);
                        n0 = fmaf(lo, lo, n0);
                        n1 = fmaf(hi, hi, n1);
                    }
                }
                const int key = i * kTileKeys + key_lane;
                const bool in = (kSample ? ((chunk + i * a.chunks) * kSlices + key_lane / kSliceKeys) * a.slice_step + key_lane % kSliceKeys
                                        : (t0 + i) * kTileKeys + key_lane) < d.N;
                // (a key past the end of the row: NaN, which no comparison and no maximum takes)
                const float inv = in ? 1.0f / fmaxf(sqrtf(n0 + n1), kNormEps) : __int_as_float(0x7fc00000);
                if (!kSample && col0 == 0) inv_norm[key] = inv;
                if constexpr (kSample) tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(s_empty0 + 8 * st);
                tmem_ld_fence(raw);
#pragma unroll
                for (int c = 0; c < kCols; ++c) best[c] = fmaxf(best[c], __uint_as_float(raw[c]) * inv);
            }
            pc.mark();
            // every tile's copies and MMAs are complete once every warp is here: the ring is free
            if (!ok && lane == 0) *failed = 1;
            asm volatile("bar.sync 1, 512;" ::: "memory");
            pc.mark();
#pragma unroll
            for (int c = 0; c < kCols; ++c) maxima[(col0 + c) * kParts + tile0 * 128 + key_lane] = best[c] * src_inv[col0 + c];
        }
        const bool all_ok = *reinterpret_cast<volatile int *>(failed) == 0;
        const int keys = n_local * kTileKeys, j0 = t0 * kTileKeys;
        asm volatile("bar.sync 1, 512;" ::: "memory");
        if (!kSample && all_ok) {
            // 1. bounds
            for (int c = ew; c < n_src; c += 16) {
                const float bound = warp_bound_of_maxima<kParts>(maxima + c * kParts, d.m);
                if (lane == 0) tau[c] = bound;
            }
            if (et == 0) *failed = 0;
            asm volatile("bar.sync 1, 512;" ::: "memory");
            pc.mark();
            // 2. theta is the bound brought to the scale of dot / |k_j|, lowered so that no edge whose cosine rounds up
            //    to the bound is missed
            float theta[kCols];
#pragma unroll
            for (int c = 0; c < kCols; ++c) {
                const float q = col0 + c < n_src ? (tau[col0 + c] - 2.4e-7f) * src_norm[col0 + c] : INFINITY;
                theta[c] = q - fabsf(q) * 3.6e-7f - 1e-30f;
                if (q == -INFINITY) theta[c] = -INFINITY;
            }
            uint2 *const q0 = queue + et;
            const uint32_t q_first = smem_u32(q0), q_step = kSimEpiThreads * sizeof(uint2);
            const uint32_t q_last = q_first + (kSimQueue - 1) * q_step;
            uint32_t qa = q_first;
            for (int i = tile0; i < n_local; i += kTileSets) {
                uint32_t raw[kCols];
                __syncwarp();
                load(i, raw);
                const int key = i * kTileKeys + key_lane;
                const float inv = inv_norm[key];
                tmem_ld_fence(raw);
#pragma unroll
                for (int c = 0; c < kCols; ++c)
                    // (the store and the count under one predicate; the last place takes what does not fit)
                    asm volatile(
                        "{\n\t.reg .pred p;\n\t.reg .u32 a;\n\t"
                        "setp.ge.f32 p, %1, %3;\n\t"
                        "min.u32 a, %0, %4;\n\t"
                        "@p st.shared.v2.b32 [a], {%1, %2};\n\t"
                        "@p add.u32 %0, %0, %5;\n\t}"
                        : "+r"(qa)
                        : "f"(__uint_as_float(raw[c]) * inv), "r"(((uint32_t)(col0 + c) << 16) | (uint32_t)key), "f"(theta[c]),
                          "r"(q_last), "r"(q_step)
                        : "memory");
            }
            pc.mark();
            // 3. lists
            const int queued = static_cast<int>((qa - q_first) / q_step);
            if (__any_sync(0xffffffffu, queued > kSimQueue)) {
                *failed = 1;                                       // a queue has run over
            } else {
#pragma unroll 1
                for (int k = 0; k < queued; k += 4) {
                    int c[4], j[4];
                    float x[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint2 en = q0[min(k + q, kSimQueue - 1) * kSimEpiThreads];
                        const bool in = k + q < queued;
                        c[q] = in ? (int)(en.y >> 16) : -1;
                        j[q] = (int)(en.y & 0xffffu);
                        x[q] = __uint_as_float(en.x) * src_inv[max(c[q], 0)];
                    }
                    list_edges<4>(c, j, x, src_pos, j0, cnt, list);
                }
            }
            __syncwarp();
            asm volatile("bar.sync 1, 512;" ::: "memory");
            if (*reinterpret_cast<volatile int *>(failed) != 0) {
                // keys close to many sources: the lists anew, without queues
                asm volatile("bar.sync 1, 512;" ::: "memory");
                if (et < n_src) cnt[et] = 0;
                asm volatile("bar.sync 1, 512;" ::: "memory");
                list_anew<NP, kD>(gen, tmem_base, n_local, n_src, j0);
                asm volatile("bar.sync 1, 512;" ::: "memory");
            }
            // the sources whose list has overflowed (every warp for itself)
            const unsigned over_lo = __ballot_sync(0xffffffffu, lane < n_src && list_overflowed(cnt, lane));
            const unsigned over_hi = NP < 64 ? 0u : __ballot_sync(0xffffffffu, lane + 32 < n_src && list_overflowed(cnt, lane + 32));
            const unsigned long long over = (unsigned long long)over_hi << 32 | over_lo;
            pc.mark();
            if (over) {
                // 4. ties: cosines in full for 8 or 16 sources at a time, a warp for each source that needs them; the
                //    search starts from the bound
                float *cosines = maxima;                                        // [round][keys]
                const int round = 16 * keys * 4 <= kSimRing ? 16 : 8;
                for (int g0 = 0; g0 < n_src; g0 += round) {
                    if (!(over >> g0 & ((1ull << round) - 1ull))) continue;
                    asm volatile("bar.sync 1, 512;" ::: "memory");
                    for (int i = set; i < n_local; i += 4) {
                        uint32_t r[8];
                        const int key = i * kTileKeys + key_lane;
                        const float inv = inv_norm[key];
                        for (int h8 = 0; h8 < round && g0 + h8 < n_src; h8 += 8) {
                            __syncwarp();
                            tmem_ld8_issue(lane_addr - col0 + i * NP + g0 + h8, r);
                            tmem_ld_fence(r);
#pragma unroll
                            for (int c = 0; c < 8; ++c)
                                if (g0 + h8 + c < n_src) {
                                    const float e = clamped_edge(__uint_as_float(r[c]) * inv * src_inv[g0 + h8 + c]);
                                    cosines[(h8 + c) * keys + key] = j0 + key == src_pos[g0 + h8 + c] ? kCandEmpty : e;
                                }
                        }
                    }
                    asm volatile("bar.sync 1, 512;" ::: "memory");
                    const int c = g0 + ew;
                    if (ew < round && c < n_src && (over >> c & 1ull)) {
                        const float *x = cosines + ew * keys;
                        float bound;
                        const int n = warp_list_top(keys, d.m, fmaxf(tau[c] - 2.4e-7f, -1.0f), [&](int i) { return x[i]; },
                                                    [&](int at, float e, int i) { list[c * kCandCap + at] = Cand{e, j0 + i}; }, &bound);
                        if (lane == 0) cnt[c] = n;
                    }
                    __syncwarp();
                }
                asm volatile("bar.sync 1, 512;" ::: "memory");
            }
            // write the lists out (unused slots marked empty) and count the listed edges per bin
            for (int idx = et; idx < n_src * kCandCap; idx += kSimEpiThreads) {
                const int c = idx / kCandCap, q = idx % kCandCap;
                const long long at = (long long)unit * d.K_src + src0 + c;
                Cand cd{kCandEmpty, -1};
                if (q < cnt[c]) {
                    cd = list[idx];
                    atomicAdd(a.cand_hist + at * kCandBins + cand_bin(cd.e), 1u);
                }
                a.cand[(at * a.chunks + chunk) * kCandCap + q] = cd;
            }
            pc.mark();
        }
        if (!kSample && !all_ok)
            // a wait ran out: publish empty lists so the merge reads nothing undefined
            for (int i = et; i < n_src * kCandCap; i += kSimEpiThreads) {
                const long long slot = ((long long)unit * d.K_src + src0 + i / kCandCap) * a.chunks + chunk;
                a.cand[slot * kCandCap + i % kCandCap] = Cand{kCandEmpty, -1};
            }
        tc_fence_before();
    }
    if (!ok && a.status) atomicExch(a.status, (int)GRAPHKV_ERR_TIMEOUT);
    tc_fence_before();
    if constexpr (kSample) {
        // (where a wait ran out, the maxima are of fewer keys, whose edges reach the bound all the same)
        namespace cg = cooperative_groups;
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();
        if (warp >= 2)
            for (int c = chunk + a.chunks * (warp - 2); c < n_src; c += a.chunks * 16) {
                float *row = maxima + c * kParts;
                float4 x[kParts / 128], y[3][kParts / 128];               // (clusters of up to four: all loads in flight)
#pragma unroll
                for (int q = 0; q < kParts / 128; ++q) x[q] = reinterpret_cast<float4 *>(row)[q * 32 + lane];
#pragma unroll
                for (int p = 0; p < 3; ++p) {
                    const float4 *other = reinterpret_cast<const float4 *>(cl.map_shared_rank(row, (chunk + 1 + min(p, a.chunks - 1)) % a.chunks));
#pragma unroll
                    for (int q = 0; q < kParts / 128; ++q) y[p][q] = other[q * 32 + lane];
                }
#pragma unroll
                for (int q = 0; q < kParts / 128; ++q) {
#pragma unroll
                    for (int p = 0; p < 3; ++p)
                        x[q] = make_float4(fmaxf(x[q].x, y[p][q].x), fmaxf(x[q].y, y[p][q].y), fmaxf(x[q].z, y[p][q].z), fmaxf(x[q].w, y[p][q].w));
                    reinterpret_cast<float4 *>(row)[q * 32 + lane] = x[q];
                }
                __syncwarp();
                const float bound = warp_bound_of_maxima<kParts>(row, d.m);
                if (lane == 0) a.tau[(long long)unit * d.K_src + src0 + c] = bound;
            }
        cl.sync();                              // (nobody leaves while its maxima are read)
    }
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    pc.mark();
    pc.flush(kSample ? 9 : 2);
}

}  // namespace tc
}  // namespace graphkv
