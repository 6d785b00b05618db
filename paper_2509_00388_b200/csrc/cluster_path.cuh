// The whole path in one kernel, for few units with short rows: one cluster of C CTAs (any C up to 16 of which as many
// clusters as units are resident) per (sequence, KV head) unit, each CTA owning a run of key tiles from the first
// score to the gather.
//
// Bound: latency.  At these sizes the four kernels of the general path take 8-20 us each for 1-3 us of
// work: launch, set-up, the first loads, writes that the next kernel reads back, a tail.  Here the key
// tiles come from memory once and stay in shared memory for all three sweeps (which limits the row: four tiles per CTA,
// eight at D = 64), and every CTA holds the unit's row of scores, selects and decays it without asking the others.
// What the CTAs exchange is pushed: the one that has it stores it into the shared memory of those that
// need it (row statistics, masses and neighbour lists into all, the cosines of a source with all keys into the one CTA that picks
// its neighbours), so that an exchange is stores and one cluster barrier (0.3 us); reading from the others after
// the barrier took 1 to 2 us more each time.
//
// Every arithmetic step is the general kernels': the same accumulators, the row statistics folded and
// merged over the same key chunks in the same order (one chunk per CTA), the same pooling, cosines
// and decay order; so the results agree with them to the bit.
// 512 threads; warp 0 issues copies and MMAs between the barriers of the sweeps.
//
// Measured on one B200, 8 KV heads, W = 32, 16 sources (four kernels; this kernel with clusters of 2, 4 or 8 that read from
// one another and per-CTA lists of edges; now): 1003 tokens 43, 31.6, 24.1 us; 2000 tokens 47, 37.1, 28.1; 3000 tokens 53,
// 46.0, 33.0; 4060 tokens 55.6, -, 38.0; 5000 tokens 53.6, -, 44.5; 8191 tokens at D = 64 51.5, -, 46.0.
#pragma once

#include "block_select.cuh"
#include "edge_search.cuh"
#include "row_finish.cuh"
#include "score_simt.cuh"
#include "score_tc.cuh"

namespace graphkv {
namespace cp {

namespace cg = cooperative_groups;
using rf::kThreads;
using rf::kWarps;

constexpr int kMaxCluster = 16;
constexpr int kMaxTiles = 8;            // key tiles per CTA: all of them stay in its shared memory
__host__ __device__ constexpr int max_tiles(int D) { return D == 64 ? kMaxTiles : kMaxTiles / 2; }
constexpr int kMaxSources = 64;
constexpr int kMaxNeighbours = 32;

// Shared memory, from a 1024-byte aligned base.  What is dead is used again: the queries' place holds the source rows
// and, behind them, the unit's scores where they fit; the tiles' place, once the sweeps are over, the unit's
// neighbour lists [k][m] (position, factor) and, at its end, the kept positions [B]; the place of the row statistics
// [C][GW] the cosines [rows][N].  Those come from other CTAs, which do not know whether this one's sweep is over:
// in the tiles' place (behind the lists) they cost one more cluster barrier, so only where they do not fit otherwise.
struct Layout {
    int tiles, lists, mass, row, inv, row_c, parts, cosines, scratch, small, bars, total;
};
constexpr int kScratch = 6656;                  // partial statistics or exchange (4 KB each), histogram, groups' lists
static_assert(kScratch >= 4 * bs::GroupScratch<128>::kBytes && kScratch >= bs::GroupScratch<kThreads>::kBytes &&
                  kScratch >= (bs::kBins + bs::kRankCap) * 4, "scratch");
struct Sizes {                                  // what the layout follows from
    int N, C, GW, tiles, np, rows, lists, kept, cosines_in_tiles;
};
template <int kD, int kTiles> __host__ __device__ inline Layout layout(const Sizes &z)
{
    Layout l;
    const int row = (z.N + 3) / 4 * 16, parts = (z.C * z.GW * 8 + 15) / 16 * 16, queries = 128 * kTiles * 2 * kD;
    const int cosines = z.rows * row, region = z.lists + z.kept + (z.cosines_in_tiles ? cosines : 0);
    int off = queries;
    l.tiles = l.lists = off;
    off += z.tiles * tc::tile_bytes<kD>() > region ? z.tiles * tc::tile_bytes<kD>() : region;
    l.mass = off;    off += row;                // the unit's attention mass before pooling
    l.row = z.np * 2 * kD;                      // the unit's scores
    if (l.row + row > queries) {
        l.row = off;
        off += row;
    }
    l.inv = off;     off += z.tiles * tc::kTileKeys * 4;    // 1 / |k| of this CTA's keys
    l.row_c = off;   off += 2 * 128 * kTiles * 4;
    l.parts = off;
    l.cosines = z.cosines_in_tiles ? l.tiles + z.lists : off;
    off += z.cosines_in_tiles || cosines < parts ? parts : cosines;
    l.scratch = off; off += kScratch;
    l.small = off;   off += 1024;
    l.bars = off;    off += (kMaxTiles + 2) * 8 + 16;
    l.total = off + 1024;
    return l;
}

struct PathArgs {
    Dims d;
    const void *Q, *K;         // bf16 or fp32
    int C;                     // CTAs per unit, and key chunks of the row statistics
    int n_tiles;               // key tiles per unit
    Sizes z;                   // tiles: most key tiles a CTA owns; np: sources padded to 16, 32 or 64; rows: sources whose
                               // cosines a CTA holds at a time; lists, kept: bytes; cosines_in_tiles: they take the tiles' place
    int *status;
    float *scores;             // optional [units][N]: final scores (scores_only: the pooled ones)
    int scores_only;
    int has_graph;
    int *src_out, *nbr_idx;    // [units][K_src], [units][K_src][m]
    float *nbr_e;
    int *idx_out;
    int vpr_log2;              // 16-byte pieces per row: 1 << vpr_log2
    const unsigned char *Kb, *V;
    unsigned char *K_out, *V_out;
    long long wait_cycles;
    int withhold_commit;       // test hook: 1: the first accumulator is never announced
    int per_batch_budget;
    int budget_of[rf::kMaxBudgets];
};

// ---- stores into another CTA of the cluster -----------------------------------------------------
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void peer_store(uint32_t addr, float x)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(x) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t addr, float2 x)
{
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(x.x), "f"(x.y) : "memory");
}

// The small arrays.
struct Small {
    uint32_t *wcnt, *misc;     // [2 * kWarps], [32]
    int *src_pos;              // [kMaxSources]
    float *src_inv;            // [kMaxSources]
    uint32_t *range;           // [2 * kWarps] least and greatest pooled score per warp
    __device__ __forceinline__ explicit Small(uint8_t *p)
        : wcnt(reinterpret_cast<uint32_t *>(p)), misc(wcnt + 2 * kWarps), src_pos(reinterpret_cast<int *>(misc + 32)),
          src_inv(reinterpret_cast<float *>(src_pos + kMaxSources)), range(reinterpret_cast<uint32_t *>(src_inv + kMaxSources)) {}
};

// What follows the masses, in both forms of the kernel: pooling, sources, neighbourhoods, decay, selection and gather.
// kEs: bytes per element.  base: first key of this CTA.  prepare(src_pos): the products of the sources with this CTA's
// keys (sources known, ends with a barrier); push(c0, c1, put): put(c, c / C, c % C, i, cosine) for sources c0 .. c1 and every
// key i of this CTA.
template <int kEs, typename Prepare, typename Push>
__device__ __forceinline__ void finish_path(const PathArgs &a, const Layout &lay, cg::cluster_group &cl, uint8_t *gen, uint32_t base_s,
                                            int base, const bool &alive, PhaseClock &pc, Prepare prepare, Push push)
{
    const Dims &d = a.d;
    const int C = a.C, rank = C > 1 ? (int)cl.block_rank() : 0, unit = blockIdx.x / C, b = unit / d.hkv, h = unit % d.hkv, N = d.N;
    const int tid = threadIdx.x, lane = tid & 31, warp = tc::warp_index();
    const float *mass = reinterpret_cast<const float *>(gen + lay.mass);  // [N] the unit's masses, written by all its CTAs
    float *row = reinterpret_cast<float *>(gen + lay.row);                // [N] the unit's scores, whole
    uint8_t *scratch = gen + lay.scratch;
    uint32_t *hist = reinterpret_cast<uint32_t *>(scratch);
    const Small sm(gen + lay.small);
    uint32_t *wcnt = sm.wcnt, *misc = sm.misc, *range = sm.range;
    int *src_pos = sm.src_pos;
    // ---- the row of masses, which every CTA now has, pooled ----
    auto unit_sync = [&]() { if (C > 1) cl.sync(); else __syncthreads(); };
    unit_sync();
    pc.mark();
    const int half = (d.kp - 1) / 2;
    uint32_t key_lo = 0xffffffffu, key_hi = 0u;
    for (int i = tid; i < N; i += kThreads) {
        float best;
        if (d.pool_avg) {
            best = i >= half ? mass[i - half] : 0.f;
            for (int t = 1 - half; t <= half; ++t) best += i + t >= 0 && i + t < N ? mass[i + t] : 0.f;
            if (d.kp > 1) best /= (float)(2 * half + 1);
        } else {
            best = mass[i];
#pragma unroll 4
            for (int j = max(i - half, 0); j <= min(i + half, N - 1); ++j) best = fmaxf(best, mass[j]);
        }
        row[i] = best;
        key_lo = min(key_lo, float_to_key(best));
        key_hi = max(key_hi, float_to_key(best));
    }
    key_lo = __reduce_min_sync(0xffffffffu, key_lo);
    key_hi = __reduce_max_sync(0xffffffffu, key_hi);
    if (lane == 0) {
        range[warp] = key_lo;
        range[kWarps + warp] = key_hi;
    }
    __syncthreads();
    key_lo = __reduce_min_sync(0xffffffffu, range[lane & (kWarps - 1)]);
    key_hi = __reduce_max_sync(0xffffffffu, range[kWarps + (lane & (kWarps - 1))]);
    const int s0 = (int)((long long)N * rank / C), s1 = (int)((long long)N * (rank + 1) / C);      // this CTA's share of what is written
    if (a.scores_only)
        for (int i = s0 + tid; i < s1; i += kThreads) a.scores[(long long)unit * N + i] = row[i];
    pc.mark();

    uint8_t *region = gen + lay.lists;                                    // once the sweeps are over
    if (a.has_graph && !a.scores_only) {
        // ---- Eq. 2 ----
        const int k = d.K_src;
        auto take = [&](int t, int i) {
            src_pos[t] = i;
            if (rank == 0) a.src_out[(long long)unit * k + t] = i;
        };
        bool found = false;
        if (k <= bs::kTopMax) {
            const bs::GroupScratch<kThreads> gs(scratch);
            found = bs::group_top<kThreads>(row, N, k, 0, tid, gs) <= kThreads;
            if (found && warp == 0) {
                const int pos = lane < k ? rf::position_of(gs.top[lane]) : 0x7fffffff;
                int t = 0;
#pragma unroll
                for (int u = 0; u < 32; ++u) t += __shfl_sync(0xffffffffu, pos, u) < pos;
                if (lane < k) take(t, pos);
            }
        }
        if (!found) {
            const bs::Kept th = bs::block_kth(row, N, (uint32_t)k, key_lo, key_hi, hist, wcnt, misc);
            bs::emit_kept(row, N, th, wcnt, take);
        }
        __syncthreads();
        pc.mark();

        prepare(src_pos);
        pc.mark();

        // ---- Eq. 3: source c belongs to CTA c % C, which gets its cosines with all keys; a.z.rows sources per CTA at a time ----
        const int m = d.m, per_cta = ceil_div(k, C);
        int *nb_j = reinterpret_cast<int *>(region);                                  // [k m] the unit's lists, in every CTA
        float *nb_f = reinterpret_cast<float *>(nb_j + k * m);                        // [k m]
        const float *cosines = reinterpret_cast<const float *>(gen + lay.cosines);    // [rows][row_step]
        const int row_step = (N + 3) & ~3;
        for (int r0 = 0; r0 < per_cta; r0 += a.z.rows) {
            const int c_first = r0 * C, c_last = min(k, (r0 + a.z.rows) * C);
            if (r0 > 0 || a.z.cosines_in_tiles) unit_sync();    // (the round before has been read; nobody reads tiles any more)
            push(c_first, c_last, [&](int c, int slot, int owner, int i, float e) {
                peer_store(peer_addr(base_s + lay.cosines + ((slot - r0) * row_step + base + i) * 4, owner),
                           base + i == src_pos[c] || !alive ? kCandEmpty : e);
            });
            unit_sync();
            pc.mark();
            // the sources' lists, a group of threads each, and each list to all CTAs of the unit
            constexpr int T = 128;
            const int mine = min(a.z.rows, per_cta - r0), gang = tid / T, gt = tid % T;
            const bs::GroupScratch<T> gs(scratch + gang * bs::GroupScratch<T>::kBytes);
            for (int s = gang; s < mine; s += kThreads / T) {
                const int c = (r0 + s) * C + rank;
                if (c >= k) break;
                const float *x = cosines + s * row_step;
                if (bs::group_top<T>(x, N, m, 1 + gang, gt, gs) > T) {
                    // ties: one warp finds exactly the m
                    if (gt < 32) {
                        float reached;
                        const int n = warp_list_top(N, m, -1.0f, [&](int i) { return x[i]; },
                                                    [&](int at, float e, int i) { gs.cand[at] = edge_key(e, i); }, &reached);
                        if (lane == 0) gs.word[0] = (uint32_t)n;
                    }
                    bs::group_bar<T>(1 + gang);
                    bs::group_rank(gs, (int)gs.word[0], m, 1 + gang, gt);
                }
                if (lane < m) {
                    const unsigned long long key = gs.top[lane];
                    const float e = rf::edge_of(key);
                    const bool is = key != 0ull && e >= -1.0f;
                    const int j = is ? rf::position_of(key) : -1;
                    const float f = is ? signal_factor(e, d.lambda, d.T, d.signal) : 1.f;
                    if (gt < 32 && is) {
                        a.nbr_idx[((long long)unit * k + c) * m + lane] = j;
                        a.nbr_e[((long long)unit * k + c) * m + lane] = e;
                    }
                    const uint32_t to = base_s + lay.lists + (c * m + lane) * 4;
                    for (int p = gt >> 5; p < C; p += T / 32) {
                        peer_store(peer_addr(to, p), __int_as_float(j));
                        peer_store(peer_addr(to + k * m * 4, p), f);
                    }
                }
                bs::group_bar<T>(1 + gang);
            }
        }
        unit_sync();
        pc.mark();

        // ---- Eq. 5: every CTA applies the unit's lists to its copy of the row, sources in order ----
        const bool evict = d.signal == GRAPHKV_SIGNAL_EVICT;
        for (int q0 = 0; q0 < k; q0 += 4) {
            int slot[4];
            float f[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool in = lane < m && q0 + u < k;
                slot[u] = in ? nb_j[(q0 + u) * m + lane] : -1;
                f[u] = in ? nb_f[(q0 + u) * m + lane] : 1.f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if ((uint32_t)slot[u] < (uint32_t)N && (slot[u] & (kWarps - 1)) == warp)
                    row[slot[u]] = evict ? -INFINITY : row[slot[u]] * f[u];
                __syncwarp();
            }
        }
        __syncthreads();
        pc.mark();
    }
    if (!a.scores_only) {
        if (a.scores)
            for (int i = s0 + tid; i < s1; i += kThreads) a.scores[(long long)unit * N + i] = row[i];
        // ---- the B largest, in ascending position; a CTA takes its share of them ----
        const int B = a.per_batch_budget ? a.budget_of[b] : d.B;
        const bs::Kept th = bs::block_kth(row, N, (uint32_t)B, key_lo, key_hi, hist, wcnt, misc);
        pc.mark();
        const int first = B * rank / C, count = B * (rank + 1) / C - first;
        int *kept = reinterpret_cast<int *>(region + a.z.lists + (a.z.cosines_in_tiles ? a.z.rows * ((N + 3) / 4 * 16) : 0));         // [count]
        int *idx = a.idx_out + (long long)unit * d.B;
        bs::emit_kept(row, N, th, wcnt, [&](int t, int i) {
            if (t >= first && t < first + count) {
                idx[t] = i;
                kept[t - first] = i;
            }
        });
        __syncthreads();
        pc.mark();
        // ---- gather: the CTA's share of the kept rows and of the window rows ----
        const int vl = a.vpr_log2;
        const unsigned char *k0 = a.Kb + (b * d.ks[0] + h * d.ks[1]) * kEs, *v0 = a.V + (b * d.vs[0] + h * d.vs[1]) * kEs;
        const long long out0 = (long long)unit * (d.B + d.W);
        const int w0 = d.W * rank / C, w1 = d.W * (rank + 1) / C, n_rows = count + (w1 - w0);
        for (int p0 = tid; p0 < n_rows << (vl + 1); p0 += 4 * kThreads) {
            uint4 v[4];
            unsigned char *dst[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = p0 + u * kThreads, t = p >> (vl + 1), c = p & ((1 << vl) - 1);
                dst[u] = nullptr;
                if (t < n_rows) {
                    const bool is_v = (p >> vl) & 1;
                    const int w = w0 + (t - count);
                    const long long from = t < count ? kept[t] : N + w, to = out0 + (t < count ? first + t : B + w);
                    v[u] = *reinterpret_cast<const uint4 *>((is_v ? v0 + from * d.vs[2] * kEs : k0 + from * d.ks[2] * kEs) + c * 16);
                    dst[u] = (is_v ? a.V_out : a.K_out) + ((to << vl) + c) * 16;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (dst[u]) *reinterpret_cast<uint4 *>(dst[u]) = v[u];
        }
    }
}

// kTiles = 1 (G*W <= 128) or 2 (G*W <= 256).  grid = units * C CTAs in clusters of C.
template <int kD, int kTiles>
__global__ void __launch_bounds__(kThreads, 1)
cluster_path_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ PathArgs a)
{
    using namespace tc;
    extern __shared__ uint8_t smem_raw[];
    cg::cluster_group cl = cg::this_cluster();
    constexpr int kRowsPad = 128 * kTiles, kBufCols = 128 * kTiles;
    constexpr int kGroups = 2 / kTiles, kSets = 4 / kGroups, kParts = 4 / kTiles;     // as in the score kernels
    constexpr int kTile = tile_bytes<kD>();
    const Dims &d = a.d;
    const int C = a.C, rank = C > 1 ? (int)cl.block_rank() : 0, unit = blockIdx.x / C;
    const int b = unit / d.hkv, h = unit % d.hkv, N = d.N;
    const int tid = threadIdx.x, lane = tid & 31, warp = tc::warp_index(), quad = warp & 3, set = warp >> 2;
    const long long lim = a.wait_cycles;
    const uint32_t base_s = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base_s - smem_u32(smem_raw));
    const Layout lay = layout<kD, kTiles>(a.z);
    float *inv_norm = reinterpret_cast<float *>(gen + lay.inv);
    float *row_c = reinterpret_cast<float *>(gen + lay.row_c), *row_w = row_c + kRowsPad;
    uint8_t *scratch = gen + lay.scratch;
    float *src_inv = Small(gen + lay.small).src_inv;
    const uint32_t bar_full = base_s + lay.bars, bar_done = bar_full + 8 * kMaxTiles, tmem_slot = bar_done + 16;
    PhaseClock pc(tid == 0);
    pc.mark();
    if (C > 1) cl.barrier_arrive();

    int t0, n_tiles;
    tile_range(a.n_tiles, C, rank, &t0, &n_tiles);
    n_tiles -= t0;
    const int base = t0 * kTileKeys, n_local = max(0, min(N - base, n_tiles * kTileKeys));
    const int n_emit = (n_local + kTileKeys - 1) / kTileKeys;             // tiles with prefix keys

    // ---- set-up: barriers, tensor memory, the first tiles, the queries ----
    auto tile_landed = [&](int t) { return mbar_wait(bar_full + 8 * t, 0, lim); };
    if (tid == 0) {
        for (int i = 0; i < kMaxTiles; ++i) mbar_init(bar_full + 8 * i, 1);
        mbar_init(bar_done, 1);
        mbar_init(bar_done + 8, 1);
        mbar_fence_init();
        tma_prefetch_desc(&tmK);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    // (the launch may be early: nothing of the stream before it, inputs included, is touched ahead of this)
    pdl_wait();
    pdl_launch_dependents();
    if (tid == 0) {
        for (int t = 0; t < n_tiles; ++t)
            tma_load_tile<kD>(base_s + lay.tiles + t * kTile, &tmK, bar_full + 8 * t, (t0 + t) * kTileKeys, h, b);
        if (rank == 0 && unit == 0) *a.status = 0;
    }
    stage_q<kD>(gen, kRowsPad, d, static_cast<const __nv_bfloat16 *>(a.Q), b, h, tid, kThreads);
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (C > 1) cl.barrier_wait();   // (every CTA of the unit has started: its shared memory may be written to)
    const uint32_t tmem = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(gen + (tmem_slot - base_s)), 0);
    const uint32_t tmem_lane = tmem + ((uint32_t)(quad * 32) << 16);
    bool alive = true;              // no wait of this CTA has run out (the same in all its threads)
    int batch = 0;                  // batches of MMAs so far; the announcements alternate between two barriers
    auto batch_done = [&](int bt) { return __all_sync(0xffffffffu, mbar_wait(bar_done + 8 * (bt & 1), (bt >> 1) & 1, lim)) != 0; };
    pc.mark();

    const uint32_t q_lo = umma_desc_lo(base_s), tiles_lo = umma_desc_lo(base_s + lay.tiles);
    // ---- statistics: D = Q K^T, kGroups tiles per batch, two batches under way ----
    const float scale = rsqrtf((float)kD) * kLog2e;
    {
        bool ok = true, issued_ok = true;                                 // (issued_ok: the issuing warp's own waits)
        const int n_batches = ceil_div(n_tiles, kGroups);
        // (by all lanes of warp 0: see umma_tile)
        auto issue = [&](int bt) {
            const int first = bt * kGroups, last = min(first + kGroups, n_tiles);
            for (int t = first; t < last && issued_ok; ++t) issued_ok = __all_sync(0xffffffffu, tile_landed(t));
            if (!issued_ok) return;
            tc_fence_after();
            if (elect_one()) {
                for (int t = first; t < last; ++t)
#pragma unroll
                    for (int rt = 0; rt < kTiles; ++rt)
                        umma_tile<kD>(tmem + ((bt & 1) * kGroups + t - first) * kBufCols + rt * 128, q_lo + rt * (128 * 128 >> 4),
                                      kRowsPad * 128 >> 4, tiles_lo + t * (kTile >> 4), kHalfBytes >> 4, umma_idesc_bf16(128, 128));
                if (!(a.withhold_commit == 1 && bt == 0)) umma_commit(bar_done + 8 * (bt & 1));
            }
            __syncwarp();
        };
        if (warp == 0)
            for (int bt = 0; bt < min(2, n_batches); ++bt) issue(bt);
        const int grp = set / (4 / kGroups), col0 = (set % (4 / kGroups)) * 64, rt = col0 >> 7, key_off = col0 & 127;
        const int r = rt * 128 + quad * 32 + lane, last = N + (r < d.GW ? r % d.W : 0);      // last visible key of the row
        float mx = kNegBig, z = 0.f;
        for (; batch < n_batches && alive; ++batch) {
            const int tile = batch * kGroups + grp;
            ok = batch_done(batch);
            if (ok && tile < n_tiles) {
                tc_fence_after();
                uint32_t raw[2][32];
                const uint32_t from = tmem_lane + ((batch & 1) * kGroups + grp) * kBufCols + col0;
                tmem_ld32_issue(from, raw[0]);
                tmem_ld32_issue(from + 32, raw[1]);
                tmem_ld_fence(raw[0]);
                tmem_ld_fence(raw[1]);
                const int key0 = (t0 + tile) * kTileKeys + key_off;
                const bool masked = key0 + 63 > N;                          // window keys or the tail past L
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    float v[32];
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(raw[c][e]);
                    if (masked) {
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (key0 + c * 32 + e > last) v[e] = -INFINITY;
                    }
                    stats_fold<kD>(v, scale, mx, z);
                }
            }
            tc_fence_before();
            float2 *cta_part = reinterpret_cast<float2 *>(scratch);
            if (batch == n_batches - 1) cta_part[(kTiles == 1 ? set : set & 1) * kRowsPad + r] = make_float2(mx, z);
            alive = __syncthreads_and(ok && issued_ok ? 1 : 0) != 0;
            if (alive && warp == 0 && batch + 2 < n_batches) issue(batch + 2);
        }
        if (alive && tid < d.GW) {
            // the chunk's statistics of this row, to every CTA of the unit
            const float2 *cta_part = reinterpret_cast<const float2 *>(scratch);
            float2 p[kParts];
            float m = kNegBig, sum = 0.f;
#pragma unroll
            for (int k = 0; k < kParts; ++k) {
                p[k] = cta_part[k * kRowsPad + tid];
                m = fmaxf(m, p[k].x);
            }
#pragma unroll
            for (int k = 0; k < kParts; ++k) sum += p[k].y * ex2(p[k].x - m);
            const uint32_t to = base_s + lay.parts + (rank * d.GW + tid) * 8;
            for (int p = 0; p < C; ++p) peer_store(peer_addr(to, p), make_float2(m, sum));
        }
    }
    pc.mark();

    // ---- row constants from all chunks of the unit ----
    if (C > 1) cl.barrier_arrive(); // (this CTA's statistics are with everybody)
    // the keys' norms meanwhile, a warp set per tile
    constexpr int kPieces = kD / 8;
    if (a.has_graph && !a.scores_only && alive) {
        bool ok = true;
        for (int t = set; t < n_emit && ok; t += 4) {
            ok = __all_sync(0xffffffffu, tile_landed(t));
            if (!ok) break;
            const uint8_t *tile = gen + lay.tiles + t * kTile;
            float n0 = 0.f, n1 = 0.f;
#pragma unroll
            for (int c16 = 0; c16 < kPieces; ++c16) {
                const uint4 raw = *reinterpret_cast<const uint4 *>(tile + sw128_offset(128, quad * 32 + lane, c16));
                const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float lo = __uint_as_float(w[q] << 16), hi = __uint_as_float(w[q] & 0xffff0000u);
                    n0 = fmaf(lo, lo, n0);
                    n1 = fmaf(hi, hi, n1);
                }
            }
            inv_norm[t * kTileKeys + quad * 32 + lane] = 1.0f / fmaxf(sqrtf(n0 + n1), kNormEps);
        }
    }
    if (C > 1) cl.barrier_wait();
    else __syncthreads();
    pc.mark();
    {
        constexpr int kTpr = 4 / kTiles;
        static_assert(kRowsPad * kTpr == kThreads, "every thread has a share of a row");
        const int r = tid / kTpr, sub = tid % kTpr;
        const float2 *parts = reinterpret_cast<const float2 *>(gen + lay.parts);
        const float2 mz = merge_row_partials<kTpr>([&](int q) { return parts[q * d.GW + r]; }, C, d.GW, r, sub);
        if (sub == 0) {
            row_c[r] = r < d.GW ? -(weighted<kD>() ? mz.x : mz.x + log2f(mz.y)) : -INFINITY;
            if (weighted<kD>()) row_w[r] = r < d.GW ? 1.0f / mz.y : 0.f;
        }
    }
    __syncthreads();
    pc.mark();

    // ---- emission: D = K Q^T, the prefix tiles from the last to the first ----
    if (alive && n_emit > 0) {
        bool ok = true, issued_ok = true;
        const int n_cols = (d.GW + 31) & ~31, n_batches = ceil_div(n_emit, kGroups), batch0 = batch;
        const uint32_t idesc = umma_idesc_bf16(128, n_cols);
        auto issue = [&](int q) {
            const int bt = batch0 + q, n = min(kGroups, n_emit - q * kGroups), last = n_emit - 1 - q * kGroups;
            for (int g = 0; g < n && issued_ok; ++g) issued_ok = __all_sync(0xffffffffu, tile_landed(last - g));
            if (!issued_ok) return;
            tc_fence_after();
            if (elect_one()) {
                for (int g = 0; g < n; ++g)
                    umma_tile<kD>(tmem + ((bt & 1) * kGroups + g) * kBufCols, tiles_lo + (last - g) * (kTile >> 4), kHalfBytes >> 4, q_lo,
                                  kRowsPad * 128 >> 4, idesc);
                umma_commit(bar_done + 8 * (bt & 1));
            }
            __syncwarp();
        };
        if (warp == 0) {
            issue(0);
            if (n_batches > 1) issue(1);
        }
        const int grp = set / kSets, part = set % kSets;
        const int n_slices = (d.GW + 31) >> 5, s_begin = (part * n_slices) / kSets, s_end = ((part + 1) * n_slices) / kSets;
        const uint64_t scale2 = pack2(scale, scale);
        float *xchg = reinterpret_cast<float *>(scratch);                 // [2][kGroups][kSets][128]
        for (int q = 0; q < n_batches; ++q) {
            ok = batch_done(batch);
            float acc[2] = {0.f, 0.f};
            if (ok && q * kGroups + grp < n_emit) {
                tc_fence_after();
                const uint32_t from = tmem_lane + ((batch & 1) * kGroups + grp) * kBufCols + s_begin * 32;
                uint32_t raw[2][32];
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    if (s_begin + c < s_end) tmem_ld32_issue(from + c * 32, raw[c]);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    if (s_begin + c >= s_end) continue;
                    tmem_ld_fence(raw[c]);
                    float v[32];
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = __uint_as_float(raw[c][e]);
                    const ulonglong2 *c4 = reinterpret_cast<const ulonglong2 *>(row_c + (s_begin + c) * 32);
                    const ulonglong2 *w4 = reinterpret_cast<const ulonglong2 *>(row_w + (s_begin + c) * 32);
                    acc[c] = ex2_sum32<poly_pairs<kD>(), weighted<kD>()>(v, scale2, [&](int i) { return c4[i]; },
                                                                         [&](int i) { return w4[i]; });
                }
            }
            float *x = xchg + (batch & 1) * (4 * 128);
            x[(grp * kSets + part) * 128 + quad * 32 + lane] = s_end - s_begin == 2 ? acc[0] + acc[1] : acc[0];
            tc_fence_before();
            alive = __syncthreads_and(ok && issued_ok ? 1 : 0) != 0;
            if (!alive) break;
            if (warp == 0 && q + 2 < n_batches) issue(q + 2);
            if (tid < kGroups * 128 && q * kGroups + tid / 128 < n_emit) {
                const int t = n_emit - 1 - (q * kGroups + tid / 128), key = tid & 127;
                const float *xs = x + (tid / 128) * kSets * 128 + key;
                const float aj = kSets == 4 ? (xs[0] + xs[128]) + (xs[256] + xs[384]) : xs[0] + xs[128];
                const uint32_t to = base_s + lay.mass + (base + t * kTileKeys + key) * 4;
                if (t * kTileKeys + key < n_local)
                    for (int p = 0; p < C; ++p) peer_store(peer_addr(to, p), aj);
            }
            ++batch;
        }
    }
    if (!alive) {
        // a wait ran out: no scores, and the copies still under way land before their place is used again
        for (int i = tid; i < n_local; i += kThreads)
            for (int p = 0; p < C; ++p) peer_store(peer_addr(base_s + lay.mass + (base + i) * 4, p), 0.f);
        if (tid == 0)
            for (int t = 0; t < n_tiles; ++t) tile_landed(t);
    }
    pc.mark();

    finish_path<2>(a, lay, cl, gen, base_s, base, alive, pc, [&](const int *src_pos) {
        // ---- Eq. 1: the sources' rows as an operand, all tiles against them ----
        const int np = a.z.np, k = d.K_src;
        const __nv_bfloat16 *Kh = static_cast<const __nv_bfloat16 *>(a.K) + b * d.ks[0] + (long long)h * d.ks[1];
        for (int i = tid; i < np * kPieces; i += kThreads) {
            const int r = i / kPieces, c16 = i % kPieces;
            uint4 v = make_uint4(0, 0, 0, 0);
            if (r < k) v = *reinterpret_cast<const uint4 *>(Kh + (long long)src_pos[r] * d.ks[2] + c16 * 8);
            *reinterpret_cast<uint4 *>(gen + sw128_offset(np, r, c16)) = v;
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            float n2 = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float lo = __uint_as_float(w[q] << 16), hi = __uint_as_float(w[q] & 0xffff0000u);
                n2 = fmaf(lo, lo, fmaf(hi, hi, n2));
            }
#pragma unroll
            for (int o = kPieces / 2; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
            if (c16 == 0) src_inv[r] = 1.0f / fmaxf(sqrtf(n2), kNormEps);
        }
        fence_proxy_async();
        __syncthreads();
        bool ok = true;
        if (n_emit > 0 && alive) {
            if (warp == 0) {
                tc_fence_after();
                if (elect_one()) {
                    for (int t = 0; t < n_emit; ++t)
                        umma_tile<kD>(tmem + t * np, tiles_lo + t * (kTile >> 4), kHalfBytes >> 4, q_lo, np * 128 >> 4, umma_idesc_bf16(128, np));
                    umma_commit(bar_done + 8 * (batch & 1));
                }
                __syncwarp();
            }
            ok = batch_done(batch);
            tc_fence_before();
            alive = __syncthreads_and(ok ? 1 : 0) != 0;
            ++batch;
        }
        tc_fence_after();
    }, [&](int c_first, int c_last, auto put) {
        for (int t = set; t < n_emit; t += 4) {
            const int i = t * kTileKeys + quad * 32 + lane;
            const float inv = inv_norm[i];
            int slot = (c_first & ~7) / C, owner = (c_first & ~7) - slot * C;
            for (int g0 = c_first & ~7; g0 < c_last; g0 += 8) {
                uint32_t raw[8];
                __syncwarp();
                tmem_ld8_issue(tmem_lane + t * a.z.np + g0, raw);
                tmem_ld_fence(raw);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int c = g0 + q;
                    if (c >= c_first && c < c_last && i < n_local)
                        put(c, slot, owner, i, fminf(fmaxf(__uint_as_float(raw[q]) * inv * src_inv[c], -1.0f), 1.0f));
                    if (++owner == C) owner = 0, ++slot;
                }
            }
        }
        tc_fence_before();
    });
    pc.mark();
    if (!alive && tid == 0) atomicExch(a.status, (int)GRAPHKV_ERR_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
    pc.flush(7);
}

// ---- fp32 rows ------------------------------------------------------------------------------------
// The same path with the products on the FMA pipe (simt_dots, so that cosines have the bits of the general fp32 sweep):
// a CTA owns 128 keys, its 16 warps two halves of 64 keys, or, where clusters of that many CTAs are resident, 64 keys, its
// warps two halves of the query rows; a thread's products of queries and keys stay in registers from the row statistics
// to the masses, so they are computed once.  kR times 16 rows per row tile, kRowTiles of them.  (One head of 512 keys: six launches
// 38.3 us, 128 keys per CTA 25.7, 64 keys 21.)
template <int kD> __host__ __device__ inline Layout layout_f32(const Sizes &z)
{
    Layout l{};
    const int row = (z.N + 3) / 4 * 16, parts = (z.tiles * z.C * z.GW * 8 + 15) / 16 * 16, cosines = z.rows * row;
    const int rows = z.GW <= 32 ? 32 : z.GW <= 64 ? 64 : 128, step = (kD + 4) * 4;
    int off = (rows > z.np ? rows : z.np) * step;       // the queries [kRows][kD + 4]; then the sources' unit vectors
    l.tiles = off;   off += z.tiles * 64 * step;        // the keys [64 or 128][kD + 4]
    l.lists = off;   off += z.lists + z.kept;
    l.mass = off;    off += row;
    l.row = off;     off += row;
    l.inv = off;     off += tc::kTileKeys * 4;
    l.row_c = off;   off += 2 * 128 * 4;
    l.parts = l.cosines = off;
    off += cosines > parts ? cosines : parts;           // row statistics [2 C][GW]; then cosines [rows][N]
    l.scratch = off; off += kScratch;
    l.small = off;   off += 1024;
    l.bars = off;
    l.total = off;
    return l;
}

template <int kD, int kR, int kRowTiles, int kKeys>
__global__ void __launch_bounds__(kThreads, 1) cluster_path_f32_kernel(const __grid_constant__ PathArgs a)
{
    extern __shared__ __align__(16) uint8_t path_smem[];
    cg::cluster_group cl = cg::this_cluster();
    constexpr int kStep = kD + 4, kHalfRows = 16 * kR * kRowTiles, kRows = kKeys == 64 ? 2 * kHalfRows : kHalfRows, kPieces = kD / 4;
    constexpr int kParts = kKeys / 64;          // partial statistics per row and CTA
    static_assert(kRows <= 128 && (kKeys == 64 || kKeys == 128), "four threads per row");
    const Dims &d = a.d;
    const int C = a.C, rank = C > 1 ? (int)cl.block_rank() : 0, unit = blockIdx.x / C;
    const int b = unit / d.hkv, h = unit % d.hkv, N = d.N;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, half = warp >> 3, kh = kKeys == 128 ? half : 0, rh = kKeys == 64 ? half : 0, kg = lane & 15, rg = (warp & 7) * 2 + (lane >> 4);
    uint8_t *gen = path_smem;
    const uint32_t base_s = tc::smem_u32(path_smem);
    const Layout lay = layout_f32<kD>(a.z);
    float *rows = reinterpret_cast<float *>(gen), *keys = reinterpret_cast<float *>(gen + lay.tiles);
    float *inv_norm = reinterpret_cast<float *>(gen + lay.inv);
    float *row_mx = reinterpret_cast<float *>(gen + lay.row_c), *row_w = row_mx + 128;
    float *xchg = reinterpret_cast<float *>(gen + lay.scratch);           // [kWarps][64]
    const int base = rank * kKeys, n_local = max(0, min(N - base, kKeys));
    const float *Q = static_cast<const float *>(a.Q);
    const float *Kh = static_cast<const float *>(a.K) + b * d.ks[0] + (long long)h * d.ks[1];
    const bool alive = true;                                              // (no wait here can run out)
    PhaseClock pc(tid == 0);
    pc.mark();
    if (C > 1) cl.barrier_arrive();
    pdl_wait();
    pdl_launch_dependents();
    if (tid == 0 && rank == 0 && unit == 0) *a.status = 0;
#pragma unroll 8
    for (int i = tid; i < kKeys * kPieces; i += kThreads) {
        const int r = i / kPieces, c = i % kPieces;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (base + r < d.L) v = *reinterpret_cast<const float4 *>(Kh + (long long)(base + r) * d.ks[2] + c * 4);
        *reinterpret_cast<float4 *>(keys + r * kStep + c * 4) = v;
    }
    const float scale = rsqrtf((float)kD) * kLog2e;
#pragma unroll 4
    for (int i = tid; i < kRows * kPieces; i += kThreads) {
        const int r = i / kPieces, c = i % kPieces;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < d.GW) v = *reinterpret_cast<const float4 *>(Q + b * d.qs[0] + (long long)(h * d.G + r / d.W) * d.qs[1] + (r % d.W) * d.qs[2] + c * 4);
        *reinterpret_cast<float4 *>(rows + r * kStep + c * 4) = make_float4(v.x * scale, v.y * scale, v.z * scale, v.w * scale);
    }
    __syncthreads();
    if (C > 1) cl.barrier_wait();               // (every CTA of the unit has started: its shared memory may be written to)
    pc.mark();

    // ---- logits, and the row statistics of each half ----
    const float *mine = keys + kh * 64 * kStep;
    const int row0 = rh * kHalfRows;
    float l2[kRowTiles][kR][4];
#pragma unroll
    for (int rt = 0; rt < kRowTiles; ++rt) simt_dots<kD, kR>(rows + (row0 + rt * 16 * kR) * kStep, mine, rg, kg, l2[rt]);
    pc.mark();
#pragma unroll
    for (int rt = 0; rt < kRowTiles; ++rt)
#pragma unroll
        for (int i = 0; i < kR; ++i) {
            const int r = row0 + rt * 16 * kR + rg + 16 * i, last = N + (r < d.GW ? r % d.W : 0);     // last visible key of the row
            float m = kNegBig;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (base + kh * 64 + kg + 16 * e > last) l2[rt][i][e] = -INFINITY;
                m = fmaxf(m, l2[rt][i][e]);
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            float z = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) z += exp2f(l2[rt][i][e] - m);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
            if (r < d.GW)                                                 // (the 16 lanes of a row share the CTAs)
                for (int p = kg; p < C; p += 16)
                    peer_store(peer_addr(base_s + lay.parts + ((rank * kParts + kh) * d.GW + r) * 8, p), make_float2(m, z));
        }
    if (C > 1) cl.barrier_arrive();
    if (a.has_graph && !a.scores_only && tid < kKeys) {
        // the keys' norms meanwhile
        const float4 *k4 = reinterpret_cast<const float4 *>(keys + tid * kStep);
        float n2 = 0.f;
#pragma unroll 8
        for (int c = 0; c < kPieces; ++c) {
            const float4 v = k4[c];
            n2 = fmaf(v.x, v.x, n2); n2 = fmaf(v.y, v.y, n2); n2 = fmaf(v.z, v.z, n2); n2 = fmaf(v.w, v.w, n2);
        }
        inv_norm[tid] = 1.0f / fmaxf(sqrtf(n2), kNormEps);
    }
    if (C > 1) cl.barrier_wait();
    else __syncthreads();
    pc.mark();
    // ---- row constants, four threads a row ----
    {
        const int r = tid >> 2, sub = tid & 3;
        const float2 *parts = reinterpret_cast<const float2 *>(gen + lay.parts);
        float m = kNegBig, z = 0.f;
        if (r < d.GW) {
            for (int q = sub; q < kParts * C; q += 4) m = fmaxf(m, parts[q * d.GW + r].x);
        }
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        if (r < d.GW) {
            for (int q = sub; q < kParts * C; q += 4) z = fmaf(parts[q * d.GW + r].y, exp2f(parts[q * d.GW + r].x - m), z);
        }
        z += __shfl_xor_sync(0xffffffffu, z, 1);
        z += __shfl_xor_sync(0xffffffffu, z, 2);
        if (sub == 0 && r < kRows) {
            row_mx[r] = r < d.GW ? m : 0.f;
            row_w[r] = r < d.GW ? 1.0f / z : 0.f;
        }
    }
    __syncthreads();
    pc.mark();
    // ---- masses ----
    {
        float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int rt = 0; rt < kRowTiles; ++rt)
#pragma unroll
            for (int i = 0; i < kR; ++i) {
                const int r = row0 + rt * 16 * kR + rg + 16 * i;
                const float m = row_mx[r], w = row_w[r];
#pragma unroll
                for (int e = 0; e < 4; ++e) s[e] = fmaf(exp2f(l2[rt][i][e] - m), w, s[e]);
            }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            s[e] += __shfl_xor_sync(0xffffffffu, s[e], 16);
            if (lane < 16) xchg[warp * 64 + kg + 16 * e] = s[e];
        }
        __syncthreads();
        if (tid < n_local) {
            const float *x = xchg + (tid >> 6) * (8 * 64) + (tid & 63);
            float sum = 0.f;
#pragma unroll
            for (int w = 0; w < 16 / kParts; ++w) sum += x[w * 64];
            for (int p = 0; p < C; ++p) peer_store(peer_addr(base_s + lay.mass + (base + tid) * 4, p), sum);
        }
    }
    pc.mark();
    finish_path<4>(a, lay, cl, gen, base_s, base, alive, pc, [&](const int *src_pos) {
        // ---- Eq. 1: the sources' unit vectors, a warp each ----
        for (int c = warp; c < a.z.np; c += kWarps) {
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (c < d.K_src && lane * 4 < kD) {
                const float4 raw = *reinterpret_cast<const float4 *>(Kh + (long long)src_pos[c] * d.ks[2] + lane * 4);
                v[0] = raw.x; v[1] = raw.y; v[2] = raw.z; v[3] = raw.w;
            }
            simt_unit_row(v);
            if (lane * 4 < kD) *reinterpret_cast<float4 *>(rows + c * kStep + lane * 4) = make_float4(v[0], v[1], v[2], v[3]);
        }
        __syncthreads();
    }, [&](int c_first, int c_last, auto put) {
        for (int a0 = (c_first & ~15) + 16 * rh; a0 < c_last; a0 += kKeys == 64 ? 32 : 16) {
            float dot[1][4];
            simt_dots<kD, 1>(rows + a0 * kStep, mine, rg, kg, dot);
            const int c = a0 + rg, slot = c / C;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = kh * 64 + kg + 16 * e;
                if (c >= c_first && c < c_last && i < n_local)
                    put(c, slot, c - slot * C, i, fminf(fmaxf(dot[0][e] * inv_norm[i], -1.0f), 1.0f));
            }
        }
    });
    pc.mark();
    pc.flush(7);
}

}  // namespace cp
}  // namespace graphkv
