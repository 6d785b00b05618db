// The last kernel of a call: the neighbourhoods of Eq. 3 merged from the candidate lists of the
// similarity sweep, the decay rounds of Eq. 5 / Algorithm 2 over them, the final k_l selection and
// the gather of the compact cache.  One cluster of C CTAs per unit.
//
// Bound: latency.  The row has up to 262144 scores, but only few of them can be kept or change:
// with P listed edges at most P positions lose score, so the kept ones lie among the B + P highest
// scores as they were before.  So
//   1. the digit (top 11 bits of the ordered image) that holds the (B + P)-th largest comes from a
//      histogram of the row, which the pooling kernel leaves behind or the cluster counts here
//      (further digits only if too many elements tie in it);
//   2. every CTA writes one bit per element, "reaches that digit", into the first CTA's shared memory;
//   3. the other CTAs merge neighbour lists, sources spread over their warps, and push them to the
//      first, which meanwhile expands the bits into position-ordered candidates and fetches their scores;
//   4. the first CTA applies the decay and selects the B largest (one more histogram over the few
//      digits they can lie in, the rest ranked by counting), the others copy the window rows;
//   5. all CTAs gather.
// Steps 1 and 2 need nothing of the similarity sweep and run ahead of the wait for it.  A short row is
// all candidates: no histogram, no bits.  Three to five cluster barriers in all (about 0.35 us each),
// and no pass over the row after step 2.  Code that runs once pays for its instruction fetches, so
// loops are kept rolled.  512 threads: barriers at half the price of 1024, and two CTAs per SM, so
// that one gathers while the other selects when there are more units than SMs.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "block_select.cuh"

namespace graphkv {
namespace rf {

namespace cg = cooperative_groups;

constexpr int kThreads = bs::kThreads;      // 512
constexpr int kWarps = kThreads / 32;
constexpr int kMaxCluster = 8;
constexpr int kBins = 2048;
constexpr int kSurvCap = 256;           // merged candidates a group ranks in shared memory
constexpr int kMaxRow = 262144;         // scores per row
constexpr int kMaxBudgets = 64;         // batch elements with a budget of their own per launch
constexpr int kScratch = kWarps * kSurvCap * 8;     // bytes: histograms, the merges' survivors, the ranking's lists
static_assert(kScratch >= 2 * kBins * 4, "two histograms");

struct FinishArgs {
    Dims d;
    int C;                     // CTAs per cluster (one cluster per unit)
    int chunk;                 // elements of the row per CTA (a multiple of 32)
    int dense;                 // every element of the row is a candidate
    int cap;                   // candidates the first CTA holds
    int sel_cap;               // of them, for elements that reach the threshold (the others: listed positions)
    int list_bytes;            // bytes of the neighbour lists (8 per edge) or of the kept positions, whichever is more
    int group_warps;           // warps that merge one source's lists: 1, 2 or 4
    const uint32_t *row_hist;  // optional [units][kBins]: the rows' elements per digit
    float *s;                  // [units][N] scores; decayed ones are written back when keep_scores
    int *nbr_idx;              // [units][K_src][m] neighbour lists (has_graph); written when merging
    float *nbr_e;              // [units][K_src][m] their cosines
    int has_graph;             // apply the decay rounds
    int merge;                 // build the neighbour lists from the per-chunk candidate lists first
    const Cand *cand;          // [units][K_src][cand_chunks][kCandCap]
    const uint32_t *cand_hist; // [units][K_src][kCandBins]
    int cand_chunks;
    int do_select;             // pick the budget and gather
    int *idx_out;              // [units][B]
    int elem_bytes, vpr_log2;  // 16-byte pieces per row: 1 << vpr_log2
    const unsigned char *K, *V;
    unsigned char *K_out, *V_out;
    int wait_prior;            // launched with programmatic stream serialization
    int early_row;             // the scores are complete when this kernel starts (the kernel before has waited for
                               // theirs), so that only the neighbour lists need the wait
    int keep_scores;           // write the decayed scores back to `s` (0: nobody reads them)
    int per_batch_budget;      // budgets differ per batch element: budget_of[unit / hkv] (d.B: output rows)
    int budget_of[kMaxBudgets];
};

__host__ __device__ inline int row_words(int N) { return (N + 31) / 32; }

// Dynamic shared memory: scratch | candidate keys, positions | lists | bits, their prefix sums | words
__host__ __device__ inline size_t smem_bytes(int N, int cap, int list_bytes, bool dense)
{
    return (size_t)kScratch + (size_t)cap * 8 + list_bytes + (dense ? 0 : (size_t)row_words(N) * 12) + 256;
}

struct Smem {
    uint32_t *hist, *tot;      // [kBins] each, in the scratch
    float *val;                // [cap] candidates' scores
    int *pos;                  // [cap] their positions (unused when dense)
    int *nb_j;                 // [K_src * m] listed positions, then candidate slots
    float *nb_f;               // [K_src * m] factors over all rounds
    int *kept;                 // [B] kept positions (takes the lists' place)
    uint32_t *bits, *ties, *before;   // [row_words] (not when dense)
    uint32_t *wcnt;            // [2 * kWarps]
    uint32_t *misc;            // [16]
};

// Exclusive prefix of v over the CTA's threads; *total: the sum.  One barrier; `wcnt` is free again
// after the caller's next barrier.
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t *wcnt, uint32_t *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t incl = bs::incl_scan(v, lane);
    if (lane == 31) wcnt[warp] = incl;
    __syncthreads();
    const uint32_t w = lane < kWarps ? wcnt[lane] : 0u;
    *total = __reduce_add_sync(0xffffffffu, w);
    return incl - v + __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
}

// The digit (of `nb` counted in `hist`, the largest first) that holds the `need`-th element:
// misc[0] = digit, misc[1] = elements above it, misc[2] = elements in it; misc[6] = the digit that holds
// the `need2`-th.  Ends with a barrier.
__device__ __forceinline__ void find_digit(const uint32_t *hist, int nb, uint32_t need, uint32_t *wcnt, uint32_t *misc,
                                           uint32_t need2 = 0)
{
    const int per = nb / kThreads;
    const int top = nb - 1 - (int)threadIdx.x * per;
    uint32_t sum = 0, total;
    for (int q = 0; q < per; ++q) sum += hist[top - q];
    uint32_t run = block_exclusive(sum, wcnt, &total);
    if (run < need2 && run + sum >= need2) {
        uint32_t r2 = run;
        for (int q = 0; q < per; ++q) {
            r2 += hist[top - q];
            if (r2 >= need2) {
                misc[6] = (uint32_t)(top - q);
                break;
            }
        }
    }
    if (run < need && run + sum >= need) {
        for (int q = 0; q < per; ++q) {
            const uint32_t c = hist[top - q];
            if (run + c >= need) {
                misc[0] = (uint32_t)(top - q);
                misc[1] = run;
                misc[2] = c;
                break;
            }
            run += c;
        }
    }
    __syncthreads();
}

// Counts `bin` of every lane with `valid` (lanes that share a bin with one addition).
__device__ __forceinline__ void count_bin(uint32_t *hist, uint32_t bin, bool valid)
{
    const uint32_t key = valid ? bin : 0xffffffffu;
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    if (valid && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&hist[bin], (uint32_t)__popc(peers));
}

__device__ __forceinline__ int digit_shift(int pass) { return pass <= 0 ? 21 : pass == 1 ? 10 : 0; }
__device__ __forceinline__ int digit_count(int pass) { return pass == 2 ? 1024 : 2048; }

__device__ __forceinline__ void group_bar(int id, int threads)
{
    if (threads == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ float edge_of(unsigned long long key)
{
    const uint32_t u = (uint32_t)(key >> 32);
    return __uint_as_float((u & 0x80000000u) ? (u ^ 0x80000000u) : ~u);
}
__device__ __forceinline__ int position_of(unsigned long long key) { return (int)(0xffffffffu - (uint32_t)key); }

// Survivors of the lists when more than kSurvCap edges reach the bound (ties): the exact m-th
// largest 64-bit edge key (keys are distinct) by a byte-wise radix search over the lists, then the
// edges that reach it.  `surv` (also the search's scratch) and *count as in merge_source.
__device__ __noinline__ void merge_exact(const unsigned long long *cand, int slots, int m, unsigned long long *surv,
                                         uint32_t *count, int bar_id, int threads, int t)
{
    uint32_t *rh = reinterpret_cast<uint32_t *>(surv);          // [256] counts, [2] result
    const int lane = threadIdx.x & 31;
    unsigned long long t64 = 0ull;
    uint32_t remaining = (uint32_t)m;
    for (int byte = 7; byte >= 0; --byte) {
        const unsigned long long hi_mask = byte == 7 ? 0ull : ~0ull << (8 * (byte + 1));
        for (int i = t; i < 256; i += threads) rh[i] = 0u;
        group_bar(bar_id, threads);
        for (int i0 = 0; i0 < slots; i0 += threads) {
            const int i = i0 + t;
            bool valid = false;
            uint32_t bin = 0;
            if (i < slots) {
                const unsigned long long raw = __ldcg(cand + i);
                const float e = __uint_as_float((uint32_t)raw);
                const unsigned long long key = edge_key(e, (int)(raw >> 32));
                valid = e >= -1.0f && (key & hi_mask) == t64;
                bin = (uint32_t)(key >> (8 * byte)) & 0xffu;
            }
            count_bin(rh, bin, valid);
        }
        group_bar(bar_id, threads);
        if (t < 32) {
            // lane l holds digits 255 - 8 l - q (q < 8)
            uint32_t sum = 0;
            for (int q = 0; q < 8; ++q) sum += rh[255 - 8 * lane - q];
            uint32_t run = bs::incl_scan(sum, lane) - sum;
            if (lane == 0) {
                rh[256] = 0u;                                   // fewer edges than m: all are kept
                rh[257] = remaining;
            }
            __syncwarp();
            if (run < remaining && run + sum >= remaining) {
                for (int q = 0; q < 8; ++q) {
                    const uint32_t c = rh[255 - 8 * lane - q];
                    if (run + c >= remaining) {
                        rh[256] = (uint32_t)(255 - 8 * lane - q);
                        rh[257] = remaining - run;
                        break;
                    }
                    run += c;
                }
            }
        }
        group_bar(bar_id, threads);
        t64 |= (unsigned long long)rh[256] << (8 * byte);
        remaining = rh[257];
        group_bar(bar_id, threads);
    }
    if (t == 0) *count = 0u;
    group_bar(bar_id, threads);
    for (int i0 = 0; i0 < slots; i0 += threads) {
        const int i = i0 + t;
        if (i < slots) {
            const unsigned long long raw = __ldcg(cand + i);
            const float e = __uint_as_float((uint32_t)raw);
            const unsigned long long key = edge_key(e, (int)(raw >> 32));
            if (e >= -1.0f && key >= t64) {
                const uint32_t p = atomicAdd(count, 1u);
                if (p < (uint32_t)kSurvCap) surv[p] = key;
            }
        }
    }
    group_bar(bar_id, threads);
}

// Eq. 3 for one source: the m largest edges (cosine descending, position ascending) among the lists
// its key chunks wrote, which together hold every member of the top-m.  `hist` counts the listed
// edges per cosine bin: the highest bin b with m listed edges in bins >= b bounds the m-th largest
// from below, so only edges with e >= b / kCandBins are ranked.  A group of `threads` threads (t: this
// one's number); `surv`: kSurvCap words, `count`: one word of shared memory of the group.
// The list goes to nbr_idx / nbr_e and, as (position, factor over all rounds), to nb_j / nb_f.
__device__ __forceinline__ void merge_source(const Dims &d, const Cand *cand_in, const uint32_t *hist, int slots,
                                             unsigned long long *surv, uint32_t *count, int bar_id, int threads, int t,
                                             int *nbr_idx, float *nbr_e, int *nb_j, float *nb_f)
{
    const unsigned long long *cand = reinterpret_cast<const unsigned long long *>(cand_in);
    const int lane = threadIdx.x & 31;
    // the counts and the first slots are requested together (eight slots per thread in flight: a round of loads
    // costs about a microsecond, four at a time it was 18 us for 154 sources of 1152 slots)
    constexpr int kAhead = 8;
    unsigned long long raw[kAhead];
#pragma unroll
    for (int q = 0; q < kAhead; ++q) raw[q] = q * threads + t < slots ? __ldcg(cand + q * threads + t) : 0ull;
    uint32_t h[8];
    *reinterpret_cast<uint4 *>(h) = __ldcg(reinterpret_cast<const uint4 *>(hist) + lane * 2);
    *reinterpret_cast<uint4 *>(h + 4) = __ldcg(reinterpret_cast<const uint4 *>(hist) + lane * 2 + 1);
    if (t == 0) *count = 0u;
    uint32_t mine = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) mine += h[q];
    const uint32_t up_to = bs::incl_scan(mine, lane), total = __shfl_sync(0xffffffffu, up_to, 31);
    uint32_t run = total - up_to;               // listed edges in the bins above this lane's
    int bstar = -1;
#pragma unroll
    for (int q = 7; q >= 0; --q) {
        run += h[q];
        if (bstar < 0 && run >= (uint32_t)d.m) bstar = lane * 8 + q;
    }
    bstar = __reduce_max_sync(0xffffffffu, bstar);
    const float bound = bstar <= 0 ? -1.0f : (float)bstar / (float)kCandBins;
    group_bar(bar_id, threads);
    for (int i0 = 0; i0 < slots; i0 += kAhead * threads) {
        if (i0 > 0) {
#pragma unroll
            for (int q = 0; q < kAhead; ++q) {
                const int i = i0 + q * threads + t;
                raw[q] = i < slots ? __ldcg(cand + i) : 0ull;
            }
        }
        // (one place-taking addition for all eight: each is a chain of about 100 clocks)
        unsigned kept[kAhead];
        uint32_t n = 0;
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            const float e = __uint_as_float((uint32_t)raw[q]);
            kept[q] = __ballot_sync(0xffffffffu, i0 + q * threads + t < slots && e >= bound);
            n += __popc(kept[q]);
        }
        if (n == 0) continue;
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(count, n);
        base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
        for (int q = 0; q < kAhead; ++q) {
            const uint32_t at = base + __popc(kept[q] & ((1u << lane) - 1u));
            if (((kept[q] >> lane) & 1u) && at < (uint32_t)kSurvCap)
                surv[at] = edge_key(__uint_as_float((uint32_t)raw[q]), (int)(raw[q] >> 32));
            base += __popc(kept[q]);
        }
    }
    group_bar(bar_id, threads);
    int ns = (int)*count;
    if (ns > kSurvCap) {
        merge_exact(cand, slots, d.m, surv, count, bar_id, threads, t);
        ns = min((int)*count, kSurvCap);
    }
    // rank by counting: 1, 2 or 4 neighbouring threads per edge
    const int share = ns * 4 <= threads ? 4 : ns * 2 <= threads ? 2 : 1, sub = t & (share - 1);
    for (int i0 = 0; i0 < ns; i0 += threads / share) {
        const int i = i0 + t / share;
        const unsigned long long me = i < ns ? surv[i] : ~0ull;
        int rank = 0;
#pragma unroll 4
        for (int u = sub; u < ns; u += share) rank += surv[u] > me;
        if (share > 1) rank += __shfl_xor_sync(0xffffffffu, rank, 1);
        if (share > 2) rank += __shfl_xor_sync(0xffffffffu, rank, 2);
        if (i < ns && sub == 0 && rank < d.m) {
            const int j = position_of(me);
            const float e = edge_of(me);
            nbr_idx[rank] = j;
            nbr_e[rank] = e;
            nb_j[rank] = j;
            nb_f[rank] = signal_factor(e, d.lambda, d.T, d.signal);
        }
    }
    for (int u = ns + t; u < d.m; u += threads) nb_j[u] = -1;
    group_bar(bar_id, threads);                  // the survivors' words may be reused
}

// grid = units * C CTAs in clusters of C; block kThreads.
__global__ void __launch_bounds__(kThreads, 2) finish_kernel(FinishArgs a)
{
    extern __shared__ __align__(16) uint8_t rf_smem[];
    cg::cluster_group cl = cg::this_cluster();
    const Dims &d = a.d;
    const int C = a.C, rank = C > 1 ? (int)cl.block_rank() : 0;
    const int unit = (gridDim.x - 1 - blockIdx.x) / C;   // the last units first: their keys are still in L2
    const int N = d.N, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = unit / d.hkv, h = unit % d.hkv;
    const int B = a.per_batch_budget ? a.budget_of[b] : d.B;
    const int pairs = a.has_graph ? d.K_src * d.m : 0, words = row_words(N);
    Smem s;
    s.hist = reinterpret_cast<uint32_t *>(rf_smem);
    s.tot = s.hist + kBins;
    s.val = reinterpret_cast<float *>(rf_smem + kScratch);
    s.pos = reinterpret_cast<int *>(s.val + a.cap);
    s.nb_j = s.pos + a.cap;
    s.nb_f = reinterpret_cast<float *>(s.nb_j + pairs);
    s.kept = s.nb_j;
    s.wcnt = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(s.nb_j) + a.list_bytes);
    s.misc = s.wcnt + 2 * kWarps;
    s.bits = s.misc + 16;
    s.ties = s.bits + words;
    s.before = s.ties + words;
    float *row = a.s + (long long)unit * N;
    PhaseClock pc(tid == 0);
    pc.mark();
    if (C > 1) cl.barrier_arrive();            // (every CTA runs before another one writes to its shared memory)

    // Rows t0 ... of the output from rows src_of(t): the threads of `ctas` CTAs from rank `first` share the 16-byte pieces, four in
    // flight per thread, or eight where a thread has more than that to copy (long loops hide their fetches).
    const int rows_out = d.B + d.W, vl = a.vpr_log2;
    auto copy_pieces = [&](auto in_flight, int t0, int n_rows, int first, int ctas, auto src_of) {
        constexpr int kU = decltype(in_flight)::value;
        const unsigned char *k0 = a.K + (b * d.ks[0] + h * d.ks[1]) * a.elem_bytes;
        const unsigned char *v0 = a.V + (b * d.vs[0] + h * d.vs[1]) * a.elem_bytes;
        const long long k_stride = d.ks[2] * a.elem_bytes, v_stride = d.vs[2] * a.elem_bytes;
        const long long out0 = (long long)unit * rows_out;
        const int n_pieces = n_rows << (vl + 1), stride = ctas * kThreads;
        for (int p0 = (rank - first) * kThreads + tid; p0 < n_pieces; p0 += kU * stride) {
            uint4 v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int p = p0 + u * stride;
                const bool is_v = (p >> vl) & 1;
                if (p < n_pieces && (is_v ? a.V != nullptr : a.K != nullptr))
                    v[u] = *reinterpret_cast<const uint4 *>((is_v ? v0 : k0) + src_of(t0 + (p >> (vl + 1))) * (is_v ? v_stride : k_stride) +
                                                            (p & ((1 << vl) - 1)) * 16);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int p = p0 + u * stride;
                const bool is_v = (p >> vl) & 1;
                if (p < n_pieces && (is_v ? a.V != nullptr : a.K != nullptr))
                    *reinterpret_cast<uint4 *>((is_v ? a.V_out : a.K_out) +
                                               (((out0 + t0 + (p >> (vl + 1))) << vl) + (p & ((1 << vl) - 1))) * 16) = v[u];
            }
        }
    };
    auto copy_rows = [&](int t0, int n_rows, int first, int ctas, auto src_of) {
        if ((n_rows << (vl + 1)) > 8 * ctas * kThreads) copy_pieces(std::integral_constant<int, 8>{}, t0, n_rows, first, ctas, src_of);
        else copy_pieces(std::integral_constant<int, 4>{}, t0, n_rows, first, ctas, src_of);
    };
    const bool gathers = a.do_select && (a.K || a.V);
    if (a.wait_prior && !a.early_row) pdl_wait();
    pc.mark();

    // ---- which elements can be kept ----
    const bool lowers = a.has_graph && d.signal != GRAPHKV_SIGNAL_ENHANCE;
    uint32_t tie_room = 0;                     // with `some_ties`: elements of the tie bits to keep
    bool some_ties = false;
    uint32_t lo_key = 0, hi_digits = 0;        // the final threshold lies in these digits from lo_key on (0: unknown)
    if (C > 1) cl.barrier_wait();
    if (a.do_select && !a.dense) {
        const int base = rank * a.chunk, n_local = max(0, min(a.chunk, N - base));
        const float *mine = row + base;
        const uint32_t need = (uint32_t)min(N, B + (lowers ? pairs : 0));
        uint32_t prefix = 0, mask = 0, remaining = need;
        static_assert(kBins == 4 * kThreads, "four counts per thread");
        auto load8 = [&](int i0, float (&x)[8]) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int i = i0 + q * kThreads + lane;
                x[q] = i < n_local ? mine[i] : 0.f;
            }
        };
        float x[8];
        load8(warp * 32, x);
        for (int pass = 0; pass < 3; ++pass) {
            const int shift = digit_shift(pass), nb = digit_count(pass);
            const uint32_t *total = s.hist;
            if (pass == 0 && a.row_hist) {
                reinterpret_cast<uint4 *>(s.hist)[tid] =
                    __ldcg(reinterpret_cast<const uint4 *>(a.row_hist + (long long)unit * kBins) + tid);
                __syncthreads();
            } else {
                for (int i = tid; i < nb; i += kThreads) s.hist[i] = 0u;
                __syncthreads();
                for (int i0 = warp * 32; i0 < n_local; i0 += 8 * kThreads) {
                    if (i0 >= 8 * kThreads || pass > 0) load8(i0, x);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int i = i0 + q * kThreads + lane;
                        const uint32_t key = float_to_key(x[q]);
                        if (i - lane < n_local)
                            count_bin(s.hist, (key >> shift) & (uint32_t)(nb - 1), i < n_local && (key & mask) == prefix);
                    }
                }
                if (C > 1) {
                    cl.sync();
                    // a CTA adds up a slice of the digits and gives everybody the sums
                    const int slice = nb / C;
                    for (int i = tid; i < slice; i += kThreads) {
                        const int bin = rank * slice + i;
                        uint32_t part[kMaxCluster], sum = 0;
#pragma unroll
                        for (int p = 0; p < kMaxCluster; ++p) part[p] = p < C ? cl.map_shared_rank(s.hist, p)[bin] : 0u;
#pragma unroll
                        for (int p = 0; p < kMaxCluster; ++p) sum += part[p];
#pragma unroll
                        for (int p = 0; p < kMaxCluster; ++p)
                            if (p < C) cl.map_shared_rank(s.tot, p)[bin] = sum;
                    }
                    cl.sync();
                    total = s.tot;
                } else {
                    __syncthreads();
                }
            }
            find_digit(total, nb, remaining, s.wcnt, s.misc, pass == 0 ? (uint32_t)B : 0u);
            const uint32_t above = s.misc[1], in = s.misc[2];
            prefix |= s.misc[0] << shift;
            mask |= (uint32_t)(nb - 1) << shift;
            const bool fits = need - remaining + above + in <= (uint32_t)a.sel_cap;
            remaining -= above;
            if (fits) {
                // (the B-th largest, as the scores are now, bounds the final one from above unless scores rise)
                if (pass == 0 && prefix > 0u) lo_key = prefix, hi_digits = s.misc[6] - s.misc[0] + 1u;
                break;
            }
            some_ties = pass == 2;
            __syncthreads();
        }
        tie_room = remaining;
        // one bit per element, and one per tie of the last value where not all of them are wanted
        uint32_t *bits0 = C > 1 ? cl.map_shared_rank(s.bits, 0) : s.bits;
        uint32_t *ties0 = C > 1 ? cl.map_shared_rank(s.ties, 0) : s.ties;
        for (int i0 = warp * 32; i0 < n_local; i0 += 8 * kThreads) {
            if (i0 >= 8 * kThreads || n_local > 8 * kThreads) load8(i0, x);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int i = i0 + q * kThreads + lane;
                const uint32_t key = float_to_key(x[q]) & mask;
                const unsigned ge = __ballot_sync(0xffffffffu, i < n_local && key >= prefix);
                if (some_ties) {
                    const unsigned eq = __ballot_sync(0xffffffffu, i < n_local && key == prefix);
                    if (lane == 0 && i < n_local) {
                        bits0[(base + i) >> 5] = ge & ~eq;
                        ties0[(base + i) >> 5] = eq;
                    }
                } else if (lane == 0 && i < n_local) {
                    bits0[(base + i) >> 5] = ge;
                }
            }
        }
        __syncthreads();                       // (the histogram's words become the merges' survivors)
    } else if (!a.dense && rank == 0) {
        for (int i = tid; i < words; i += kThreads) s.bits[i] = 0u;
    }
    pc.mark();

    // ---- the candidates, by position (first CTA) ----
    int n = N;
    const bool late = !a.dense && (a.has_graph && (a.keep_scores || !a.do_select || !lowers));
    auto list_candidates = [&]() {
        if (!a.dense) {
            const int per = ceil_div(words, kThreads), w0 = min(tid * per, words), w1 = min(w0 + per, words);
            uint32_t total;
            if (some_ties) {
                // the first tie_room of the ties join
                uint32_t sum = 0;
                for (int w = w0; w < w1; ++w) sum += __popc(s.ties[w]);
                uint32_t run = block_exclusive(sum, s.wcnt, &total);
                for (int w = w0; w < w1; ++w) {
                    uint32_t t = s.ties[w];
                    for (; t != 0u && run < tie_room; ++run) {
                        s.bits[w] |= t & (0u - t);
                        t &= t - 1u;
                    }
                    run += __popc(t);
                }
                __syncthreads();
            }
            if (late) {
                // every listed position: its score is written back, or may rise to the top
                for (int i = tid; i < pairs; i += kThreads) {
                    const int j = s.nb_j[i];
                    if (j >= 0) atomicOr(&s.bits[j >> 5], 1u << (j & 31));
                }
                __syncthreads();
            }
            uint32_t sum = 0;
            for (int w = w0; w < w1; ++w) sum += __popc(s.bits[w]);
            uint32_t run = block_exclusive(sum, s.wcnt, &total);
            n = (int)total;
            for (int w = w0; w < w1; ++w) {
                s.before[w] = run;
                for (uint32_t t = s.bits[w]; t != 0u; t &= t - 1u) s.pos[run++] = w * 32 + __ffs(t) - 1;
            }
            __syncthreads();
        }
#pragma unroll 4
        for (int i = tid; i < n; i += kThreads) s.val[i] = __ldcg(row + (a.dense ? i : s.pos[i]));
    };
    if (!late) {
        if (C > 1 && !a.dense) cl.sync();
        if (rank == 0) list_candidates();
        pc.mark();
    }

    // ---- Eq. 3: the neighbour lists, into the first CTA's shared memory ----
    if (a.wait_prior) pdl_wait();
    pdl_launch_dependents();
    pc.mark();
    if (a.has_graph) {
        int *ni = a.nbr_idx + (long long)unit * pairs;
        float *ne = a.nbr_e + (long long)unit * pairs;
        if (a.merge) {
            const int threads = a.group_warps * 32, group = tid / threads, groups = kThreads / threads;
            unsigned long long *surv = reinterpret_cast<unsigned long long *>(rf_smem) + group * kSurvCap;
            uint32_t *count = s.wcnt + group;
            int *nb_j = C > 1 ? cl.map_shared_rank(s.nb_j, 0) : s.nb_j;
            float *nb_f = C > 1 ? cl.map_shared_rank(s.nb_f, 0) : s.nb_f;
            // (the first CTA of a cluster has its candidates to list)
            const int M = C > 1 ? C - 1 : 1, r = C > 1 ? rank - 1 : 0;
            for (int src = group * M + r; r >= 0 && src < d.K_src; src += groups * M) {
                const long long list = (long long)unit * d.K_src + src;
                merge_source(d, a.cand + list * a.cand_chunks * kCandCap, a.cand_hist + list * kCandBins,
                             a.cand_chunks * kCandCap, surv, count, 1 + group, threads, tid - group * threads,
                             ni + src * d.m, ne + src * d.m, nb_j + src * d.m, nb_f + src * d.m);
            }
        } else if (rank == 0) {
            for (int i = tid; i < pairs; i += kThreads) {
                s.nb_j[i] = __ldcg(ni + i);
                s.nb_f[i] = signal_factor(__ldcg(ne + i), d.lambda, d.T, d.signal);
            }
        }
    }
    pc.mark();
    if (C > 1) cl.sync(); else __syncthreads();
    pc.mark();
    if (rank == 0) {
        if (late) list_candidates();
        // ---- Eq. 5, the T rounds folded into each edge's factor ----
        if (a.has_graph) {
            for (int p = tid; p < pairs; p += kThreads) {
                const int j = s.nb_j[p];
                int slot = j;
                if (!a.dense && j >= 0) {
                    const uint32_t w = s.bits[j >> 5], bit = 1u << (j & 31);
                    slot = (w & bit) ? (int)(s.before[j >> 5] + __popc(w & (bit - 1u))) : -1;
                }
                s.nb_j[p] = slot;
            }
            __syncthreads();
            pc.mark();
            // A candidate belongs to one warp, which walks the sources in order (the neighbours of a
            // source are distinct), so that overlapping neighbourhoods multiply in a fixed order.
            const bool evict = d.signal == GRAPHKV_SIGNAL_EVICT;
            auto apply = [&](int slot, float f) {
                if (slot >= 0 && (slot & (kWarps - 1)) == warp) s.val[slot] = evict ? -INFINITY : s.val[slot] * f;
                __syncwarp();
            };
            if (d.m <= 32) {
                for (int q0 = 0; q0 < d.K_src; q0 += 4) {
                    int slot[4];
                    float f[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const bool in = lane < d.m && q0 + k < d.K_src;
                        slot[k] = in ? s.nb_j[(q0 + k) * d.m + lane] : -1;
                        f[k] = in ? s.nb_f[(q0 + k) * d.m + lane] : 1.f;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) apply(slot[k], f[k]);
                }
            } else {
                for (int q = 0; q < d.K_src; ++q)
                    for (int u = lane; u - lane < d.m; u += 32)
                        apply(u < d.m ? s.nb_j[q * d.m + u] : -1, u < d.m ? s.nb_f[q * d.m + u] : 1.f);
            }
            __syncthreads();
            if (a.keep_scores)
                for (int p = tid; p < pairs; p += kThreads) {
                    const int slot = s.nb_j[p];
                    if (slot >= 0) row[a.dense ? slot : s.pos[slot]] = s.val[slot];
                }
        }
        __syncthreads();
        pc.mark();
        if (a.do_select) {
            // ---- the B largest candidates, in ascending position ----
            uint32_t lo = lo_key, hi = 0xffffffffu;
            if (hi_digits > 0 && (lowers || !a.has_graph)) {
                if (hi_digits <= (0xffffffffu - lo_key) >> 21) hi = lo_key + (hi_digits << 21) - 1u;
            } else {
                bs::block_range(s.val, n, s.wcnt, lo, hi);
            }
            const bs::Kept th = bs::block_kth(s.val, n, (uint32_t)B, lo, hi, s.hist, s.wcnt, s.misc);
            pc.mark();
            int *idx = a.idx_out + (long long)unit * d.B;
            bs::emit_kept(s.val, n, th, s.wcnt, [&](int t, int i) {
                const int j = a.dense ? i : s.pos[i];
                idx[t] = j;
                s.kept[t] = j;
            });
        }
        pc.mark();
    }
    // ---- gather ----
    if (gathers) {
        // the window rows, while the first CTA of the cluster selects
        if (C == 1 || rank > 0) copy_rows(B, d.W, C > 1 ? 1 : 0, C > 1 ? C - 1 : 1, [&](int t) { return (long long)(N + (t - B)); });
        if (C > 1) cl.sync(); else __syncthreads();
        pc.mark();
        if (C > 1) {
            if (rank > 0)
                for (int t = tid; t < B; t += kThreads) s.kept[t] = cl.map_shared_rank(s.kept, 0)[t];
            cl.barrier_arrive();               // the first CTA's positions have been read
            __syncthreads();
        }
        copy_rows(0, B, 0, C, [&](int t) { return (long long)s.kept[t]; });
        if (C > 1) cl.barrier_wait();
    }
    pc.mark();
    pc.flush(rank == 0 ? 4 : 6);
}

}  // namespace rf
}  // namespace graphkv
