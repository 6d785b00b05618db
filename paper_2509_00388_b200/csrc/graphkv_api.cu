// C ABI of the GraphKV library: argument validation, workspace layout and kernel launches.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "cluster_path.cuh"
#include "cluster_select.cuh"
#include "common.cuh"
#include "decode_attn.cuh"
#include "gather.cuh"
#include "row_finish.cuh"
#include "propagate_simt.cuh"
#include "score_simt.cuh"
#include "score_tc.cuh"
#include "select.cuh"
#include "sim_stream.cuh"
#include "sim_tc.cuh"

using namespace graphkv;

namespace {

constexpr size_t kAlign = 256;
constexpr size_t kMaxSmem = 227 * 1024;      // dynamic shared memory a CTA may ask for
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// Workspace carve-up; every region starts 256-byte aligned.
struct Layout {
    size_t status;      // int status word (256 bytes reserved)
    size_t arrivals;    // counters of score CTAs per unit [2 * units] (directly after the status word)
    size_t a_hist;      // histogram of the attention mass [units][2048] (directly after the counters)
    size_t row_c;       // softmax row constants [units][2][GW]
    size_t row_hist;    // histogram of the scores [units][2048], cleared by the sweeps
    size_t part;        // softmax row statistics per key chunk
    size_t a;           // attention mass before pooling [units][N]
    size_t s;           // scores when the caller gives no array [units][N]
    size_t src;         // source nodes [units][K_src]
    size_t sims;        // edges of the sources [units][K_src][N]
    size_t nbr_idx;     // neighbourhoods [units][K_src][m]
    size_t nbr_e;
    size_t cand;        // per-chunk neighbour candidates [units][K_src][sim_chunks][kCandCap]
    size_t cand_hist;   // [units][K_src][kCandBins]
    size_t tau;         // bounds of the sources' m-th edges [units][K_src]
    size_t spill;       // edges that full lists did not take, per CTA of the streaming sweep
    size_t total;
    int max_parts;      // partial statistics per row the region can hold
};

graphkv_status resolve(const graphkv_params *p, Dims *d)
{
    if (!p) return GRAPHKV_ERR_INVALID_ARG;
    if (p->batch < 1 || p->n_q_heads < 1 || p->n_kv_heads < 1 || p->window < 1 ||
        p->seq_len <= p->window || p->n_q_heads % p->n_kv_heads != 0)
        return GRAPHKV_ERR_INVALID_ARG;
    const int N = p->seq_len - p->window;
    if (p->budget < 1 || p->budget > N) return GRAPHKV_ERR_INVALID_ARG;
    if (p->pool_kernel < 1 || p->pool_kernel % 2 == 0) return GRAPHKV_ERR_INVALID_ARG;
    if (p->topk_nodes < 0 || p->topk_nodes > N) return GRAPHKV_ERR_INVALID_ARG;
    if (p->neighbors < 0 || p->neighbors > N - 1) return GRAPHKV_ERR_INVALID_ARG;
    if (p->rounds < 0) return GRAPHKV_ERR_INVALID_ARG;
    if (!(p->decay >= 0.0f && p->decay <= 1.0f)) return GRAPHKV_ERR_INVALID_ARG;
    if (p->dtype != GRAPHKV_BF16 && p->dtype != GRAPHKV_F32) return GRAPHKV_ERR_INVALID_ARG;
    if (p->pool_mode != GRAPHKV_POOL_MAX && p->pool_mode != GRAPHKV_POOL_AVG) return GRAPHKV_ERR_INVALID_ARG;
    if (p->signal < GRAPHKV_SIGNAL_DECAY || p->signal > GRAPHKV_SIGNAL_EVICT) return GRAPHKV_ERR_INVALID_ARG;
    if (p->reselect != 0 && p->reselect != 1) return GRAPHKV_ERR_INVALID_ARG;
    if (p->head_dim != kHeadDim && p->head_dim != 64) return GRAPHKV_ERR_UNSUPPORTED;
    const int G = p->n_q_heads / p->n_kv_heads;
    if ((long long)G * p->window > kMaxRows) return GRAPHKV_ERR_UNSUPPORTED;
    if ((long long)p->batch * p->n_kv_heads > 65535) return GRAPHKV_ERR_UNSUPPORTED;
    const int vec = p->dtype == GRAPHKV_BF16 ? 8 : 4;      // elements per 16 bytes
    for (int i = 0; i < 3; ++i) {
        if (p->q_stride[i] < 0 || p->k_stride[i] < 0 || p->v_stride[i] < 0)
            return GRAPHKV_ERR_INVALID_ARG;
        if (p->q_stride[i] % vec || p->k_stride[i] % vec || p->v_stride[i] % vec)
            return GRAPHKV_ERR_INVALID_ARG;
    }
    if (p->q_stride[2] < p->head_dim || p->k_stride[2] < p->head_dim || p->v_stride[2] < p->head_dim)
        return GRAPHKV_ERR_INVALID_ARG;
    d->batch = p->batch; d->hq = p->n_q_heads; d->hkv = p->n_kv_heads; d->G = G; d->D = p->head_dim;
    d->W = p->window; d->L = p->seq_len; d->N = N; d->GW = G * p->window;
    d->B = p->budget; d->kp = p->pool_kernel; d->K_src = p->topk_nodes;
    d->m = graphkv_resolve_neighbors(N, p->neighbors);
    d->T = p->rounds; d->lambda = p->decay; d->units = p->batch * p->n_kv_heads;
    d->bf16 = p->dtype == GRAPHKV_BF16 ? 1 : 0;
    d->pool_avg = p->pool_mode == GRAPHKV_POOL_AVG ? 1 : 0;
    d->signal = p->signal;
    d->reselect = p->reselect;
    for (int i = 0; i < 3; ++i) {
        d->qs[i] = p->q_stride[i]; d->ks[i] = p->k_stride[i]; d->vs[i] = p->v_stride[i];
    }
    return GRAPHKV_OK;
}

int env_int(const char *name, int dflt)
{
    const char *v = getenv(name);
    return v ? atoi(v) : dflt;
}

// Limit of the device-side waits in clocks: about two seconds, or GRAPHKV_WAIT_CYCLES (tests make
// a wait run out with a short one).
long long wait_cycles()
{
    const char *v = getenv("GRAPHKV_WAIT_CYCLES");
    const long long n = v ? atoll(v) : 0;
    return n > 0 ? n : tc::kWaitCycles;
}

// SMs of the current device (queried once per device).
int sm_count()
{
    static std::mutex mu;
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    std::lock_guard<std::mutex> lk(mu);
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 148;
        cached[dev] = n;
    }
    return cached[dev];
}

// Units per launch of a sweep.  By default all units go into one launch: measured on B200, the
// fixed cost of extra launches outweighs serving the later sweeps of a small group from L2
// (GRAPHKV_L2_GROUP_MB bounds the keys of a group for experiments).
int units_per_group(const Dims &d)
{
    const double mb = (double)d.L * d.D * 2 / 1.0e6;
    int n = (int)(env_int("GRAPHKV_L2_GROUP_MB", 1 << 20) / mb);
    if (n < 1) n = 1;
    if (n > d.units) n = d.units;
    return n;
}

// Key chunks (CTAs) per unit for a sweep of `tiles` key tiles per unit over `units` units, one CTA
// per SM: the count that minimises waves x (tiles per CTA + a per-CTA overhead of about three
// tile times), with at least min_chunks and at most max_chunks.
int sweep_chunks(int units, int tiles, int min_chunks, int max_chunks)
{
    const int n_sms = sm_count();
    int best = std::max(1, min_chunks);
    long long best_cost = -1;
    const int hi = std::max(best, std::min(tiles, max_chunks));
    for (int c = best; c <= hi; ++c) {
        const long long waves = ceil_div(units * c, n_sms);
        const long long cost = waves * (ceil_div(tiles, c) + 3);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

// ---- row-wise stages on clusters: which rows fit ----------------------------------------------------
struct ClusterPlan {
    bool ok;            // the row fits the cluster kernels
    int C, chunk, halo;
};

ClusterPlan cluster_plan(const Dims &d)
{
    ClusterPlan p{false, 1, 0, (d.kp - 1) / 2};
    if (env_int("GRAPHKV_NO_CLUSTER", 0)) return p;
    // as many CTAs per row as keep a chunk near 2048 scores (the finishing kernel that holds the whole row also
    // spreads its gather over them: 16384-score rows with 2048 kept rows 35 us on 8 CTAs per row against 42
    // on 4), but all clusters in one wave of the 148 SMs when the rows allow it (two waves of clusters of 8
    // measured 1.8x slower than one wave of clusters of 4 for 32 rows of 131072)
    while (p.C < cs::kMaxCluster && ceil_div(d.N, p.C) > 2048) p.C *= 2;
    while (p.C > 1 && d.units * p.C > sm_count() && ceil_div(d.N, p.C / 2) <= cs::kMaxChunk) p.C /= 2;
    // hundreds of sources: their neighbour lists are merged by groups of warps, kMergeWarps per CTA,
    // so more CTAs per row shorten that phase as long as all clusters stay in one wave
    while (d.K_src > 4 * cs::kMergeWarps * p.C && p.C < cs::kMaxCluster && d.units * p.C * 2 <= sm_count() &&
           ceil_div(d.N, p.C * 2) >= 1024)
        p.C *= 2;
    p.chunk = (ceil_div(d.N, p.C) + 31) & ~31;
    p.ok = p.chunk <= cs::kMaxChunk && p.halo <= cs::kMaxHalo;
    return p;
}

// Tensor-core similarity sweep: usable for bf16 keys and up to 32 neighbours; 64 sources per
// sweep of the keys, so a head with more sources (the paper's 0.3 x budget) is swept several times.
constexpr int kSimMaxSources = 4096;
struct SimPlan {
    bool ok;
    int NP;         // sources per sweep padded to 16, 32 or 64
    int chunks;     // CTAs (key chunks) per unit
    int n_tiles;    // 128-key tiles per unit
    int stages;
    bool stream;    // bounds from a sample, then one sweep for all sources (NP: up to 256)
    int sample, sample_ctas;    // sample tiles, and the CTAs that share them
};

SimPlan sim_plan(const Dims &d, bool bf16)
{
    SimPlan p{false, 16, 1, ceil_div(d.N, tc::kTileKeys), 5, false, 0, 0};
    if (!bf16 || d.K_src < 1 || d.K_src > kSimMaxSources || d.m < 1 ||
        d.m > tc::kSimMaxNeighbors)
        return p;
    if (env_int("GRAPHKV_FORCE_SIMT", 0)) return p;
    if (!cluster_plan(d).ok) return p;          // its candidate lists are merged by the cluster kernel
    // Sources per sweep when there are more than 32.  The tensor memory (512 columns) holds 8 key tiles of 64
    // sources or 16 of 32.  Where 8 tiles per CTA are enough to take the rows in one wave, 64 halve the
    // sweeps and their fixed cost (64 sources: 25 us against 31 at 8K keys x 8 heads, 33 against 39 at
    // 16K).  Beyond that the CTAs of 64 queue for the SMs and their maxima, of half as many keys, bound
    // the neighbours less tightly (50 us against 56 at 32K x 8, 154 sources 111 against 158, 64 sources
    // at 128K x 32: 617 against 721).
    const int group = units_per_group(d);
    p.NP = d.K_src <= 16 ? 16 : d.K_src <= 32 || (long long)group * ceil_div(p.n_tiles, 8) > sm_count() ? 32 : 64;
    p.stages = d.D == 64 ? 8 : 5;
    const int cap = 512 / p.NP;
    p.chunks = sweep_chunks(group * ceil_div(d.K_src, p.NP), p.n_tiles, ceil_div(p.n_tiles, cap), 1 << 20);
    p.ok = true;
    // A head's sources in one streaming sweep, with bounds from a sample (sim_stream.cuh), where that form would take
    // more than one wave of CTAs and the estimate below is for it.
    const int waves = ceil_div(d.units * ceil_div(d.K_src, p.NP) * p.chunks, sm_count());
    if (group >= d.units && d.K_src > 16 && p.n_tiles >= 16 && waves > 1) {
        SimPlan q = p;
        q.stream = true;
        const int sweeps = ceil_div(d.K_src, tc::kStreamMaxSources), blocks = d.units * ceil_div(d.K_src, 32);
        q.NP = ceil_div(ceil_div(d.K_src, sweeps), 32) * 32;
        // The larger the sample, the fewer edges reach the bounds, about 1.4 m n_tiles / sample of a row's, which all have to be
        // listed.  A cluster of up to four CTAs takes it: a quarter of the row, 16 tiles a CTA; where a CTA has it to itself, three
        // eighths, up to 64 tiles.
        q.sample_ctas = std::max(1, std::min(4, sm_count() / blocks));
        q.sample = std::max(1, q.sample_ctas > 1 ? std::min(p.n_tiles / 4, 16 * q.sample_ctas) : std::min(p.n_tiles * 3 / 8, 64));
        q.sample_ctas = std::min(q.sample_ctas, q.sample);
        // chunks of up to 32 tiles, with 40 such edges or fewer on the average, of the 64 that a list holds
        const double edges = 1.4 * d.m * p.n_tiles / q.sample;
        q.chunks = sweep_chunks(d.units * sweeps, p.n_tiles, std::max(ceil_div(p.n_tiles, tc::kStreamMaxTiles), (int)(edges / 40) + 1), 1 << 20);
        for (q.stages = 6; q.stages > 3; --q.stages)
            if ((d.D == 64 ? tc::stream_layout<64>(q.NP, q.stages) : tc::stream_layout<128>(q.NP, q.stages)).bytes <= kMaxSmem) break;
        // Times in us: waves of CTAs, each some us and a time per tile; an edge above its bound 15 ns where many share a list.
        const double resident = waves * (4 + (p.NP == 64 ? 2.4 : 1.2) * ceil_div(p.n_tiles, p.chunks));
        const double stream = ceil_div(blocks * q.sample_ctas, sm_count()) * (7 + 0.5 * ceil_div(q.sample, q.sample_ctas)) +
                              ceil_div(d.units * sweeps * q.chunks, sm_count()) * (6 + (0.4 + 0.012 * q.NP) * ceil_div(p.n_tiles, q.chunks)) +
                              0.015 * edges * d.units * d.K_src / sm_count();
        // Calls of up to two waves: the sample runs under the end of the pooling kernel, and both forms take the same time within some
        // percent (16 x 10000 with 60 sources, at 1.49: 108 and 108 us a call, with topics of 64 tokens 108 and 122; 8 x 8192 with
        // 160, at 1.32: 106 and 103, 117 and 125; 8 x 32K with 64, at 1.09: 123 and 123, 131 and 135).  In larger ones the estimate
        // tells (128 x 16K with 32, at 1.30: 440 and 469, 443 and 497; 64 x 8160 with 100, at 1.17: 275 and 258, 288 and 322; with 38,
        // at 1.05: 194 and 190, 198 and 215; 128 x 16K with 64, at 1.03: 608 and 563, 624 and 621; 32 x 16K with 154, at 0.97: 321 and
        // 279, 334 and 332; 32 x 128K with 32, at 0.88: 822 and 802, 822 and 765).
        if (stream < (waves <= 2 ? 1.5 : 1.05) * resident) return q;
    }
    return p;
}

Layout layout_of(const Dims &d)
{
    Layout l;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes); return o; };
    l.max_parts = std::max(148, ceil_div(d.L, 1024));
    l.status = take(kAlign);
    l.arrivals = take((size_t)d.units * 2 * sizeof(int));
    l.a_hist = take((size_t)d.units * tc::kMassBins * sizeof(uint32_t));
    l.row_hist = take((size_t)d.units * cs::kBins * sizeof(uint32_t));
    l.row_c = take((size_t)d.units * d.GW * 2 * sizeof(float));
    l.part = take((size_t)d.units * l.max_parts * d.GW * 2 * sizeof(float));
    l.a = take((size_t)d.units * d.N * sizeof(float));
    l.s = take((size_t)d.units * d.N * sizeof(float));
    l.src = take((size_t)d.units * (d.K_src > 0 ? d.K_src : 1) * sizeof(int));
    const size_t pairs = (size_t)d.units * (d.K_src > 0 ? d.K_src : 1) * (d.m > 0 ? d.m : 1);
    // the dense edge rows exist only for the generic similarity path
    const SimPlan sp0 = sim_plan(d, d.bf16 != 0);
    l.sims = take(sp0.ok ? kAlign : (size_t)d.units * (d.K_src > 0 ? d.K_src : 1) * d.N * sizeof(float));
    l.nbr_idx = take(pairs * sizeof(int));
    l.nbr_e = take(pairs * sizeof(float));
    const SimPlan sp = sim_plan(d, d.bf16 != 0);
    const size_t slots = sp.ok ? (size_t)d.units * d.K_src * sp.chunks : 1;
    l.cand = take(slots * kCandCap * sizeof(Cand));
    l.cand_hist = take((size_t)d.units * (d.K_src > 0 ? d.K_src : 1) * kCandBins * sizeof(uint32_t));
    l.tau = take((size_t)d.units * (d.K_src > 0 ? d.K_src : 1) * sizeof(float));
    l.spill = take(sp.stream ? (size_t)ceil_div(d.K_src, sp.NP) * d.units * sp.chunks * tc::kStreamSpill * sizeof(uint2) : 1);
    l.total = off;
    return l;
}

graphkv_status check_ws(const Layout &l, const void *ws, size_t ws_bytes)
{
    if (!ws || (reinterpret_cast<uintptr_t>(ws) % kAlign) != 0 || ws_bytes < l.total)
        return GRAPHKV_ERR_WORKSPACE;
    return GRAPHKV_OK;
}

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline graphkv_status launch_status()
{
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        if (getenv("GRAPHKV_LOG")) fprintf(stderr, "graphkv: launch failed: %s\n", cudaGetErrorString(e));
        return GRAPHKV_ERR_CUDA;
    }
    return GRAPHKV_OK;
}

// ---- launch accounting and optional per-kernel timing -----------------------------------------
std::atomic<long long> g_launches{0};
std::atomic<int> g_trace_on{0};
std::mutex g_trace_mu;
struct TraceEntry { const char *name; cudaEvent_t start, stop; };
std::vector<TraceEntry> g_trace;

// Counts one kernel launch; with tracing on, brackets it with CUDA events on its stream.
struct LaunchScope {
    cudaStream_t st;
    bool traced;
    TraceEntry e;
    LaunchScope(const char *name, cudaStream_t s) : st(s), traced(false)
    {
        g_launches.fetch_add(1, std::memory_order_relaxed);
        if (!g_trace_on.load(std::memory_order_relaxed)) return;
        e.name = name;
        if (cudaEventCreate(&e.start) != cudaSuccess) return;
        if (cudaEventCreate(&e.stop) != cudaSuccess) { cudaEventDestroy(e.start); return; }
        cudaEventRecord(e.start, st);
        traced = true;
    }
    ~LaunchScope()
    {
        if (!traced) return;
        cudaEventRecord(e.stop, st);
        std::lock_guard<std::mutex> lk(g_trace_mu);
        g_trace.push_back(e);
    }
};
#define GKV_LAUNCH(name, st, ...)        \
    do {                                 \
        LaunchScope _scope(name, st);    \
        __VA_ARGS__;                     \
    } while (0)

template <typename T> inline T *at(void *ws, size_t off)
{
    return reinterpret_cast<T *>(static_cast<unsigned char *>(ws) + off);
}

// ---- launches with attributes -------------------------------------------------------------------
// Every kernel is launched with programmatic stream serialization: its prologue (barriers, TMEM and,
// after the first launch of a call, operand staging and the first key tiles) overlaps the tail of the
// kernel before, and it executes griddepcontrol.wait before touching anything an earlier kernel of
// the call wrote.  The first launch of a call waits before it touches its inputs as well: whatever
// the stream held before the call may have written them.
thread_local int t_launches_in_call = 0;

inline bool next_launch_is_dependent(int *first = nullptr)
{
    static const bool enabled = [] { const char *v = getenv("GRAPHKV_PDL"); return v ? atoi(v) != 0 : true; }();
    const bool dep = enabled && !g_trace_on.load(std::memory_order_relaxed);
    if (first) *first = t_launches_in_call == 0 ? 1 : 0;
    ++t_launches_in_call;
    return dep;
}

// Set before a launch_ex whose kernel makes its CTAs wait for one another: the launch then asks
// for all CTAs of the grid to be resident together (a cooperative launch), so that no other work
// on the device can keep part of the grid waiting for SMs that the rest of it holds.
thread_local bool t_cooperative = false;

template <typename... KArgs, typename... Args>
graphkv_status launch_ex(const char *name, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                         cudaStream_t st, bool dependent, int cluster_x, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[3];
    int n = 0;
    if (t_cooperative) {
        t_cooperative = false;
        attr[n].id = cudaLaunchAttributeCooperative;
        attr[n].val.cooperative = 1;
        ++n;
    }
    if (cluster_x > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster_x;
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (dependent) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attr;
    cfg.numAttrs = n;
    cudaError_t e;
    GKV_LAUNCH(name, st, (e = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...)));
    if (e != cudaSuccess) {
        if (getenv("GRAPHKV_LOG")) fprintf(stderr, "graphkv: %s: %s\n", name, cudaGetErrorString(e));
        return GRAPHKV_ERR_CUDA;
    }
    return GRAPHKV_OK;
}

// Runs `setup` once per device (function attributes are per device); returns its result.
template <typename F> bool once_per_device(std::mutex &mu, signed char (&state)[64], F setup)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lk(mu);
    if (state[dev] == 0) state[dev] = setup() ? 1 : -1;
    return state[dev] > 0;
}

template <typename Kern> bool set_smem(Kern k, size_t bytes)
{
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

// A value for the arrival words of the kernel of both score sweeps that no earlier call of this
// process has used (never zero; the sequence starts at a clock-derived value, so a word left by
// another process matches it only by a 1 in 2^32 chance).
uint32_t next_call_tag()
{
    static std::atomic<uint32_t> tag{
        static_cast<uint32_t>(std::chrono::steady_clock::now().time_since_epoch().count() * 2654435761u) | 1u};
    uint32_t t = tag.fetch_add(1u) + 1u;
    if (t == 0u) t = tag.fetch_add(1u) + 1u;
    return t;
}

// Status word, arrival counters and the mass histogram start every scoring call at zero: a memset
// ahead of the sweeps, except where the kernel of both sweeps clears them itself.
inline graphkv_status reset_words(const Dims &d, const Layout &l, void *ws, cudaStream_t st)
{
    return cudaMemsetAsync(ws, 0, l.a_hist + (size_t)d.units * tc::kMassBins * sizeof(uint32_t), st) == cudaSuccess
               ? GRAPHKV_OK : GRAPHKV_ERR_CUDA;
}

// ---- step (I) ------------------------------------------------------------------------------
// Attention mass before pooling, a [units][N], SIMT path (any dtype).
template <typename T, int kD, int kRT>
graphkv_status launch_mass_simt(const Dims &d, const Layout &l, const T *Q, const T *K, float *a, void *ws,
                                cudaStream_t st)
{
    const size_t smem = simt_smem_bytes<kD>(kRT);
    static std::mutex mu;
    static signed char state[64] = {};
    if (!once_per_device(mu, state, [smem] {
            return set_smem(score_stats_simt<T, kD, kRT>, smem) && set_smem(score_emit_simt<T, kD, kRT>, smem);
        }))
        return GRAPHKV_ERR_CUDA;
    float *part = at<float>(ws, l.part);
    // one wave of two CTAs per SM (what the registers hold) over all units, whole tiles each
    const int row_tiles = ceil_div(d.GW, kRT), room = 2 * sm_count();
    auto ctas = [&](int keys, int per_tile) {
        const int tiles = ceil_div(keys, kSimtKeys);
        return std::max(1, std::min(tiles, room / (d.units * per_tile)));
    };
    const int chunks = std::min(ctas(d.L, row_tiles), l.max_parts);
    const graphkv_status rc = launch_ex("score_stats_simt", score_stats_simt<T, kD, kRT>, dim3(chunks, d.units, row_tiles),
                                        dim3(kSimtThreads), smem, st, next_launch_is_dependent(), 1, d, Q, K, part,
                                        chunks, at<int>(ws, l.status));
    if (rc != GRAPHKV_OK) return rc;
    return launch_ex("score_emit_simt", score_emit_simt<T, kD, kRT>, dim3(ctas(d.N, 1), d.units), dim3(kSimtThreads),
                     smem, st, next_launch_is_dependent(), 1, d, Q, K, static_cast<const float *>(part), chunks, a);
}

template <typename T>
graphkv_status run_mass_simt(const Dims &d, const Layout &l, const T *Q, const T *K, float *a,
                             void *ws, cudaStream_t st)
{
    if (d.GW <= 32)
        return d.D == 64 ? launch_mass_simt<T, 64, 32>(d, l, Q, K, a, ws, st) : launch_mass_simt<T, 128, 32>(d, l, Q, K, a, ws, st);
    return d.D == 64 ? launch_mass_simt<T, 64, 64>(d, l, Q, K, a, ws, st) : launch_mass_simt<T, 128, 64>(d, l, Q, K, a, ws, st);
}

// ---- clusters: what the device holds ---------------------------------------------------------------
template <int kD, int kTiles> bool cluster_path_ready()
{
    static std::mutex mu;
    static signed char state[64] = {};
    return once_per_device(mu, state, [] {
        return set_smem(cp::cluster_path_kernel<kD, kTiles>, kMaxSmem) &&
               cudaFuncSetAttribute(cp::cluster_path_kernel<kD, kTiles>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    });
}

// Clusters of C CTAs that are all resident, one CTA per SM, for C = 1 .. cp::kMaxCluster (nullptr: no device): the device
// is asked once (148, 74, 33, 15, 11, 7 clusters of 1, 2, 4, 8, 10, 16 on a B200).
const int *resident_clusters()
{
    static std::once_flag once[64];
    static int fits[64][cp::kMaxCluster + 1] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::call_once(once[dev], [dev] {
        if (!cluster_path_ready<128, 1>()) return;
        for (int q = 1; q <= cp::kMaxCluster; ++q) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(q);
            cfg.blockDim = dim3(cp::kThreads);
            cfg.dynamicSmemBytes = kMaxSmem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = q;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, cp::cluster_path_kernel<128, 1>, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            fits[dev][q] = n;
        }
    });
    return fits[dev];
}

// Largest power-of-two cluster size (up to 8) at which `units` clusters are all resident.
int resident_cluster_size(int units)
{
    const int *fits = resident_clusters();
    for (int C = 8; fits && C >= 1; C /= 2)
        if (fits[C] >= units) return C;
    return 0;
}

// How the cluster path cuts a row of n_tiles key tiles: the smallest cluster whose CTAs have the fewest tiles, all
// clusters resident (C = 0: none).
struct ShortRow {
    int C, tiles;
};

ShortRow short_row(const Dims &d)
{
    ShortRow s{0, 0};
    const int n_tiles = ceil_div(d.L, tc::kTileKeys), most = cp::max_tiles(d.D);
    if (n_tiles > cp::kMaxCluster * most || d.units > sm_count()) return s;
    const int *fits = resident_clusters();
    if (!d.bf16) {              // 64 keys per CTA, or 128 where the clusters would not all be resident; up to 128 query rows
        for (int tiles = 1; tiles <= 2 && s.C == 0; ++tiles) {
            const int C = ceil_div(d.L, 64 * tiles);
            if (fits && C <= cp::kMaxCluster && fits[C] >= d.units && d.GW <= 128) s = ShortRow{C, tiles};
        }
        return s;
    }
    for (int C = 1; fits && C <= std::min(cp::kMaxCluster, n_tiles); ++C) {
        if (fits[C] < d.units) continue;
        const int tiles = ceil_div(n_tiles, C);
        if (tiles <= most && (s.C == 0 || tiles < s.tiles)) s = ShortRow{C, tiles};
    }
    return s;
}

// The graph's parameters are ones the cluster path takes, and a call in stages would have its cosines from the tensor
// cores too (wide pooling sends that to the register-tiled products, which round differently).
inline bool short_row_graph(const Dims &d)
{
    return d.K_src <= cp::kMaxSources && d.m <= cp::kMaxNeighbours && !(d.reselect && d.T > 1) &&
           (!d.bf16 || cluster_plan(d).ok);
}

// ---- step (I), tensor-core path (bf16) -----------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// Tensor map over K [batch][hkv][rows][D] bf16 with the caller's strides; boxes of 128 rows x 64
// columns, 128-byte swizzle, zero fill past the last row.  slice_step > 0: boxes of kSlices times kSliceKeys
// rows, one such slice every slice_step rows (zero fill past the last whole one).
bool make_k_tensormap(CUtensorMap *tm, const void *K, const Dims &d, int rows, const long long *ks = nullptr, int slice_step = 0)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    if (!ks) ks = d.ks;
    const cuuint64_t row_b = (cuuint64_t)ks[2] * 2;
    cuuint64_t head_b = (cuuint64_t)ks[1] * 2, batch_b = (cuuint64_t)ks[0] * 2;
    if (d.hkv == 1 || head_b == 0) head_b = row_b * (cuuint64_t)rows;
    if (d.batch == 1 || batch_b == 0) batch_b = head_b * (cuuint64_t)d.hkv;
    cuuint64_t dims[5] = {(cuuint64_t)d.D}, strides[4] = {row_b};
    cuuint32_t box[5] = {64}, estr[5] = {1, 1, 1, 1, 1};
    int n = 1;
    auto dim = [&](cuuint64_t size, cuuint32_t taken, cuuint64_t stride) {
        dims[n] = size;
        box[n] = taken;
        strides[n - 1] = stride;
        ++n;
    };
    if (slice_step > 0) {
        dim(tc::kSliceKeys, tc::kSliceKeys, row_b);
        dim((rows - tc::kSliceKeys) / slice_step + 1, tc::kSlices, (cuuint64_t)slice_step * row_b);
    } else {
        dim(rows, tc::kTileKeys, row_b);
    }
    dim(d.hkv, 1, head_b);
    dim(d.batch, 1, batch_b);
    return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, n, const_cast<void *>(K), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// What the sweeps do besides the attention mass: words cleared for the kernels that follow.
struct EmitExtras {
    uint32_t *zero;
    int zero_words;
    int stat_chunks;        // key chunks of the row statistics; 0: as suits the sweep
};

// Attention mass before pooling, a [units][N], tensor-core path (bf16).
template <int kD>
graphkv_status run_mass_tc(const Dims &d, const Layout &l, const __nv_bfloat16 *Q,
                           const __nv_bfloat16 *K, float *a, void *ws, cudaStream_t st,
                           const EmitExtras &ex)
{
    CUtensorMap tmK;
    if (!make_k_tensormap(&tmK, K, d, d.L)) return GRAPHKV_ERR_CUDA;
    const int row_tiles = d.GW <= 128 ? 1 : 2;
    const int rows_pad = 128 * row_tiles;
    const int stages = row_tiles == 1 ? 5 : 4;
    const size_t smem = tc::score_smem_bytes<kD>(rows_pad, stages);
    constexpr int kStages2 = kD == 64 ? 5 : 2;       // two CTAs per SM: what fits half its shared memory
    static std::mutex mu;
    static signed char state[64] = {};
    if (!once_per_device(mu, state, [] {
        const size_t mx = std::max(tc::score_smem_bytes<kD>(256, 4), tc::score_smem_bytes<kD>(128, 5));
        const size_t two = tc::score_smem_bytes<kD>(128, kStages2, 2);
        return set_smem(tc::score_stats_tc<1, kD, 1>, mx) && set_smem(tc::score_stats_tc<2, kD, 1>, mx) &&
                  set_smem(tc::score_emit_tc<1, kD, 1>, mx) && set_smem(tc::score_emit_tc<2, kD, 1>, mx) &&
                  set_smem(tc::score_stats_tc<1, kD, 2>, two) && set_smem(tc::score_emit_tc<1, kD, 2>, two) &&
                  set_smem(tc::score_fused_tc<1, kD>, mx) && set_smem(tc::score_fused_tc<2, kD>, mx);
        }))
        return GRAPHKV_ERR_CUDA;
    const int tiles_stats = ceil_div(d.L, tc::kTileKeys), tiles_emit = ceil_div(d.N, tc::kTileKeys);
    const int group = units_per_group(d);
    graphkv_status rc = GRAPHKV_OK;
    // the kernel of both sweeps (one launch of all units, all CTAs resident) clears the head of the
    // workspace itself; every other form gets a memset first
    const bool one_kernel = group >= d.units &&
                            d.units * (ex.stat_chunks ? ex.stat_chunks : sweep_chunks(d.units, tiles_stats, 1, l.max_parts)) <= sm_count() &&
                            !env_int("GRAPHKV_TWO_SCORE_KERNELS", 0);
    if (!one_kernel && reset_words(d, l, ws, st) != GRAPHKV_OK) return GRAPHKV_ERR_CUDA;
    for (int u0 = 0; u0 < d.units && rc == GRAPHKV_OK; u0 += group) {
        const int nu = std::min(group, d.units - u0);
        const int chunks_s = ex.stat_chunks ? ex.stat_chunks : sweep_chunks(nu, tiles_stats, 1, l.max_parts);
        // The two separate kernels run two CTAs per SM: a launch of several waves then pays for its set-ups and
        // tails once (256 units of 16K keys: 259 -> 229 us and 255 -> 228 us for the two sweeps).  A chunk
        // leaves four partials per row, which a launch of few units and many chunks has no room for.
        const bool two = !one_kernel && row_tiles == 1 && 4 * chunks_s <= l.max_parts;
        const int chunks_e = sweep_chunks(two ? ceil_div(nu, 2) : nu, tiles_emit, 1, l.max_parts);
        tc::ScoreTcArgs sa{d, Q, at<float>(ws, l.part), at<float>(ws, l.row_c), at<int>(ws, l.arrivals), a,
                           at<uint32_t>(ws, l.a_hist), at<int>(ws, l.status), u0,
                           chunks_s, tiles_stats, chunks_s, stages, 0, 0,
                           nullptr, 0, wait_cycles(), 0, 0u, env_int("GRAPHKV_DEBUG_WITHHOLD_COMMIT", 0)};
        tc::ScoreTcArgs ea = sa;
        ea.chunks = chunks_e;
        ea.n_tiles = tiles_emit;
        ea.zero = ex.zero;
        ea.zero_words = ex.zero_words;
        // one kernel for both sweeps when all its CTAs are resident at once (one per SM): the CTAs
        // of a unit wait for one another between the passes, so the launch is a cooperative one
        // (the device starts the grid only when all of it fits beside whatever else is running);
        // a device that refuses it gets the two kernels
        if (one_kernel) {
            tc::ScoreTcArgs fa = ea;
            fa.chunks = chunks_s;
            fa.n_tiles = tiles_stats;
            fa.clear_head = 1;
            fa.call_tag = next_call_tag();
            fa.wait_prior = next_launch_is_dependent(&fa.first);
            t_cooperative = true;
            rc = launch_ex("score_fused_tc", row_tiles == 1 ? tc::score_fused_tc<1, kD> : tc::score_fused_tc<2, kD>,
                           dim3(chunks_s, nu), dim3(tc::kScoreThreads), smem, st, fa.wait_prior != 0, 1, tmK, fa);
            if (rc == GRAPHKV_OK) continue;
            cudaGetLastError();
            if (reset_words(d, l, ws, st) != GRAPHKV_OK) return GRAPHKV_ERR_CUDA;
            rc = GRAPHKV_OK;
        }
        sa.wait_prior = next_launch_is_dependent(&sa.first);
        if (two) sa.stages = ea.stages = kStages2;
        const dim3 block(two ? tc::score_threads<2>() : tc::kScoreThreads);
        const size_t bytes = two ? tc::score_smem_bytes<kD>(128, kStages2, 2) : smem;
        rc = launch_ex("score_stats_tc", two ? tc::score_stats_tc<1, kD, 2> : row_tiles == 1 ? tc::score_stats_tc<1, kD, 1>
                       : tc::score_stats_tc<2, kD, 1>,
                       dim3(two ? 2 * chunks_s : chunks_s, nu), block, bytes, st, sa.wait_prior != 0, 1, tmK, sa);
        if (rc != GRAPHKV_OK) break;
        ea.wait_prior = next_launch_is_dependent();
        rc = launch_ex("score_emit_tc", two ? tc::score_emit_tc<1, kD, 2> : row_tiles == 1 ? tc::score_emit_tc<1, kD, 1>
                       : tc::score_emit_tc<2, kD, 1>,
                       dim3(chunks_e, nu), block, bytes, st, ea.wait_prior != 0, 1, tmK, ea);
    }
    return rc;
}

constexpr EmitExtras kPlainEmit{nullptr, 0, 0};

inline bool tc_mass(const __nv_bfloat16 *, const Dims &d) { (void)d; return !env_int("GRAPHKV_FORCE_SIMT", 0); }
inline bool tc_mass(const float *, const Dims &) { return false; }

inline graphkv_status run_mass(const Dims &d, const Layout &l, const __nv_bfloat16 *Q,
                               const __nv_bfloat16 *K, float *a, void *ws, cudaStream_t st,
                               const EmitExtras &ex = kPlainEmit)
{
    if (!tc_mass(Q, d)) return run_mass_simt(d, l, Q, K, a, ws, st);
    return d.D == 64 ? run_mass_tc<64>(d, l, Q, K, a, ws, st, ex) : run_mass_tc<kHeadDim>(d, l, Q, K, a, ws, st, ex);
}
inline graphkv_status run_mass(const Dims &d, const Layout &l, const float *Q, const float *K,
                               float *a, void *ws, cudaStream_t st, const EmitExtras & = kPlainEmit)
{
    return run_mass_simt(d, l, Q, K, a, ws, st);
}

// ---- row-wise stages on clusters -------------------------------------------------------------
template <typename Args>
graphkv_status launch_cluster(const char *name, void (*kern)(Args), Args args, int clusters, int C,
                              size_t smem, cudaStream_t st)
{
    static std::mutex mu;
    static signed char state[64] = {};
    if (!once_per_device(mu, state, [] {
        const size_t mx = kMaxSmem;
        return set_smem(cs::pool_select_kernel<1>, mx) && set_smem(cs::pool_select_kernel<2>, mx) &&
                  set_smem(cs::pool_select_kernel<4>, mx) && set_smem(cs::pool_select_kernel<8>, mx) &&
                  set_smem(cs::pool_select_kernel<16>, mx) && set_smem(cs::pool_select_kernel<32>, mx) &&
                  set_smem(cs::finish_kernel, mx);
        }))
        return GRAPHKV_ERR_CUDA;
    args.wait_prior = next_launch_is_dependent();
    return launch_ex(name, kern, dim3(clusters * C), dim3(cs::kThreads), smem, st, args.wait_prior != 0, C,
                     args);
}

// Pooling of a -> s (when a != nullptr) and the k source nodes of Eq. 2 (when k > 0).
// `zero` (optional): zero_words words per unit cleared on the way, for the kernels that follow.
// `mass_hist` (optional): per unit, a histogram of values the scores dominate (see the kernel).
graphkv_status run_pool_sources(const Dims &d, const float *a, float *s, int k, int *src,
                                const uint32_t *mass_hist, uint32_t *zero, int zero_words,
                                cudaStream_t st, uint32_t *row_hist = nullptr)
{
    if (!a && k == 0) return GRAPHKV_OK;
    const ClusterPlan cp = cluster_plan(d);
    if (cp.ok) {
        cs::PoolSelectArgs pa{d, cp.C, cp.chunk, a ? cp.halo : 0, 0, a, s, k, src, mass_hist, zero, zero_words, 0, row_hist};
        const char *name = a ? (k ? "pool_select_sources" : "pool_max") : "select_sources";
        const size_t smem = cs::smem_bytes(cp.chunk, pa.halo);
        const int per = ceil_div(cp.chunk, cs::kThreads);
        void (*kern)(cs::PoolSelectArgs) =
            per <= 1 ? cs::pool_select_kernel<1> : per <= 2 ? cs::pool_select_kernel<2>
            : per <= 4 ? cs::pool_select_kernel<4> : per <= 8 ? cs::pool_select_kernel<8>
            : per <= 16 ? cs::pool_select_kernel<16> : cs::pool_select_kernel<32>;
        return launch_cluster(name, kern, pa, d.units, cp.C, smem, st);
    }
    if (zero && cudaMemsetAsync(zero, 0, (size_t)d.units * zero_words * 4, st) != cudaSuccess)
        return GRAPHKV_ERR_CUDA;
    if (a)
        GKV_LAUNCH("pool_max", st,
                   (pool_max_kernel<<<dim3(ceil_div(d.N, 256), d.units), 256, 0, st>>>(d.N, d.kp, d.pool_avg, a, s)));
    if (k > 0) {
        SelectArgs sa{s, d.N, d.N, k, nullptr, src, nullptr};
        GKV_LAUNCH("select_sources", st, (topk_select_kernel<<<d.units, kSelectThreads, 0, st>>>(sa)));
    }
    return launch_status();
}

// ---- steps (II)+(III): the graph ------------------------------------------------------------------
inline bool graph_active(const Dims &d) { return d.K_src > 0 && d.T > 0 && d.m > 0; }

// Edges of the sources (Eq. 1) and their top-m neighbourhoods (Eq. 3) -> neighbour lists in the
// workspace.  `src` holds the sources in ascending position.
// The tensors an edge compares: the sources' vectors come from S, the swept vectors from A.
template <typename T> struct EdgeOperands {
    const T *S;
    const long long *ss;
    const T *A;
    const long long *as;
};

template <int NP, int kD>
graphkv_status launch_similarity(const CUtensorMap &tmK, const tc::SimTcArgs &sa, dim3 grid, dim3 block, cudaStream_t st)
{
    static std::mutex mu;
    static signed char state[64] = {};
    if (!once_per_device(mu, state, [] { return set_smem(tc::similarity_tc<NP, kD>, tc::sim_smem_bytes<NP, kD>()); }))
        return GRAPHKV_ERR_CUDA;
    return launch_ex("similarity_tc", tc::similarity_tc<NP, kD>, grid, block, tc::sim_smem_bytes<NP, kD>(), st,
                     sa.wait_prior != 0, 1, tmK, sa);
}

// Keys from one slice of the sample to the next.
inline int slice_step(const Dims &d, const SimPlan &sp) { return ceil_div(d.N, sp.sample * tc::kSlices); }

// Bounds from a sample of the row, then one sweep for all sources (sim_stream.cuh).
template <int kD>
graphkv_status run_stream(const Dims &d, const Layout &l, const SimPlan &sp, const CUtensorMap &tmK, const CUtensorMap &tmSlices, const __nv_bfloat16 *S,
                          const long long *ss, const int *src, void *ws, cudaStream_t st)
{
    static std::mutex mu;
    static signed char state[64] = {};
    if (!once_per_device(mu, state, [] {
            return set_smem(tc::similarity_tc<32, kD, true>, tc::sim_smem_bytes<32, kD>()) && set_smem(tc::sim_stream_tc<kD>, kMaxSmem);
        }))
        return GRAPHKV_ERR_CUDA;
    tc::SimTcArgs ba{d, S, {ss[0], ss[1], ss[2]}, src, nullptr, nullptr, at<int>(ws, l.status), 0, sp.sample_ctas, sp.sample,
                     d.D == 64 ? 8 : 5, 0, wait_cycles(), slice_step(d, sp), at<float>(ws, l.tau), env_int("GRAPHKV_DEBUG_WITHHOLD_COMMIT", 0) == 3};
    ba.wait_prior = next_launch_is_dependent();
    const graphkv_status rc = launch_ex("similarity_bounds", tc::similarity_tc<32, kD, true>, dim3(sp.sample_ctas, d.units, ceil_div(d.K_src, 32)),
                                        dim3(tc::kSimThreads), tc::sim_smem_bytes<32, kD>(), st, ba.wait_prior != 0, sp.sample_ctas, tmSlices, ba);
    if (rc != GRAPHKV_OK) return rc;
    tc::SimStreamArgs sa{d, S, {ss[0], ss[1], ss[2]}, src, at<float>(ws, l.tau), at<Cand>(ws, l.cand), at<uint32_t>(ws, l.cand_hist),
                         at<uint2>(ws, l.spill), at<int>(ws, l.status), sp.chunks, sp.n_tiles, sp.NP, sp.stages, 0, wait_cycles(), env_int("GRAPHKV_DEBUG_WITHHOLD_COMMIT", 0) == 4};
    sa.wait_prior = next_launch_is_dependent();
    return launch_ex("similarity_stream", tc::sim_stream_tc<kD>, dim3(sp.chunks, d.units, ceil_div(d.K_src, sp.NP)), dim3(tc::kStreamThreads),
                     tc::stream_layout<kD>(sp.NP, sp.stages).bytes, st, sa.wait_prior != 0, 1, tmK, sa);
}

template <typename T>
graphkv_status run_graph(const Dims &d, const Layout &l, const EdgeOperands<T> &eo, const int *src, void *ws,
                         cudaStream_t st)
{
    const SimPlan sp = sim_plan(d, sizeof(T) == 2);
    if (sp.ok) {
        CUtensorMap tmK;
        if (!make_k_tensormap(&tmK, eo.A, d, d.L, eo.as)) return GRAPHKV_ERR_CUDA;
        if (sp.stream) {
            CUtensorMap tmSlices;
            if (!make_k_tensormap(&tmSlices, eo.A, d, d.L, eo.as, slice_step(d, sp))) return GRAPHKV_ERR_CUDA;
            const auto *S = reinterpret_cast<const __nv_bfloat16 *>(eo.S);
            return d.D == 64 ? run_stream<64>(d, l, sp, tmK, tmSlices, S, eo.ss, src, ws, st) : run_stream<128>(d, l, sp, tmK, tmSlices, S, eo.ss, src, ws, st);
        }
        const int group = units_per_group(d);
        for (int u0 = 0; u0 < d.units; u0 += group) {
            const int nu = std::min(group, d.units - u0);
            // one launch takes every source: grid.z counts the sweeps of sp.NP sources each
            tc::SimTcArgs sa{d, reinterpret_cast<const __nv_bfloat16 *>(eo.S), {eo.ss[0], eo.ss[1], eo.ss[2]}, src, at<Cand>(ws, l.cand),
                             at<uint32_t>(ws, l.cand_hist), at<int>(ws, l.status), u0, sp.chunks,
                             sp.n_tiles, sp.stages, 0, wait_cycles(), 0, nullptr, 0};
            sa.wait_prior = next_launch_is_dependent();
            const dim3 grid(sp.chunks, nu, ceil_div(d.K_src, sp.NP)), block(tc::kSimThreads);
            const auto launch = d.D == 64 ? (sp.NP == 16 ? launch_similarity<16, 64> : sp.NP == 32 ? launch_similarity<32, 64>
                                                                                                  : launch_similarity<64, 64>)
                                          : (sp.NP == 16 ? launch_similarity<16, 128> : sp.NP == 32 ? launch_similarity<32, 128>
                                                                                                   : launch_similarity<64, 128>);
            const graphkv_status rc = launch(tmK, sa, grid, block, st);
            if (rc != GRAPHKV_OK) return rc;
        }
        return GRAPHKV_OK;
    }
    float *sims = at<float>(ws, l.sims);
    const dim3 grid_sim(ceil_div(d.N, kSimtKeys), d.units);
    const Strides3 st_s{{eo.ss[0], eo.ss[1], eo.ss[2]}}, st_a{{eo.as[0], eo.as[1], eo.as[2]}};
    const auto sim = d.D == 64 ? similarity_simt<T, 64> : similarity_simt<T, 128>;
    const size_t smem = d.D == 64 ? sim_simt_smem_bytes<64>() : sim_simt_smem_bytes<128>();
    const graphkv_status rc = launch_ex("similarity_simt", sim, grid_sim, dim3(kSimtThreads), smem, st,
                                        next_launch_is_dependent(), 1, d, eo.S, st_s, eo.A, st_a, src, sims);
    if (rc != GRAPHKV_OK) return rc;
    SelectArgs na{sims, d.N, d.N, d.m, src, at<int>(ws, l.nbr_idx), at<float>(ws, l.nbr_e)};
    return launch_ex("select_neighbors", topk_select_kernel, dim3(d.units * d.K_src), dim3(kSelectThreads), 0, st,
                     next_launch_is_dependent(), 1, na);
}

// The finishing kernel that holds the whole row of scores in the shared memory of a cluster, an equal chunk
// per CTA (cluster_select.cuh): it takes what the one below does not.
struct FinishPlan {
    bool ok;
    int C, chunk;
};

FinishPlan finish_plan(const Dims &d, int halo)
{
    FinishPlan p{false, 1, 0};
    if (env_int("GRAPHKV_NO_CLUSTER", 0) || halo > cs::kMaxHalo) return p;
    const ClusterPlan cp = cluster_plan(d);
    p.C = cp.C;
    p.chunk = cp.chunk;
    p.ok = p.chunk <= cs::kMaxChunk;
    return p;
}

// Rows up to this length are candidates as a whole: no histogram, no bits.
constexpr int kDenseRow = 4096;

// Per-batch-element budgets of the call in flight (graphkv_compress_layers), or none.
thread_local const int32_t *t_budgets = nullptr;
// The caller of the call in flight wants the final scores (graphkv_compress without scores_out
// does not: its last kernel then leaves them in shared memory).
thread_local bool t_keep_scores = true;

// The finishing kernel that works on the candidates of a row (row_finish.cuh).
struct CandidatePlan {
    bool ok;
    int C, chunk, dense, cap, sel_cap, list_bytes;
    size_t smem;
};

CandidatePlan candidate_plan(const Dims &d, bool has_graph, bool do_select, bool keep_scores, int max_budget)
{
    CandidatePlan p{};
    if (env_int("GRAPHKV_NO_CLUSTER", 0) || d.N > rf::kMaxRow) return p;
    const long long pairs = has_graph ? (long long)d.K_src * d.m : 0;
    if (pairs > 16384) return p;
    const bool raises = has_graph && d.signal == GRAPHKV_SIGNAL_ENHANCE;
    const int need = do_select ? (int)std::min<long long>(d.N, max_budget + (raises ? 0 : pairs)) : 0;
    p.dense = d.N <= kDenseRow || (do_select && 2LL * need > d.N);
    // room for half as many again: the digit of the last one needed brings its fellows along
    p.sel_cap = p.dense ? d.N : std::min(d.N, need + need / 2 + 256);
    p.cap = p.dense ? d.N : std::min<long long>(d.N, p.sel_cap + (has_graph && (keep_scores || !do_select || raises) ? pairs : 0));
    p.cap = (p.cap + 31) & ~31;
    p.list_bytes = (int)(std::max<long long>(8 * pairs, do_select ? 4LL * max_budget : 0) + 15) & ~15;
    p.smem = rf::smem_bytes(d.N, p.cap, p.list_bytes, p.dense);
    p.C = 1;
    while (p.C < rf::kMaxCluster && d.units * p.C * 2 <= sm_count()) p.C *= 2;
    p.chunk = (ceil_div(d.N, p.C) + 31) & ~31;
    p.ok = p.smem <= kMaxSmem;
    return p;
}

// Decay rounds (when has_graph) on s in place, then (when do_select) the budget selection and
// the gather of the compact cache.
graphkv_status run_finish(const Dims &d, const Layout &l, int elem_bytes, const float *a, float *s,
                          bool has_graph, bool merge, bool do_select, const void *K, const void *V,
                          void *K_out, void *V_out, int *idx_out, void *ws, cudaStream_t st,
                          const uint32_t *row_hist = nullptr)
{
    if (!has_graph && !do_select && !a) return GRAPHKV_OK;
    const bool keep = has_graph && (t_keep_scores || !do_select);
    const CandidatePlan cd = a ? CandidatePlan{} : candidate_plan(d, has_graph, do_select, keep, d.B);
    if (cd.ok) {
        rf::FinishArgs fa{};
        fa.d = d;
        fa.C = cd.C;
        fa.chunk = cd.chunk;
        fa.dense = cd.dense;
        fa.cap = cd.cap;
        fa.sel_cap = cd.sel_cap;
        fa.list_bytes = cd.list_bytes;
        // enough groups for every source at once where that leaves a group more than one warp
        fa.group_warps = d.K_src <= 4 * cd.C ? 4 : d.K_src <= 8 * cd.C ? 2 : 1;
        fa.row_hist = row_hist;
        fa.s = s;
        fa.nbr_idx = at<int>(ws, l.nbr_idx);
        fa.nbr_e = at<float>(ws, l.nbr_e);
        fa.has_graph = has_graph;
        fa.merge = has_graph && merge;
        fa.cand = at<Cand>(ws, l.cand);
        fa.cand_hist = at<uint32_t>(ws, l.cand_hist);
        fa.cand_chunks = merge ? sim_plan(d, d.bf16 != 0).chunks : 0;
        fa.do_select = do_select;
        fa.idx_out = idx_out;
        fa.elem_bytes = elem_bytes;
        for (fa.vpr_log2 = 0; (16 << fa.vpr_log2) < d.D * elem_bytes;) ++fa.vpr_log2;
        fa.K = static_cast<const unsigned char *>(K);
        fa.V = static_cast<const unsigned char *>(V);
        fa.K_out = static_cast<unsigned char *>(K_out);
        fa.V_out = static_cast<unsigned char *>(V_out);
        fa.early_row = has_graph;
        fa.keep_scores = keep;
        if (t_budgets && do_select) {
            fa.per_batch_budget = 1;
            for (int i = 0; i < d.batch; ++i) fa.budget_of[i] = t_budgets[i];
        }
        static std::mutex mu;
        static signed char state[64] = {};
        if (!once_per_device(mu, state, [] { return set_smem(rf::finish_kernel, kMaxSmem); })) return GRAPHKV_ERR_CUDA;
        fa.wait_prior = next_launch_is_dependent();
        const char *name = has_graph ? (do_select ? "decay_select_gather" : "decay_rounds") : "select_gather";
        return launch_ex(name, rf::finish_kernel, dim3(d.units * cd.C), dim3(rf::kThreads), cd.smem, st,
                         fa.wait_prior != 0, cd.C, fa);
    }
    const int halo = a ? (d.kp - 1) / 2 : 0;
    const FinishPlan fp = finish_plan(d, halo);
    if (fp.ok && cluster_plan(d).ok) {
        cs::FinishArgs fa{d, fp.C, fp.chunk, halo, 0, a, s, at<int>(ws, l.nbr_idx), at<float>(ws, l.nbr_e),
                          has_graph ? 1 : 0, has_graph && merge ? 1 : 0, at<Cand>(ws, l.cand),
                          at<uint32_t>(ws, l.cand_hist), sim_plan(d, d.bf16 != 0).chunks, do_select ? 1 : 0, idx_out, elem_bytes,
                          static_cast<const unsigned char *>(K), static_cast<const unsigned char *>(V),
                          static_cast<unsigned char *>(K_out), static_cast<unsigned char *>(V_out), 0, cs::kStage,
                          (t_keep_scores || !do_select) ? 1 : 0, 0, {}};
        if (t_budgets && do_select) {
            fa.per_batch_budget = 1;
            for (int i = 0; i < d.batch; ++i) fa.budget_of[i] = t_budgets[i];
        }
        // the neighbour lists of a unit are staged in shared memory when K_src * m entries fit
        const int pairs = has_graph ? d.K_src * d.m : 0;
        if (pairs > cs::kStage && cs::smem_bytes(fp.chunk, halo, (pairs + 255) & ~255) <= kMaxSmem)
            fa.stage_cap = (pairs + 255) & ~255;
        const char *name = has_graph ? (do_select ? "decay_select_gather" : "decay_rounds") : "select_gather";
        return launch_cluster(name, cs::finish_kernel, fa, d.units, fp.C,
                              cs::smem_bytes(fp.chunk, halo, fa.stage_cap), st);
    }
    if (t_budgets && do_select) return GRAPHKV_ERR_UNSUPPORTED;      // only the cluster kernel takes budgets per layer
    if (a)
        GKV_LAUNCH("pool_max", st,
                   (pool_max_kernel<<<dim3(ceil_div(d.N, 256), d.units), 256, 0, st>>>(d.N, d.kp, d.pool_avg, a, s)));
    if (has_graph)
        GKV_LAUNCH("decay_rounds", st,
                   (decay_rounds_kernel<<<d.units, 256, 0, st>>>(d, at<int>(ws, l.nbr_idx),
                                                                 at<float>(ws, l.nbr_e), s)));
    if (do_select) {
        SelectArgs sa{s, d.N, d.N, d.B, nullptr, idx_out, nullptr};
        GKV_LAUNCH("select_budget", st, (topk_select_kernel<<<d.units, kSelectThreads, 0, st>>>(sa)));
        if (K || V) {
            const long long total = (long long)d.units * (d.B + d.W) * (d.D * elem_bytes / 16);
            const int blocks = (int)std::min<long long>((total + kGatherThreads - 1) / kGatherThreads,
                                                        148LL * 16);
            GKV_LAUNCH("gather_rows", st,
                       (gather_rows_kernel<<<blocks, kGatherThreads, 0, st>>>(
                           d, elem_bytes, static_cast<const unsigned char *>(K),
                           static_cast<const unsigned char *>(V), idx_out,
                           static_cast<unsigned char *>(K_out), static_cast<unsigned char *>(V_out))));
        }
    }
    return launch_status();
}


// ---- the whole path in one kernel (cluster_path.cuh) ------------------------------------------------
struct ClusterPathPlan {
    bool ok;
    int C, n_tiles;
    cp::Sizes z;
    size_t smem;
};

ClusterPathPlan cluster_path_plan(const Dims &d, bool graph)
{
    ClusterPathPlan p{};
    if (units_per_group(d) < d.units || (graph && !short_row_graph(d))) return p;
    const ShortRow sr = short_row(d);
    if (sr.C == 0) return p;
    p.C = sr.C;
    p.n_tiles = ceil_div(d.L, tc::kTileKeys);
    p.z = cp::Sizes{d.N, sr.C, d.GW, sr.tiles, !graph || d.K_src <= 16 ? 16 : d.K_src <= 32 ? 32 : 64, 0,
                    graph ? (d.K_src * d.m * 8 + 15) / 16 * 16 : 0, (d.B * 4 + 15) / 16 * 16, 0};
    const auto layout_of_path = !d.bf16 ? (d.D == 64 ? cp::layout_f32<64> : cp::layout_f32<128>) : d.D == 64 ? (d.GW <= 128 ? cp::layout<64, 1> : cp::layout<64, 2>)
                                          : (d.GW <= 128 ? cp::layout<128, 1> : cp::layout<128, 2>);
    // The cosines of all a CTA's sources at once where that fits, in the tiles' place if need be: a second round costs more than
    // the barrier of that place (5000 tokens x 8 heads, 16 sources: 43.0 -> 38.4 us, with inputs and code out of the caches 63.5 ->
    // 57.3; 7000 x 2 46.6 -> 40.9, 65.5 -> 59.4; 8191 x 4 at D = 64 49.1 -> 43.4, 67.6 -> 61.4).
    const int per_cta = graph ? ceil_div(d.K_src, p.C) : 0;
    for (int rounds = 1; rounds <= std::max(1, std::min(2, per_cta)) && !p.ok; ++rounds)
        for (int in_tiles = 0; in_tiles <= (graph && d.bf16 ? 1 : 0) && !p.ok; ++in_tiles) {
            p.z.cosines_in_tiles = in_tiles;
            p.z.rows = ceil_div(per_cta, rounds);
            p.smem = layout_of_path(p.z).total;
            p.ok = p.smem <= kMaxSmem;
        }
    return p;
}
bool cluster_path_on()
{
    for (const char *off : {"GRAPHKV_NO_CLUSTER", "GRAPHKV_FORCE_SIMT", "GRAPHKV_TWO_SCORE_KERNELS"})
        if (env_int(off, 0)) return false;
    return env_int("GRAPHKV_DEBUG_WITHHOLD_COMMIT", 0) != 2;
}
// Key chunks of the row statistics of a row whose scores the cluster path can take (0: as suits the sweep): the general
// kernels cut it the same way, so that a call has the same bits on either path, in stages or fused, whatever its graph.
inline int short_row_chunks(const Dims &d)
{
    const ClusterPathPlan p = cluster_path_plan(d, false);
    return p.ok ? p.C : 0;
}

template <int kD, int kR, int kRowTiles, int kKeys> bool cluster_path_f32_ready()
{
    static std::mutex mu;
    static signed char state[64] = {};
    return once_per_device(mu, state, [] {
        return set_smem(cp::cluster_path_f32_kernel<kD, kR, kRowTiles, kKeys>, kMaxSmem) &&
               cudaFuncSetAttribute(cp::cluster_path_f32_kernel<kD, kR, kRowTiles, kKeys>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    });
}

graphkv_status run_cluster_path(const Dims &d, const Layout &l, const ClusterPathPlan &pl, const void *Q,
                                const void *K, const void *V, void *K_out, void *V_out, int *idx_out, float *scores,
                                bool scores_only, bool graph, void *ws, cudaStream_t st)
{
    CUtensorMap tmK;
    if (d.bf16 && !make_k_tensormap(&tmK, K, d, d.L)) return GRAPHKV_ERR_CUDA;
    cp::PathArgs a{};
    a.d = d;
    a.Q = Q;
    a.K = K;
    a.C = pl.C;
    a.n_tiles = pl.n_tiles;
    a.z = pl.z;
    a.status = at<int>(ws, l.status);
    a.scores = scores;
    a.scores_only = scores_only;
    a.has_graph = graph;
    if (!scores_only) {
        a.src_out = at<int>(ws, l.src);
        a.nbr_idx = at<int>(ws, l.nbr_idx);
        a.nbr_e = at<float>(ws, l.nbr_e);
        a.idx_out = idx_out;
        a.vpr_log2 = (d.D == 64 ? 3 : 4) + (d.bf16 ? 0 : 1);
        a.Kb = static_cast<const unsigned char *>(K);
        a.V = static_cast<const unsigned char *>(V);
        a.K_out = static_cast<unsigned char *>(K_out);
        a.V_out = static_cast<unsigned char *>(V_out);
        if (t_budgets) {
            a.per_batch_budget = 1;
            for (int i = 0; i < d.batch; ++i) a.budget_of[i] = t_budgets[i];
        }
    }
    a.wait_cycles = wait_cycles();
    a.withhold_commit = env_int("GRAPHKV_DEBUG_WITHHOLD_COMMIT", 0);
    auto launch_f32 = [&](auto kern, bool ready) -> graphkv_status {
        if (!ready) return GRAPHKV_ERR_CUDA;
        return launch_ex("cluster_path", kern, dim3(d.units * pl.C), dim3(cp::kThreads), pl.smem, st, next_launch_is_dependent(), pl.C, a);
    };
    if (!d.bf16) {
#define GKV_F32(kD, kR, kRowTiles, kKeys) \
    launch_f32(cp::cluster_path_f32_kernel<kD, kR, kRowTiles, kKeys>, cluster_path_f32_ready<kD, kR, kRowTiles, kKeys>())
        const int rows = d.GW <= 32 ? 0 : d.GW <= 64 ? 1 : 2;
        if (pl.z.tiles == 1) {
            if (d.D == 64) return rows == 0 ? GKV_F32(64, 1, 1, 64) : rows == 1 ? GKV_F32(64, 2, 1, 64) : GKV_F32(64, 4, 1, 64);
            return rows == 0 ? GKV_F32(128, 1, 1, 64) : rows == 1 ? GKV_F32(128, 2, 1, 64) : GKV_F32(128, 4, 1, 64);
        }
        if (d.D == 64) return rows == 0 ? GKV_F32(64, 2, 1, 128) : rows == 1 ? GKV_F32(64, 4, 1, 128) : GKV_F32(64, 4, 2, 128);
        return rows == 0 ? GKV_F32(128, 2, 1, 128) : rows == 1 ? GKV_F32(128, 4, 1, 128) : GKV_F32(128, 4, 2, 128);
#undef GKV_F32
    }
    auto launch = [&](auto kern, bool ready) -> graphkv_status {
        if (!ready) return GRAPHKV_ERR_CUDA;
        return launch_ex("cluster_path", kern, dim3(d.units * pl.C), dim3(cp::kThreads), pl.smem, st,
                         next_launch_is_dependent(), pl.C, tmK, a);
    };
    if (d.D == 64)
        return d.GW <= 128 ? launch(cp::cluster_path_kernel<64, 1>, cluster_path_ready<64, 1>())
                           : launch(cp::cluster_path_kernel<64, 2>, cluster_path_ready<64, 2>());
    return d.GW <= 128 ? launch(cp::cluster_path_kernel<128, 1>, cluster_path_ready<128, 1>())
                       : launch(cp::cluster_path_kernel<128, 2>, cluster_path_ready<128, 2>());
}

// ---- the calls, typed ---------------------------------------------------------------------------

template <typename T>
graphkv_status do_score(const Dims &d, const Layout &l, const T *Q, const T *K, float *scores,
                        void *ws, cudaStream_t st)
{
    EmitExtras ex = kPlainEmit;
    const ClusterPathPlan pl = cluster_path_plan(d, false);
    ex.stat_chunks = pl.ok ? pl.C : 0;
    if (pl.ok && cluster_path_on()) return run_cluster_path(d, l, pl, Q, K, nullptr, nullptr, nullptr, nullptr, scores, true, false, ws, st);
    float *a = d.kp > 1 ? at<float>(ws, l.a) : scores;
    graphkv_status rc = run_mass(d, l, Q, K, a, ws, st, ex);
    if (rc != GRAPHKV_OK || d.kp == 1) return rc;
    return run_pool_sources(d, a, scores, 0, nullptr, nullptr, nullptr, 0, st);
}

// One pass of steps (II)+(III) from the scores as they stand: sources, edges, neighbourhoods,
// d.T rounds over that graph.
template <typename T>
graphkv_status propagate_once(const Dims &d, const Layout &l, const EdgeOperands<T> &eo, float *scores,
                              int *src, void *ws, cudaStream_t st)
{
    const bool tc_graph = graph_active(d) && sim_plan(d, sizeof(T) == 2).ok;
    graphkv_status rc = run_pool_sources(d, nullptr, scores, d.K_src, src, nullptr,
                                         tc_graph ? at<uint32_t>(ws, l.cand_hist) : nullptr,
                                         d.K_src * kCandBins, st);
    if (rc != GRAPHKV_OK || !graph_active(d)) return rc;
    if ((rc = run_graph(d, l, eo, src, ws, st)) != GRAPHKV_OK) return rc;
    return run_finish(d, l, (int)sizeof(T), nullptr, scores, true, sim_plan(d, sizeof(T) == 2).ok, false,
                      nullptr, nullptr, nullptr, nullptr, nullptr, ws, st);
}

// Steps (II)+(III).  With d.reselect every round is a pass of its own: the sources are re-picked
// from the scores the round before left and their neighbourhoods rebuilt (src_out then holds the
// sources of the last round).
template <typename T>
graphkv_status do_propagate(const Dims &d, const Layout &l, const EdgeOperands<T> &eo, float *scores,
                            int *src_out, void *ws, cudaStream_t st)
{
    if (d.K_src == 0) return GRAPHKV_OK;
    int *src = src_out ? src_out : at<int>(ws, l.src);
    if (!d.reselect || d.T <= 1) return propagate_once(d, l, eo, scores, src, ws, st);
    Dims one = d;
    one.T = 1;
    for (int t = 0; t < d.T; ++t) {
        const graphkv_status rc = propagate_once(one, l, eo, scores, src, ws, st);
        if (rc != GRAPHKV_OK) return rc;
    }
    return GRAPHKV_OK;
}

template <typename T>
graphkv_status do_compress(const Dims &d, const Layout &l, const T *Q, const T *K, const void *V,
                           void *K_out, void *V_out, int *idx_out, float *s, void *ws,
                           cudaStream_t st)
{
    const bool graph = graph_active(d);
    EmitExtras ex = kPlainEmit;
    bool scored = false;                    // `s` holds the pooled scores already
    {
        const ClusterPathPlan pl = cluster_path_plan(d, graph);
        if (pl.ok && cluster_path_on())
            return run_cluster_path(d, l, pl, Q, K, V, K_out, V_out, idx_out, t_keep_scores ? s : nullptr, false, graph, ws, st);
        // a graph that the cluster path does not take: the scores must not depend on it
        if (sizeof(T) == 2) {
            ex.stat_chunks = pl.ok ? pl.C : short_row_chunks(d);
        } else if (const ClusterPathPlan ps = cluster_path_plan(d, false); ps.ok && cluster_path_on()) {
            const graphkv_status rc = run_cluster_path(d, l, ps, Q, K, nullptr, nullptr, nullptr, nullptr, s, true, false, ws, st);
            if (rc != GRAPHKV_OK) return rc;
            scored = true;
        }
    }
    float *a = d.kp > 1 ? at<float>(ws, l.a) : s;
    int *src = at<int>(ws, l.src);
    const bool tc_graph = graph && sim_plan(d, sizeof(T) == 2).ok;
    // without a graph (plain top-B) the old finishing kernel pools where the new one does not apply
    const bool finish_pools = !graph && !scored && d.kp > 1 && !d.pool_avg && !candidate_plan(d, false, true, false, d.B).ok &&
                              finish_plan(d, (d.kp - 1) / 2).ok && cluster_plan(d).ok;
    graphkv_status rc;
    uint32_t *row_hist = nullptr;
    if (!graph) {
        if (!scored && (rc = run_mass(d, l, Q, K, a, ws, st, ex)) != GRAPHKV_OK) return rc;
        if (!scored && d.kp > 1 && !finish_pools &&
            (rc = run_pool_sources(d, a, s, 0, nullptr, nullptr, nullptr, 0, st)) != GRAPHKV_OK)
            return rc;
    } else {
        // (the sweeps clear the words the pooling kernel counts the scores in)
        if (cluster_plan(d).ok && tc_mass(Q, d) && (!d.reselect || d.T <= 1)) {
            const CandidatePlan cd = candidate_plan(d, true, true, t_keep_scores, d.B);
            if (cd.ok && !cd.dense) row_hist = at<uint32_t>(ws, l.row_hist);
        }
        ex.zero = row_hist;
        ex.zero_words = cs::kBins;
        if (!scored && (rc = run_mass(d, l, Q, K, a, ws, st, ex)) != GRAPHKV_OK) return rc;
        // the tensor-core emit sweep leaves a histogram of the attention mass behind
        rc = run_pool_sources(d, d.kp > 1 && !scored ? a : nullptr, s, d.K_src, src,
                              tc_mass(Q, d) ? at<uint32_t>(ws, l.a_hist) : nullptr,
                              tc_graph ? at<uint32_t>(ws, l.cand_hist) : nullptr, d.K_src * kCandBins, st, row_hist);
        if (rc != GRAPHKV_OK) return rc;
    }
    const EdgeOperands<T> eo{K, d.ks, K, d.ks};
    if (graph && d.reselect && d.T > 1) {
        // every round its own pass: the first one rides on the sources picked above, the rounds
        // after it start from the scores in `s`; the last pass also selects and gathers
        Dims one = d;
        one.T = 1;
        if ((rc = run_graph(one, l, eo, src, ws, st)) != GRAPHKV_OK) return rc;
        if ((rc = run_finish(one, l, (int)sizeof(T), finish_pools ? a : nullptr, s, true, tc_graph, false,
                             nullptr, nullptr, nullptr, nullptr, nullptr, ws, st)) != GRAPHKV_OK)
            return rc;
        for (int t = 1; t < d.T; ++t)
            if ((rc = propagate_once(one, l, eo, s, src, ws, st)) != GRAPHKV_OK) return rc;
        return run_finish(one, l, (int)sizeof(T), nullptr, s, false, false, true, K, V, K_out, V_out, idx_out,
                          ws, st);
    }
    if (graph && (rc = run_graph(d, l, eo, src, ws, st)) != GRAPHKV_OK) return rc;
    return run_finish(d, l, (int)sizeof(T), finish_pools ? a : nullptr, s, graph, tc_graph, true, K, V,
                      K_out, V_out, idx_out, ws, st, row_hist);
}

// ---- KNorm initial score ---------------------------------------------------------------------
// s_j = 1 / max(||k_j||, eps) for the prefix keys: 16 threads share a key row (16 bytes each of a
// bf16 row, 32 of an fp32 row), eight rows in flight per thread.  grid (CTAs per unit, units).
template <typename T, int kD>
__global__ void __launch_bounds__(256) knorm_score_kernel(Dims d, const T *__restrict__ K, float *__restrict__ scores)
{
    constexpr int kTpr = kD / 8;                 // threads per key row, eight elements each
    const int sub = threadIdx.x & (kTpr - 1), unit = blockIdx.y;
    const T *Kh = K + (unit / d.hkv) * d.ks[0] + (long long)(unit % d.hkv) * d.ks[1] + sub * 8;
    float *out = scores + (long long)unit * d.N;
    const int stride = (gridDim.x * blockDim.x) / kTpr;
    pdl_wait();
    pdl_launch_dependents();
    for (int j0 = (blockIdx.x * blockDim.x + threadIdx.x) / kTpr; j0 < d.N; j0 += 8 * stride) {
        float n2[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int j = j0 + u * stride;
            n2[u] = 0.f;
            if (j < d.N) {
                float v[8];
                load8(Kh + (long long)j * d.ks[2], v);
#pragma unroll
                for (int e = 0; e < 8; ++e) n2[u] = fmaf(v[e], v[e], n2[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
#pragma unroll
            for (int o = kTpr / 2; o > 0; o >>= 1) n2[u] += __shfl_xor_sync(0xffffffffu, n2[u], o);
            const int j = j0 + u * stride;
            if (sub == 0 && j < d.N) out[j] = 1.0f / fmaxf(sqrtf(n2[u]), kNormEps);
        }
    }
}

// ---- built-in scratch for graphkv_score_noalloc ---------------------------------------------------
// Device memory that is part of the library image.  In host code the array's name is only a handle
// for cudaGetSymbolAddress; kernels get the address looked up once per device.
static __device__ __align__(256) unsigned char g_builtin_scratch[GRAPHKV_BUILTIN_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_builtin_mu;
void *g_builtin_ptr[kMaxDevices] = {};

// Address of the built-in scratch on the current device (nullptr on failure).
void *builtin_scratch()
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lk(g_builtin_mu);
    if (!g_builtin_ptr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_builtin_scratch) != cudaSuccess) return nullptr;
        g_builtin_ptr[dev] = p;
    }
    return g_builtin_ptr[dev];
}

}  // namespace

extern "C" {

int32_t graphkv_resolve_neighbors(int32_t n_prefix, int32_t neighbors)
{
    if (neighbors > 0) return neighbors;
    int32_t m = n_prefix / 1000;
    m = m < 1 ? 1 : (m > 32 ? 32 : m);
    if (m > n_prefix - 1) m = n_prefix - 1;
    return m;
}

size_t graphkv_workspace_bytes(const graphkv_params *params)
{
    Dims d;
    if (resolve(params, &d) != GRAPHKV_OK) return 0;
    return layout_of(d).total;
}

graphkv_status graphkv_score(const graphkv_params *params, const void *Qw, const void *K,
                             float *scores, void *workspace, size_t workspace_bytes, void *stream)
{
    Dims d;
    graphkv_status rc = resolve(params, &d);
    if (rc != GRAPHKV_OK) return rc;
    t_launches_in_call = 0;
    if (!Qw || !K || !scores || !aligned16(Qw) || !aligned16(K)) return GRAPHKV_ERR_INVALID_ARG;
    const Layout l = layout_of(d);
    if ((rc = check_ws(l, workspace, workspace_bytes)) != GRAPHKV_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (params->dtype == GRAPHKV_BF16)
        return do_score(d, l, static_cast<const __nv_bfloat16 *>(Qw),
                        static_cast<const __nv_bfloat16 *>(K), scores, workspace, st);
    return do_score(d, l, static_cast<const float *>(Qw), static_cast<const float *>(K), scores,
                    workspace, st);
}

size_t graphkv_builtin_scratch_needed(const graphkv_params *params)
{
    Dims d;
    if (resolve(params, &d) != GRAPHKV_OK) return 0;
    return layout_of(d).s;       // the scoring call uses the regions laid out before `s`
}

graphkv_status graphkv_score_noalloc(const graphkv_params *params, const void *Qw, const void *K,
                                     float *scores, void *stream)
{
    Dims d;
    graphkv_status rc = resolve(params, &d);
    if (rc != GRAPHKV_OK) return rc;
    t_launches_in_call = 0;
    if (!Qw || !K || !scores || !aligned16(Qw) || !aligned16(K)) return GRAPHKV_ERR_INVALID_ARG;
    const Layout l = layout_of(d);
    if (l.s > GRAPHKV_BUILTIN_SCRATCH_BYTES) return GRAPHKV_ERR_BUILTIN_SCRATCH;
    void *ws = builtin_scratch();
    if (!ws) return GRAPHKV_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (params->dtype == GRAPHKV_BF16)
        return do_score(d, l, static_cast<const __nv_bfloat16 *>(Qw),
                        static_cast<const __nv_bfloat16 *>(K), scores, ws, st);
    return do_score(d, l, static_cast<const float *>(Qw), static_cast<const float *>(K), scores, ws, st);
}

graphkv_status graphkv_read_status_noalloc(void *stream)
{
    void *ws = builtin_scratch();
    if (!ws) return GRAPHKV_ERR_CUDA;
    return graphkv_read_status(ws, stream);
}

graphkv_status graphkv_propagate_edges(const graphkv_params *params, const void *K, const void *V,
                                       int32_t src_tensor, int32_t all_tensor, float *scores,
                                       int32_t *src_idx_out, void *workspace, size_t workspace_bytes,
                                       void *stream)
{
    Dims d;
    graphkv_status rc = resolve(params, &d);
    if (rc != GRAPHKV_OK) return rc;
    t_launches_in_call = 0;
    if ((src_tensor != GRAPHKV_TENSOR_K && src_tensor != GRAPHKV_TENSOR_V) ||
        (all_tensor != GRAPHKV_TENSOR_K && all_tensor != GRAPHKV_TENSOR_V))
        return GRAPHKV_ERR_INVALID_ARG;
    const void *S = src_tensor == GRAPHKV_TENSOR_K ? K : V, *A = all_tensor == GRAPHKV_TENSOR_K ? K : V;
    const long long *ss = src_tensor == GRAPHKV_TENSOR_K ? d.ks : d.vs;
    const long long *as = all_tensor == GRAPHKV_TENSOR_K ? d.ks : d.vs;
    if (!S || !A || !scores || !aligned16(S) || !aligned16(A)) return GRAPHKV_ERR_INVALID_ARG;
    const Layout l = layout_of(d);
    if ((rc = check_ws(l, workspace, workspace_bytes)) != GRAPHKV_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (params->dtype == GRAPHKV_BF16) {
        const EdgeOperands<__nv_bfloat16> eo{static_cast<const __nv_bfloat16 *>(S), ss,
                                             static_cast<const __nv_bfloat16 *>(A), as};
        return do_propagate(d, l, eo, scores, src_idx_out, workspace, st);
    }
    const EdgeOperands<float> eo{static_cast<const float *>(S), ss, static_cast<const float *>(A), as};
    return do_propagate(d, l, eo, scores, src_idx_out, workspace, st);
}

graphkv_status graphkv_propagate(const graphkv_params *params, const void *K, float *scores,
                                 int32_t *src_idx_out, void *workspace, size_t workspace_bytes,
                                 void *stream)
{
    return graphkv_propagate_edges(params, K, nullptr, GRAPHKV_TENSOR_K, GRAPHKV_TENSOR_K, scores,
                                   src_idx_out, workspace, workspace_bytes, stream);
}

graphkv_status graphkv_score_knorm(const graphkv_params *params, const void *K, float *scores, void *stream)
{
    Dims d;
    graphkv_status rc = resolve(params, &d);
    if (rc != GRAPHKV_OK) return rc;
    if (!K || !scores || !aligned16(K)) return GRAPHKV_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // about one wave of resident CTAs (eight of 256 threads per SM) over all units
    const int per_unit = std::max(1, std::min(ceil_div(d.N, 16 * 8), ceil_div(sm_count() * 8, d.units)));
    const dim3 grid(per_unit, d.units);
    t_launches_in_call = 0;
    auto launch = [&](auto kern, auto *keys) {
        return launch_ex("knorm_score", kern, grid, dim3(256), 0, st, next_launch_is_dependent(), 1, d, keys, scores);
    };
    const __nv_bfloat16 *Kb = static_cast<const __nv_bfloat16 *>(K);
    const float *Kf = static_cast<const float *>(K);
    if (params->dtype == GRAPHKV_BF16)
        return d.D == 64 ? launch(knorm_score_kernel<__nv_bfloat16, 64>, Kb) : launch(knorm_score_kernel<__nv_bfloat16, 128>, Kb);
    return d.D == 64 ? launch(knorm_score_kernel<float, 64>, Kf) : launch(knorm_score_kernel<float, 128>, Kf);
}

graphkv_status graphkv_select_gather(const graphkv_params *params, const float *scores,
                                     const void *K, const void *V, void *K_out, void *V_out,
                                     int32_t *idx_out, void *workspace, size_t workspace_bytes,
                                     void *stream)
{
    Dims d;
    graphkv_status rc = resolve(params, &d);
    if (rc != GRAPHKV_OK) return rc;
    t_launches_in_call = 0;
    if (!scores || !idx_out) return GRAPHKV_ERR_INVALID_ARG;
    if ((K == nullptr) != (K_out == nullptr) || (V == nullptr) != (V_out == nullptr))
        return GRAPHKV_ERR_INVALID_ARG;
    if (!aligned16(K) || !aligned16(V) || !aligned16(K_out) || !aligned16(V_out))
        return GRAPHKV_ERR_INVALID_ARG;
    const Layout l = layout_of(d);
    if ((rc = check_ws(l, workspace, workspace_bytes)) != GRAPHKV_OK) return rc;
    const int elem = params->dtype == GRAPHKV_BF16 ? 2 : 4;
    return run_finish(d, l, elem, nullptr, const_cast<float *>(scores), false, false, true, K, V, K_out,
                      V_out, idx_out, workspace, static_cast<cudaStream_t>(stream));
}

graphkv_status graphkv_compress(const graphkv_params *params, const void *Qw, const void *K,
                                const void *V, void *K_out, void *V_out, int32_t *idx_out,
                                float *scores_out, void *workspace, size_t workspace_bytes,
                                void *stream)
{
    Dims d;
    graphkv_status rc = resolve(params, &d);
    if (rc != GRAPHKV_OK) return rc;
    t_launches_in_call = 0;
    if (!Qw || !K || !V || !K_out || !V_out || !idx_out) return GRAPHKV_ERR_INVALID_ARG;
    if (!aligned16(Qw) || !aligned16(K) || !aligned16(V) || !aligned16(K_out) || !aligned16(V_out))
        return GRAPHKV_ERR_INVALID_ARG;
    const Layout l = layout_of(d);
    if ((rc = check_ws(l, workspace, workspace_bytes)) != GRAPHKV_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float *s = scores_out ? scores_out : at<float>(workspace, l.s);
    t_keep_scores = scores_out != nullptr;
    if (params->dtype == GRAPHKV_BF16)
        rc = do_compress(d, l, static_cast<const __nv_bfloat16 *>(Qw),
                         static_cast<const __nv_bfloat16 *>(K), V, K_out, V_out, idx_out, s, workspace, st);
    else
        rc = do_compress(d, l, static_cast<const float *>(Qw), static_cast<const float *>(K), V, K_out,
                         V_out, idx_out, s, workspace, st);
    t_keep_scores = true;
    return rc;
}

graphkv_status graphkv_compress_layers(const graphkv_params *params, const int32_t *budgets,
                                       const void *Qw, const void *K, const void *V, void *K_out,
                                       void *V_out, int32_t *idx_out, float *scores_out,
                                       void *workspace, size_t workspace_bytes, void *stream)
{
    if (!params || !budgets) return GRAPHKV_ERR_INVALID_ARG;
    if (params->batch > cs::kMaxBudgets) return GRAPHKV_ERR_UNSUPPORTED;
    for (int i = 0; i < params->batch; ++i)
        if (budgets[i] < 1 || budgets[i] > params->budget) return GRAPHKV_ERR_INVALID_ARG;
    t_budgets = budgets;
    const graphkv_status rc = graphkv_compress(params, Qw, K, V, K_out, V_out, idx_out, scores_out,
                                               workspace, workspace_bytes, stream);
    t_budgets = nullptr;
    return rc;
}

static bool decode_shape(const graphkv_params *p, DecodeArgs *a)
{
    if (!p || p->batch < 1 || p->n_q_heads < 1 || p->n_kv_heads < 1 || p->seq_len < 1 ||
        p->n_q_heads % p->n_kv_heads != 0 || p->head_dim != kHeadDim ||
        p->n_q_heads / p->n_kv_heads > kDecMaxG || (long long)p->batch * p->n_kv_heads > 65535 ||
        (p->dtype != GRAPHKV_BF16 && p->dtype != GRAPHKV_F32))
        return false;
    const int vec = p->dtype == GRAPHKV_BF16 ? 8 : 4;
    for (int i = 0; i < 3; ++i)
        if (p->k_stride[i] < 0 || p->v_stride[i] < 0 || p->k_stride[i] % vec || p->v_stride[i] % vec) return false;
    if (p->q_stride[0] < 0 || p->q_stride[1] < kHeadDim) return false;
    a->batch = p->batch; a->hq = p->n_q_heads; a->hkv = p->n_kv_heads; a->G = p->n_q_heads / p->n_kv_heads;
    a->rows = p->seq_len;
    a->blocks_per_unit = ceil_div(p->seq_len, p->dtype == GRAPHKV_BF16 ? dec_rows<__nv_bfloat16>() : dec_rows<float>());
    // As many CTAs per unit as one wave holds (one per SM), with kDecMinBlocks blocks each or more; a unit is one CTA from
    // 75 units on.
    const int units = p->batch * p->n_kv_heads;
    a->splits = std::max(1, std::min(sm_count() / units, ceil_div(a->blocks_per_unit, kDecMinBlocks)));
    // Somewhat more units than SMs: CTAs of half the warps, two per SM, so that no second, short wave follows (152 units
    // of 2080 rows 40.5 -> 32.2 us, 200 units 42.2 -> 38.1; 256 units, where the second wave is fuller, 46.0 against 46.6, 224 of 4096
    // rows 73.4 against 77.8).  Over short rows the waves' starts and merges weigh more, and overlap (256 units of 544 rows
    // 18.0 -> 15.4, of 128 rows 9.9 -> 7.3).  Up to 148 units splitting each over two or three such CTAs loses (96 units of 2080
    // rows 20.3 against 31.2, 128 units 25.5 against 27.1).
    a->two = units > sm_count() && (20 * units <= 27 * sm_count() || a->blocks_per_unit <= 48);
    // CTAs of a unit that fit a cluster merge through shared memory instead of global memory and a counter
    // (544 rows 6.5 -> 5.8 us).  Up to 24 blocks per CTA a cluster of eight also beats more CTAs that do not
    // fit one (1032 rows 6.8 -> 6.4 us, 3032 rows 8.5 -> 8.2; 4132 rows 9.0 -> 9.2; clusters of four lose).
    const int C = resident_cluster_size(units);
    if (C == 8 && a->splits > C && a->blocks_per_unit <= 24 * C) a->splits = C;
    a->cluster = a->splits > 1 && a->splits <= C ? 1 : 0;
    a->qs[0] = p->q_stride[0]; a->qs[1] = p->q_stride[1];
    for (int i = 0; i < 3; ++i) { a->ks[i] = p->k_stride[i]; a->vs[i] = p->v_stride[i]; }
    return true;
}

// Arrival words, parts, and room to align them: the caller's workspace may start anywhere.
static size_t decode_bytes(const DecodeArgs &a)
{
    return kAlign + align_up((size_t)a.batch * a.hkv * sizeof(unsigned long long)) +
           align_up((size_t)a.batch * a.hkv * a.splits * a.G * kDecPart * sizeof(float));
}

size_t graphkv_decode_workspace_bytes(const graphkv_params *params)
{
    DecodeArgs a;
    return decode_shape(params, &a) ? decode_bytes(a) : 0;
}

extern "C++" {
template <typename T, int kG, int kWarps>
static graphkv_status launch_decode_warps(const DecodeArgs &a, const void *q, const void *K, const void *V, cudaStream_t st)
{
    static std::mutex mu;
    static signed char state[64] = {};
    if (!once_per_device(mu, state, [] { return set_smem(decode_kernel<T, kG, kWarps>, dec_smem_bytes<kWarps>()); }))
        return GRAPHKV_ERR_CUDA;
    return launch_ex("decode_attention", decode_kernel<T, kG, kWarps>, dim3(a.splits, a.batch * a.hkv), dim3(kWarps * 32), dec_smem_bytes<kWarps>(),
                     st, next_launch_is_dependent(), a.cluster ? a.splits : 1, a, static_cast<const T *>(q), static_cast<const T *>(K),
                     static_cast<const T *>(V));
}
template <typename T, int kG>
static graphkv_status launch_decode(const DecodeArgs &a, const void *q, const void *K, const void *V, cudaStream_t st)
{
    return a.two ? launch_decode_warps<T, kG, kDecWarps2>(a, q, K, V, st) : launch_decode_warps<T, kG, kDecWarps>(a, q, K, V, st);
}
}

graphkv_status graphkv_decode_attention(const graphkv_params *params, const void *q, const void *K,
                                        const void *V, float *out, void *workspace,
                                        size_t workspace_bytes, void *stream)
{
    DecodeArgs a;
    if (!decode_shape(params, &a)) return params && params->head_dim != kHeadDim ? GRAPHKV_ERR_UNSUPPORTED
                                                                                  : GRAPHKV_ERR_INVALID_ARG;
    if (!q || !K || !V || !out || !aligned16(K) || !aligned16(V)) return GRAPHKV_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < decode_bytes(a)) return GRAPHKV_ERR_WORKSPACE;
    void *ws = reinterpret_cast<void *>(align_up(reinterpret_cast<uintptr_t>(workspace)));
    a.arrived = static_cast<unsigned long long *>(ws);
    a.part = at<float>(ws, align_up((size_t)a.batch * a.hkv * sizeof(unsigned long long)));
    a.out = out;
    a.call_tag = next_call_tag();
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (params->dtype == GRAPHKV_BF16)
        return a.G <= 4 ? launch_decode<__nv_bfloat16, 4>(a, q, K, V, st) : launch_decode<__nv_bfloat16, 8>(a, q, K, V, st);
    return a.G <= 4 ? launch_decode<float, 4>(a, q, K, V, st) : launch_decode<float, 8>(a, q, K, V, st);
}

graphkv_status graphkv_read_status(const void *workspace, void *stream)
{
    if (!workspace) return GRAPHKV_ERR_WORKSPACE;
    int word = 0;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(&word, workspace, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return GRAPHKV_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return GRAPHKV_ERR_CUDA;
    if (word < 0 || word > GRAPHKV_ERR_TIMEOUT) return GRAPHKV_ERR_CUDA;
    return static_cast<graphkv_status>(word);
}

graphkv_status graphkv_read_neighbors(const graphkv_params *params, const void *workspace,
                                      size_t workspace_bytes, int32_t *nbr_idx_out,
                                      float *nbr_e_out, void *stream)
{
    Dims d;
    graphkv_status rc = resolve(params, &d);
    if (rc != GRAPHKV_OK) return rc;
    if (!graph_active(d)) return GRAPHKV_ERR_INVALID_ARG;
    const Layout l = layout_of(d);
    if ((rc = check_ws(l, workspace, workspace_bytes)) != GRAPHKV_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t pairs = (size_t)d.units * d.K_src * d.m;
    const unsigned char *ws = static_cast<const unsigned char *>(workspace);
    if (nbr_idx_out && cudaMemcpyAsync(nbr_idx_out, ws + l.nbr_idx, pairs * sizeof(int),
                                       cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return GRAPHKV_ERR_CUDA;
    if (nbr_e_out && cudaMemcpyAsync(nbr_e_out, ws + l.nbr_e, pairs * sizeof(float),
                                     cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return GRAPHKV_ERR_CUDA;
    return GRAPHKV_OK;
}

int64_t graphkv_launch_count(void) { return g_launches.load(); }

void graphkv_trace_enable(int32_t enable)
{
    g_trace_on.store(enable ? 1 : 0);
}

int32_t graphkv_trace_read(graphkv_trace_record *out, int32_t capacity)
{
    std::lock_guard<std::mutex> lk(g_trace_mu);
    int32_t n = 0;
    for (const TraceEntry &e : g_trace) {
        float ms = -1.f;
        if (cudaEventSynchronize(e.stop) == cudaSuccess) cudaEventElapsedTime(&ms, e.start, e.stop);
        if (out && n < capacity) {
            strncpy(out[n].name, e.name, sizeof(out[n].name) - 1);
            out[n].name[sizeof(out[n].name) - 1] = 0;
            out[n].ms = ms;
            ++n;
        }
        cudaEventDestroy(e.start);
        cudaEventDestroy(e.stop);
    }
    g_trace.clear();
    return n;
}

int32_t graphkv_phase_timing_read(uint64_t *out)
{
#ifdef GRAPHKV_PHASE_TIMING
    if (!out || cudaDeviceSynchronize() != cudaSuccess) return 0;
    constexpr size_t n = (size_t)kPhaseKernels * kPhaseSlots;
    std::vector<unsigned long long> sum(n), mx(n), cnt(kPhaseKernels);
    if (cudaMemcpyFromSymbol(sum.data(), g_phase_sum, n * 8) != cudaSuccess ||
        cudaMemcpyFromSymbol(mx.data(), g_phase_max, n * 8) != cudaSuccess ||
        cudaMemcpyFromSymbol(cnt.data(), g_phase_cnt, kPhaseKernels * 8) != cudaSuccess)
        return 0;
    for (size_t i = 0; i < n; ++i) {
        out[2 * i] = sum[i];
        out[2 * i + 1] = mx[i];
    }
    for (int k = 0; k < kPhaseKernels; ++k) out[2 * n + k] = cnt[k];
    std::fill(sum.begin(), sum.end(), 0ull);
    cudaMemcpyToSymbol(g_phase_sum, sum.data(), n * 8);
    cudaMemcpyToSymbol(g_phase_max, sum.data(), n * 8);
    cudaMemcpyToSymbol(g_phase_cnt, sum.data(), kPhaseKernels * 8);
    return 1;
#else
    (void)out;
    return 0;
#endif
}

const char *graphkv_status_string(graphkv_status status)
{
    switch (status) {
        case GRAPHKV_OK: return "ok";
        case GRAPHKV_ERR_INVALID_ARG: return "invalid argument";
        case GRAPHKV_ERR_UNSUPPORTED: return "unsupported configuration";
        case GRAPHKV_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case GRAPHKV_ERR_CUDA: return "CUDA error";
        case GRAPHKV_ERR_TIMEOUT: return "device-side wait timed out";
        case GRAPHKV_ERR_BUILTIN_SCRATCH:
            return "problem needs more scratch than the built-in array of graphkv_score_noalloc holds";
    }
    return "unknown status";
}

}  // extern "C"
