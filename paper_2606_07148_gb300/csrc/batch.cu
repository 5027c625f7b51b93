// Batched (alpha, beta)-cores: many pairs over one graph in one persistent launch, replayed as a
// CUDA graph.
//
// Nested property (Section 4.2, the basis of Lemma 1): if alpha' >= alpha and beta' >= beta then
// core(alpha', beta') lies inside core(alpha, beta); and for any vertex set S containing
// core(alpha, beta), peeling G[S] gives the same core as peeling G. Algorithm 2 (GCC+) uses this
// with core numbers; here it is applied along chains: pairs that share alpha are sorted by beta,
// and one chain peels (alpha, beta_0) and then raises the V bound step by step, each step
// starting from the previous step's core. A vertex is removed at most once per chain, so a
// chain costs at most one full peel, whatever its length. The step at which each vertex falls
// is recorded (lvl), and the masks of all the chain's pairs follow from it:
//     x in core(alpha, beta_j)  <=>  x is a step-0 candidate and lvl[x] > j.
//
// The chains run concurrently, each on its own group of blocks of one cooperative launch. Inside
// a group, steps are separated by a bounded group barrier; the cascade of each step reuses the
// single peel's work queue (peel_core.cuh). A second kernel writes every pair's masks in the
// caller's ids. Memsets, both launches and the status read-back are captured once per pair list
// as a CUDA graph and replayed.
#include <algorithm>
#include <cstring>
#include <map>
#include <vector>

#include "device.cuh"
#include "internal.h"
#include "peel_core.cuh"
#include "small_peel.cuh"

namespace {

using abc::LaneStats;
using abc::WarpSmem;

constexpr int BATCH_THREADS = 256;
constexpr int MAX_CHAINS_PER_WAVE = 32;
constexpr int MAX_STEPS = 255;
// timeline of one chain (log level 2): its start, then three marks per step
constexpr int PROF_STRIDE = 1 + 3 * MAX_STEPS;
__host__ __device__ constexpr int prof_at(int step, int phase) { return 1 + 3 * step + phase; }

struct ChainDev {
    int32_t alpha;
    int32_t nsteps;
    int32_t beta_off;        // betas[beta_off .. beta_off + nsteps): ascending V bounds
    int32_t pU0, pV0;        // step-0 candidate prefixes
    int32_t searchU, searchV;
    int32_t hubcutU, hubcutV;
    int32_t first_block, nblocks;
    int32_t col;             // column of this chain in lvl
    int32_t seed_col;        // column of a finished chain with a smaller alpha and the same betas
                             // (its step-j core contains this chain's), or -1
    int64_t sa, ea, sb, eb;  // step-0 violator slices (see stream_range)
};

struct ChainMem {
    int32_t *cnt;
    int32_t *plen;
    unsigned long long *q;
    PeelCtl *ctl;
    unsigned *bar;           // group barrier: [0] arrivals, [32] generation
    uint32_t *ulive;         // bitmap over the U prefix: candidates a step's U scan must look at
};

struct BatchArgs {
    const int64_t *off;
    const int32_t *adj;
    int32_t nU, nV;
    const ChainDev *chains;
    const ChainMem *mem;
    const int32_t *betas;
    const int32_t *pvs;      // per beta: the V candidate prefix (vertices of degree >= beta)
    const float *fracs;      // per beta: the share of a U row's step-0 candidate entries below it
                             // (where the search for a fallen U row's new end starts)
    int32_t nchains;
    uint8_t *lvl;
    int32_t lvl_stride;
    int32_t chunk;
    int32_t batch_entries, flush_steps;
    int32_t packed;          // 16-bit counts (every degree below 2^16)
    int32_t swz;             // counts in the swizzled layout (PeelArgs::swz)
    uint32_t *flags;
    long long qcap;
    unsigned long long timeout_ns;
    // optional timeline: prof[c * PROF_STRIDE + 0] = globaltimer when chain c's block 0 starts,
    // then per step j three marks (prof_at): after its V walk (step 0: the count init), after its
    // U scan (step 0: the first round), after its cascade
    // (j = 0) and when its step j - 1 has closed (j >= 1); nullptr: not recorded
    unsigned long long *prof;
};

// Compiled for two occupancies: three blocks an SM (80 registers a thread, some spilled) or two
// (no spills); "blocks_per_sm" = 2 picks the second.
template <int MINB>
__global__ void __launch_bounds__(BATCH_THREADS, MINB) k_batch(BatchArgs B) {
    __shared__ WarpSmem smem[BATCH_THREADS / 32];
    __shared__ unsigned s_hubs[abc::WALK_HUBS];  // the V walk's U-hub tallies (fall_walk_v)
    int c = 0;
    while (c + 1 < B.nchains && (int)blockIdx.x >= B.chains[c + 1].first_block) ++c;
    const ChainDev cd = B.chains[c];
    const ChainMem mem = B.mem[c];
    const int G = cd.nblocks;
    const int r = (int)blockIdx.x - cd.first_block;
    const int wib = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < abc::WALK_HUBS; i += blockDim.x) s_hubs[i] = 0u;
    // (init_range's first barrier orders these stores before any walk)

    PeelArgs a{};
    a.off = B.off;
    a.adj = B.adj;
    a.cnt = mem.cnt;
    a.packed = B.packed;
    set_count_layout(a, cd.pU0, cd.pV0, B.swz != 0);  // later steps' candidates are prefixes of these
    a.plen = mem.plen;
    a.q = mem.q;
    a.qcap = B.qcap;
    a.ctl = mem.ctl;
    a.nU = B.nU;
    a.nV = B.nV;
    a.pU = cd.pU0;
    a.pV = cd.pV0;
    a.thrU = cd.alpha;
    a.thrV = B.betas[cd.beta_off];
    a.chunk = B.chunk;
    a.batch_entries = B.batch_entries;
    a.flush_steps = B.flush_steps;
    a.searchU = cd.searchU;
    a.searchV = cd.searchV;
    a.hubcutU = cd.hubcutU;
    a.hubcutV = cd.hubcutV;
    a.timeout_ns = B.timeout_ns;
    a.skip_zero = 0;  // a V bound of 0 may rise later: keep every count exact
    a.lvl = B.lvl;
    a.lvl_stride = B.lvl_stride;
    a.lvl_col = cd.col;
    a.seed_col = cd.seed_col;
    a.dead_own = cd.seed_col >= 0 ? 1 : 0;
    a.step = 0;
    a.flags = B.flags;
    a.flag_first = cd.first_block;
    a.flag_count = G;
    a.epoch = 1;
    // Grabs of an even share for half a chain's warps. With an eighth of them, a short queue is handed out in grabs
    // that leave most warps without a row while a few walk eight each. An eighth -> half: 144 pairs over 10M edges
    // 3.76 -> 2.69 ms, 64 pairs over 1M 1.07 -> 0.96, 256 pairs over 100M 17.9 -> 17.2, over 250M 39.6 -> 39.2; 16
    // pairs over 40M are the same (1.77, 1.81), and so is a share for every warp (2.58, 0.97, 17.4, 39.6, 1.85).
    const int grab_div = max(1, G * (BATCH_THREADS / 32) / 2);

    const int64_t t0 = (int64_t)r * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)G * blockDim.x;
    LaneStats ls;
    unsigned long long probes = 0, inits = 0, ents = 0, sdecs = 0;

    unsigned long long *prof = B.prof != nullptr && r == 0 && threadIdx.x == 0 ? B.prof + (size_t)c * PROF_STRIDE
                                                                               : nullptr;
    if (prof) prof[0] = abc::now_ns();
    abc::init_range(a, smem[wib].push, t0, nthreads, ls, probes, inits);
    if (!abc::group_barrier(mem.bar, G, mem.ctl, false, B.timeout_ns)) goto out;
    if (prof) prof[prof_at(0, 0)] = abc::now_ns();
    if (cd.ea > cd.sa || cd.eb > cd.sb) {
        const unsigned long long d0 = ls.decs;
        abc::stream_range(a, cd.sa, cd.ea, cd.sb, cd.eb, t0, nthreads, ls, ents);
        sdecs = ls.decs - d0;
        ls.decs = d0;
        if (!abc::group_barrier(mem.bar, G, mem.ctl, false, B.timeout_ns)) goto out;
        unsigned long long scanned = 0;
        abc::scan_range(a, smem[wib].push, t0, nthreads, ls, scanned);
        if (!abc::group_barrier(mem.bar, G, mem.ctl, false, B.timeout_ns)) goto out;
    }
    if (prof) prof[prof_at(0, 1)] = abc::now_ns();
    // A failed cascade leaves its code in ctl->err. Every warp still reaches the barrier, so no
    // block waits on warps that left, and the barrier reports the error to all of them.
    (void)abc::cascade_loop<false>(a, smem[wib], ls, grab_div, r == 0 && wib == 0);
    if (!abc::group_barrier(mem.bar, G, mem.ctl, true, B.timeout_ns)) goto out;
    if (prof) prof[prof_at(0, 2)] = abc::now_ns();
    for (int j = 1; j < cd.nsteps; ++j) {
        const int32_t prev = a.thrV;
        const int32_t pv_prev = a.pV;
        a.thrV = B.betas[cd.beta_off + j];
        a.step = j;
        a.epoch = (uint32_t)j + 1;
        // the V candidates shrink to degree >= the new bound. The live V vertices of the previous
        // prefix that miss it (all those past the new prefix among them, their degree being below
        // it; with a seed chain, also those outside its step-j core) fall first, their rows walked
        // with decrements that return nothing; the U candidates those decrements took below alpha
        // are then queued; the cascade does the rest. A fallen U vertex walks only its entries
        // inside the new prefix (process_items).
        a.pV = B.pvs[cd.beta_off + j];
        a.pV_rows = cd.pV0;
        a.frac_rows = B.fracs[cd.beta_off + j];
        {
            unsigned long long e0 = 0, d0 = 0;
            abc::fall_walk_v(a, smem[wib], pv_prev, prev, a.dead_own != 0, t0, nthreads, ls, e0, d0, s_hubs);
            ents += e0;
            sdecs += d0;
        }
        if (!abc::group_barrier(mem.bar, G, mem.ctl, false, B.timeout_ns)) goto out;
        if (prof) prof[prof_at(j, 0)] = abc::now_ns();
        {
            unsigned long long sc = 0;
            abc::fall_scan_u(a, smem[wib], t0, nthreads, ls, sc, mem.ulive, j == 1);
        }
        if (!abc::group_barrier(mem.bar, G, mem.ctl, false, B.timeout_ns)) goto out;
        if (prof) prof[prof_at(j, 1)] = abc::now_ns();
        (void)abc::cascade_loop<false>(a, smem[wib], ls, grab_div, r == 0 && wib == 0);
        if (!abc::group_barrier(mem.bar, G, mem.ctl, true, B.timeout_ns)) goto out;
        if (prof) prof[prof_at(j, 2)] = abc::now_ns();
    }
out:
    abc::flush_stats(a, ls);
    {
        unsigned long long v[4] = {inits, probes, ents, sdecs};
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = (unsigned long long)abc::warp_sum64((long long)v[i]);
        if ((threadIdx.x & 31) == 0) {
            if (v[0]) atomicAdd(&a.ctl->st[ST_INIT], v[0]);
            if (v[1]) atomicAdd(&a.ctl->st[ST_PROBES], v[1]);
            if (v[2]) atomicAdd(&a.ctl->st[ST_STREAM], v[2]);
            if (v[3]) atomicAdd(&a.ctl->st[ST_SDECS], v[3]);
        }
        if (r == 0 && threadIdx.x == 0) atomicAdd(&a.ctl->st[ST_STEPS], (unsigned long long)cd.nsteps);
    }
}

// A batch of a small graph: one block per pair (small_peel.cuh). What each did goes to the host.
template <bool LONG>
__global__ void __launch_bounds__(abc::SMALL_THREADS, 1) k_batch_small(abc::SmallGraph G, const abc::SmallQuery *__restrict__ queries,
                                                                       uint8_t *masks_u, uint8_t *masks_v, abc::SmallStats *host) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ abc::SmallStats st;
    const int p = blockIdx.x;
    abc::small_peel<LONG>(G, queries[p], smem, masks_u + (size_t)p * G.nU, masks_v + (size_t)p * G.nV, &st);
    if (threadIdx.x == 0) host[p] = st;
}

// Pairs one launch of k_batch_emit writes at most (it holds them in shared memory; 16 chains have 4,080 distinct ones)
constexpr int EMIT_PAIRS = 4096;
static_assert(sizeof(int32_t) * (4 * MAX_CHAINS_PER_WAVE + 1 + 2 * EMIT_PAIRS) <= 48 * 1024, "a launch needs no larger limit");

struct PairRef {
    int32_t chain;  // index into the wave's chains
    int32_t step;
};

// Masks of every pair of a wave, in the caller's ids. With up to 16 chains (a row of lvl is WORDS 4-byte words), layers
// that are multiples of four and aligned masks (`vec`), a thread takes four consecutive ids: their numbers
// and removal steps come in 16-byte loads, and per pair one byte-wise comparison of the four steps gives
// the 4-byte store. The pairs of a chain lie together (first[c] .. first[c + 1]); whether an id is a candidate of a chain
// does not depend on the pair (a V vertex that leaves the prefix at a later step has that step recorded). Bound
// by the masks' writes: 256 pairs on 6M vertices 1.54 GB, 0.29 ms (1.33 in four waves of four chains that
// tested every id's prefix for every pair).
template <int WORDS>
__global__ void __launch_bounds__(256) k_batch_emit(const int32_t *__restrict__ old2new, int32_t nU, int32_t nV,
                                                    const uint8_t *__restrict__ lvl, int32_t lvl_stride,
                                                    const ChainDev *__restrict__ chains, int32_t nchains,
                                                    const PairRef *__restrict__ pairs, const int32_t *__restrict__ pidx,
                                                    int32_t npairs, uint8_t *const *__restrict__ out) {
    extern __shared__ int32_t sh[];
    // the masks' addresses are read here, not captured, so one plan serves whatever buffers a call brings
    uint8_t *__restrict__ const masks_u = out[0];
    uint8_t *__restrict__ const masks_v = out[1];
    int32_t *pU0 = sh, *pV0 = sh + nchains, *col = sh + 2 * nchains, *first = sh + 3 * nchains;  // (first: nchains + 1)
    int32_t *ps = first + nchains + 1, *pi = ps + npairs;
    for (int i = threadIdx.x; i < nchains; i += blockDim.x) {
        pU0[i] = chains[i].pU0;
        pV0[i] = chains[i].pV0;
        col[i] = chains[i].col;
    }
    for (int i = threadIdx.x; i < npairs; i += blockDim.x) {  // (sorted by chain)
        ps[i] = pairs[i].step;
        pi[i] = pidx[i];
        for (int c = (i ? pairs[i - 1].chain : -1) + 1; c <= pairs[i].chain; ++c) first[c] = i;
        if (i == npairs - 1)
            for (int c = pairs[i].chain + 1; c <= nchains; ++c) first[c] = npairs;
    }
    __syncthreads();
    const int64_t n = (int64_t)nU + nV;
    if (WORDS > 0 && (nU & 3) == 0 && (nV & 3) == 0 &&
        ((reinterpret_cast<uintptr_t>(masks_u) | reinterpret_cast<uintptr_t>(masks_v)) & 3) == 0) {
        const int4 *o4 = reinterpret_cast<const int4 *>(old2new);
        for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n / 4; q += (int64_t)gridDim.x * blockDim.x) {
            const int64_t i = 4 * q;
            const int4 xv = __ldg(&o4[q]);
            const int32_t xs[4] = {xv.x, xv.y, xv.z, xv.w};
            const bool upper = i < nU;  // nU is a multiple of four: the quad is in one layer
            uint8_t *const dst = upper ? masks_u + i : masks_v + (i - nU);
            const size_t stride = upper ? (size_t)nU : (size_t)nV;
            uint32_t row[4][WORDS > 0 ? WORDS : 1];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint8_t *r = lvl + (size_t)xs[j] * (4 * WORDS);
                if constexpr (WORDS == 4) {
                    const uint4 w = __ldg(reinterpret_cast<const uint4 *>(r));
                    row[j][0] = w.x;
                    row[j][1] = w.y;
                    row[j][2] = w.z;
                    row[j][3] = w.w;
                } else {
#pragma unroll
                    for (int w = 0; w < WORDS; ++w) row[j][w] = __ldg(reinterpret_cast<const uint32_t *>(r) + w);
                }
            }
#pragma unroll
            for (int w = 0; w < WORDS; ++w) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int c = 4 * w + k;  // (a wave's chains have columns 0, 1, ... in order)
                    if (c >= nchains) break;
                    const int p0 = first[c], p1 = first[c + 1];
                    if (p0 == p1) continue;
                    // the four ids' steps for this chain in one word, 0 for one that is no candidate (never above a step)
                    const int32_t lim = upper ? pU0[c] : nU + pV0[c];
                    uint32_t lv = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) lv |= xs[j] < lim ? ((row[j][w] >> (8 * k)) & 0xffu) << (8 * j) : 0u;
                    for (int p = p0; p < p1; ++p) {
                        const uint32_t in = __vcmpgtu4(lv, (uint32_t)ps[p] * 0x01010101u) & 0x01010101u;
                        __stcs(reinterpret_cast<uint32_t *>(dst + (size_t)pi[p] * stride), in);
                    }
                }
            }
        }
        return;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t x = __ldg(&old2new[i]);
        const bool upper = i < nU;
        const uint8_t *row = lvl + (size_t)x * lvl_stride;
        for (int c = 0; c < nchains; ++c) {
            const int l = (upper ? x < pU0[c] : x - nU < pV0[c]) ? (int)__ldg(&row[col[c]]) : 0;
            for (int p = first[c]; p < first[c + 1]; ++p) {
                const uint8_t v = l > ps[p] ? 1 : 0;
                if (upper) masks_u[(size_t)pi[p] * nU + i] = v;
                else masks_v[(size_t)pi[p] * nV + (i - nU)] = v;
            }
        }
    }
}

}  // namespace

// One wave: up to MAX_CHAINS_PER_WAVE chains sharing the device at once.
struct Wave {
    std::vector<ChainDev> chains;
    std::vector<PairRef> pairs;
    std::vector<int32_t> pidx;   // caller pair index of each PairRef
    ChainDev *d_chains = nullptr;
    PairRef *d_pairs = nullptr;
    int32_t *d_pidx = nullptr;
    int grid = 0;
};

struct BatchState {
    // key of the captured graph
    std::vector<int32_t> key_a, key_b;
    int64_t key_graph_n = -1, key_graph_m = -1;
    int key_chunk = 0;
    // plan
    std::vector<Wave> waves;
    std::vector<int32_t> betas, pvs;
    std::vector<float> fracs;
    int32_t *d_betas = nullptr;
    int32_t *d_pvs = nullptr;
    float *d_fracs = nullptr;
    bool lvl_global = false;            // every chain has its own lvl column (seeding; cleared once per call)
    int nmem = 0;                       // chain workspaces allocated
    std::vector<ChainMem> mem;
    ChainMem *d_mem = nullptr;
    uint8_t *lvl = nullptr;
    int lvl_stride = 0;
    uint32_t *flags = nullptr;          // [grid * 32] per-block queue-closed flags (epochs)
    PeelCtl *ctl_host = nullptr;        // pinned: [waves x MAX_CHAINS_PER_WAVE]
    uint8_t **d_out = nullptr;          // where the call's masks go: {masks_u, masks_v}
    uint8_t **h_out = nullptr;          // pinned: its upload
    // a small graph's batch: queries (device, and their pinned upload) and what each did (pinned)
    abc::SmallQuery *d_queries = nullptr, *h_queries = nullptr;
    abc::SmallStats *h_small = nullptr;
    int32_t small_cap = 0;
    long long qcap = 0;
    bool q_dirty = false;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    bool use_graph = true;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    unsigned long long *prof = nullptr;  // [waves x MAX_CHAINS_PER_WAVE x PROF_STRIDE] (log level 2)
};

static void destroy_plan(abcore_ctx *ctx, BatchState *b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
    for (auto &w : b->waves) {
        ctx->release(w.d_chains);
        ctx->release(w.d_pairs);
        ctx->release(w.d_pidx);
    }
    b->waves.clear();
    ctx->release(b->d_betas);
    ctx->release(b->d_pvs);
    ctx->release(b->d_fracs);
    ctx->release(b->prof);
    ctx->host_release(b->ctl_host);
    b->key_a.clear();
    b->key_b.clear();
    b->key_graph_n = -1;
}

void free_batch(abcore_ctx *ctx) {
    BatchState *b = ctx->batch;
    if (!b) return;
    cudaStreamSynchronize(ctx->stream);
    destroy_plan(ctx, b);
    for (auto &m : b->mem) {
        ctx->release(m.cnt);
        ctx->release(m.plen);
        ctx->release(m.q);
        ctx->release(m.ctl);
        ctx->release(m.bar);
        ctx->release(m.ulive);
    }
    ctx->release(b->d_mem);
    ctx->release(b->lvl);
    ctx->release(b->flags);
    ctx->release(b->d_out);
    ctx->host_release(b->h_out);
    ctx->release(b->d_queries);
    ctx->host_release(b->h_queries);
    ctx->host_release(b->h_small);
    if (b->ev0) cudaEventDestroy(b->ev0);
    if (b->ev1) cudaEventDestroy(b->ev1);
    delete b;
    ctx->batch = nullptr;
}

static void (*batch_kernel(abcore_ctx *ctx))(BatchArgs) {
    return ctx->prm.blocks_per_sm == 2 ? k_batch<2> : k_batch<3>;
}

static int batch_grid(abcore_ctx *ctx) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel(ctx), BATCH_THREADS, 0);
    if (ctx->prm.blocks_per_sm > 0) per_sm = std::min(per_sm, ctx->prm.blocks_per_sm);
    return std::max(per_sm, 1) * ctx->num_sms;
}

// The removal-step record, n rows of `stride` bytes.
static int ensure_lvl(abcore_ctx *ctx, BatchState *b, int stride) {
    if (b->lvl && b->lvl_stride == stride) return ABCORE_OK;
    ctx->release(b->lvl);
    b->lvl_stride = stride;
    return ctx->alloc(&b->lvl, (size_t)std::max<int64_t>(ctx->g.n(), 1) * stride, "batch levels");
}

// Counts of a wave's chains (see batch_wave_of)
constexpr int64_t BATCH_WAVE_BYTES = 240ll << 20;
constexpr int MAX_LVL_COLS = 64;  // chains with a column of their own in lvl (beyond: one per wave slot)

// Build the plan for a pair list: chains by alpha, waves, seeds, slices, device tables.
//
// Chains are sorted by alpha. Without seeding, each wave takes the next chains in that order and
// chains share lvl columns by their slot in the wave. With seeding (and at most MAX_LVL_COLS
// chains), every chain has its own column and the chains are dealt to waves round-robin (chain k
// runs in wave k mod W), so a chain's smaller-alpha neighbours mostly ran in earlier waves: with
// the same beta steps, the closest such chain's step-j core contains this chain's (the nested
// property in alpha), and its non-members are queued as known dead.
static int make_plan(abcore_ctx *ctx, BatchState *b, int32_t n, const int32_t *alphas, const int32_t *betas) {
    const Graph &g = ctx->g;
    std::map<int32_t, std::vector<int32_t>> by_alpha;
    for (int32_t i = 0; i < n; ++i)
        if (alphas[i] >= ctx->prm.batch_plain_below) by_alpha[alphas[i]].push_back(betas[i]);
    struct Chain {
        int32_t alpha;
        std::vector<int32_t> betas;
    };
    std::vector<Chain> chains;
    for (auto &kv : by_alpha) {
        std::vector<int32_t> bs = kv.second;
        std::sort(bs.begin(), bs.end());
        bs.erase(std::unique(bs.begin(), bs.end()), bs.end());
        for (size_t s = 0; s < bs.size(); s += MAX_STEPS)
            chains.push_back({kv.first, std::vector<int32_t>(bs.begin() + s, bs.begin() + std::min(bs.size(), s + MAX_STEPS))});
    }
    const int C = (int)chains.size();
    const int grid = batch_grid(ctx);
    int per_wave = std::max(1, std::min({MAX_CHAINS_PER_WAVE, grid, b->nmem}));
    if (batch_wave_of(ctx) > 0) per_wave = std::min(per_wave, batch_wave_of(ctx));
    const int NW = (C + per_wave - 1) / per_wave;
    const bool own_cols = ctx->prm.batch_seed && C <= MAX_LVL_COLS;
    b->lvl_global = own_cols;
    const int stride = ((own_cols ? C : per_wave) + 3) / 4 * 4;
    ABC_TRY(ensure_lvl(ctx, b, stride));
    b->betas.clear();
    b->pvs.clear();
    b->fracs.clear();
    b->waves.assign(NW, Wave{});
    std::vector<int> wave_of(C), slot_of(C), col_of(C);
    for (int k = 0; k < C; ++k) {
        wave_of[k] = own_cols ? k % NW : k / per_wave;
        slot_of[k] = own_cols ? k / NW : k % per_wave;
        col_of[k] = own_cols ? k : slot_of[k];
    }
    int seeded = 0;
    for (int k = 0; k < C; ++k) {
        const Chain &ch = chains[k];
        Wave &wave = b->waves[wave_of[k]];
        ChainDev d{};
        d.alpha = ch.alpha;
        d.nsteps = (int32_t)ch.betas.size();
        d.beta_off = (int32_t)b->betas.size();
        b->betas.insert(b->betas.end(), ch.betas.begin(), ch.betas.end());
        const int32_t beta0 = ch.betas[0];
        for (size_t j = 0; j < ch.betas.size(); ++j) {
            const int32_t bj = ch.betas[j];
            b->pvs.push_back((int32_t)cnt_ge(g.cntV_ge, bj));
            // where the search for a fallen U row's end inside the new prefix starts: the share of
            // the step-0 prefix's entries that lie below the new bound
            const double eb = (double)std::max<int64_t>(cnt_ge(g.edgesV_ge, ch.betas[0]), 1);
            b->fracs.push_back((float)((double)cnt_ge(g.edgesV_ge, bj) / eb));
        }
        d.pU0 = (int32_t)cnt_ge(g.cntU_ge, ch.alpha);
        d.pV0 = (int32_t)cnt_ge(g.cntV_ge, beta0);
        const int mode = pick_mode(ctx, ch.alpha, beta0, d.pU0, d.pV0);
        // U counts by row search: a U vertex's plen is then its row's end inside the step-0 V
        // prefix, where the search for its end inside a later step's prefix ends
        d.searchU = 1;
        d.searchV = (mode >> 1) & 1;
        d.hubcutU = 0;
        d.hubcutV = ctx->prm.hub_degree > 0 ? (int32_t)std::min<int64_t>(cnt_ge(g.cntV_ge, ctx->prm.hub_degree), d.pV0) : 0;
        if (!d.searchV && d.pV0 > 0) {
            d.sb = cnt_ge(g.edgesU_ge, ch.alpha);
            d.eb = g.m;
        }
        d.col = col_of[k];
        d.seed_col = -1;
        if (own_cols && ctx->prm.batch_seed) {
            for (int s2 = k - 1; s2 >= 0; --s2)
                if (wave_of[s2] < wave_of[k] && chains[s2].alpha < ch.alpha && chains[s2].betas == ch.betas) {
                    d.seed_col = col_of[s2];
                    seeded++;
                    break;
                }
        }
        wave.chains.push_back(d);
    }
    for (auto &wave : b->waves) {
        const int cw = (int)wave.chains.size();
        wave.grid = grid;
        int first = 0;
        for (int k = 0; k < cw; ++k) {
            ChainDev &d = wave.chains[k];
            d.nblocks = grid / cw + (k < grid % cw ? 1 : 0);
            d.first_block = first;
            first += d.nblocks;
        }
    }
    // pair -> (wave, chain in wave, step); pairs left to single peels have no chain
    for (int32_t i = 0; i < n; ++i) {
        if (alphas[i] < ctx->prm.batch_plain_below) continue;
        int ci = 0;
        for (; ci < C; ++ci) {
            if (chains[ci].alpha != alphas[i]) continue;
            const auto &bs = chains[ci].betas;
            if (std::binary_search(bs.begin(), bs.end(), betas[i])) break;
        }
        const auto &bs = chains[ci].betas;
        const int step = (int)(std::lower_bound(bs.begin(), bs.end(), betas[i]) - bs.begin());
        b->waves[wave_of[ci]].pairs.push_back({slot_of[ci], step});
        b->waves[wave_of[ci]].pidx.push_back(i);
    }
    for (auto &w : b->waves) {  // the pairs of a chain together (k_batch_emit)
        std::vector<size_t> order(w.pairs.size());
        for (size_t k = 0; k < order.size(); ++k) order[k] = k;
        std::stable_sort(order.begin(), order.end(), [&](size_t x, size_t y) { return w.pairs[x].chain < w.pairs[y].chain; });
        std::vector<PairRef> pr;
        std::vector<int32_t> pi;
        for (size_t k : order) {
            pr.push_back(w.pairs[k]);
            pi.push_back(w.pidx[k]);
        }
        w.pairs.swap(pr);
        w.pidx.swap(pi);
    }
    ABC_TRY(ctx->alloc(&b->d_betas, b->betas.size(), "batch betas"));
    ABC_CU(cudaMemcpy(b->d_betas, b->betas.data(), sizeof(int32_t) * b->betas.size(), cudaMemcpyHostToDevice));
    ABC_TRY(ctx->alloc(&b->d_pvs, b->pvs.size(), "batch prefixes"));
    ABC_CU(cudaMemcpy(b->d_pvs, b->pvs.data(), sizeof(int32_t) * b->pvs.size(), cudaMemcpyHostToDevice));
    ABC_TRY(ctx->alloc(&b->d_fracs, b->fracs.size(), "batch prefix shares"));
    ABC_CU(cudaMemcpy(b->d_fracs, b->fracs.data(), sizeof(float) * b->fracs.size(), cudaMemcpyHostToDevice));
    for (auto &w : b->waves) {
        ABC_TRY(ctx->alloc(&w.d_chains, w.chains.size(), "batch chains"));
        ABC_TRY(ctx->alloc(&w.d_pairs, std::max<size_t>(w.pairs.size(), 1), "batch pairs"));
        ABC_TRY(ctx->alloc(&w.d_pidx, std::max<size_t>(w.pidx.size(), 1), "batch pairs"));
        ABC_CU(cudaMemcpy(w.d_chains, w.chains.data(), sizeof(ChainDev) * w.chains.size(), cudaMemcpyHostToDevice));
        if (!w.pairs.empty()) {
            ABC_CU(cudaMemcpy(w.d_pairs, w.pairs.data(), sizeof(PairRef) * w.pairs.size(), cudaMemcpyHostToDevice));
            ABC_CU(cudaMemcpy(w.d_pidx, w.pidx.data(), sizeof(int32_t) * w.pidx.size(), cudaMemcpyHostToDevice));
        }
    }
    ABC_TRY(ctx->host_alloc(&b->ctl_host, MAX_CHAINS_PER_WAVE * b->waves.size(), "batch control readback"));
    if (ctx->prm.log_level >= 2)
        ABC_TRY(ctx->alloc(&b->prof, b->waves.size() * MAX_CHAINS_PER_WAVE * PROF_STRIDE, "batch timeline"));
    ctx->log(1, "batch plan: %d pairs, %d chains in %d waves of up to %d, grid %d blocks, %d seeded chains", n, C,
             (int)b->waves.size(), per_wave, grid, seeded);
    return ABCORE_OK;
}

// Counts of the batch's chains are 16-bit when every degree fits (parameter "packed_counts").
static bool batch_packed(const abcore_ctx *ctx) {
    return ctx->prm.packed_counts && std::max(ctx->g.maxdegU, ctx->g.maxdegV) <= 65535;
}

// Chains sharing the GPU at once, unless "batch_wave" says otherwise: more of them leave fewer blocks waiting in
// narrow steps, until their counts no longer find room in L2. 16 chains of 6M vertices (12 MB of counts each), 256
// pairs on 100M edges: waves of 2 / 4 / 8 / 16 34.9 / 25.0 / 21.1 / 19.6 ms; 0.6M vertices, 144 pairs on 10M edges: 9.9 / 6.4 /
// 5.5 / 4.2; 30M vertices (60 MB each, 500M edges): 4 was the best.
static int wave_by_size(const abcore_ctx *ctx) {
    const int64_t bytes = (batch_packed(ctx) ? 2 : 4) * ctx->g.n();
    int w = 16;
    while (w > 4 && w * bytes > BATCH_WAVE_BYTES) w /= 2;
    return w;
}
int batch_wave_of(const abcore_ctx *ctx) { return ctx->prm.batch_wave >= 0 ? ctx->prm.batch_wave : wave_by_size(ctx); }

// Chain workspaces: counts, queue, control block and barrier per concurrent chain, plus lvl.
static int ensure_memory(abcore_ctx *ctx, BatchState *b, int want_chains) {
    const Graph &g = ctx->g;
    const int64_t n = g.n();
    const int grid = batch_grid(ctx);
    const long long qcap = n + (2 * g.m) / std::max(ctx->prm.chunk, 1) + 1024 +
                           (long long)MAX_STEPS * 2 * grid * (BATCH_THREADS / 32) * 32 / std::max(want_chains, 1) + 4096;
    if (b->nmem >= want_chains && b->qcap >= qcap) return ABCORE_OK;
    for (auto &m : b->mem) {
        ctx->release(m.cnt);
        ctx->release(m.plen);
        ctx->release(m.q);
        ctx->release(m.ctl);
        ctx->release(m.bar);
        ctx->release(m.ulive);
    }
    b->mem.clear();
    ctx->release(b->d_mem);
    b->nmem = 0;
    size_t freeb = 0, totalb = 0;
    cudaMemGetInfo(&freeb, &totalb);
    const double per_chain = (batch_packed(ctx) ? 6.0 : 8.0) * n + 8.0 * qcap + 1.0 * n;  // counts + prefixes, queue, levels
    int fit = (int)std::max(1.0, 0.6 * (double)freeb / per_chain);
    const int chains = std::max(1, std::min(want_chains, fit));
    b->qcap = qcap;
    b->mem.resize(chains);
    for (int c = 0; c < chains; ++c) {
        ChainMem &m = b->mem[c];
        // counts in the swizzled layout need each layer's power-of-two range
        uint32_t mu = 0, mv = 0;
        int64_t bv = 0;
        const int64_t slots = std::max(n, swz_layout(g.nU, g.nV, &mu, &mv, &bv));
        // (32 slots of padding: the U scan reads whole 32-vertex words of counts)
        ABC_TRY(ctx->alloc(&m.cnt, (size_t)(batch_packed(ctx) ? slots / 2 + 17 : slots + 32), "batch counts"));
        ABC_TRY(ctx->alloc(&m.ulive, (size_t)(g.nU / 32 + 1), "batch live U bitmap"));
        ABC_TRY(ctx->alloc(&m.plen, (size_t)std::max<int64_t>(n, 1), "batch prefixes"));
        ABC_TRY(ctx->alloc(&m.q, (size_t)qcap, "batch queue"));
        ABC_TRY(ctx->alloc(&m.ctl, 1, "batch control"));
        ABC_TRY(ctx->alloc(&m.bar, 64, "batch barrier"));
        ABC_CU(cudaMemsetAsync(m.q, 0xff, sizeof(unsigned long long) * (size_t)qcap, ctx->stream));
        ABC_CU(cudaMemsetAsync(m.bar, 0, 64 * sizeof(unsigned), ctx->stream));
    }
    ABC_TRY(ctx->alloc(&b->d_mem, chains, "batch chain table"));
    ABC_CU(cudaMemcpy(b->d_mem, b->mem.data(), sizeof(ChainMem) * chains, cudaMemcpyHostToDevice));
    if (!b->flags) ABC_TRY(ctx->alloc(&b->flags, (size_t)grid * 32, "batch close flags"));
    b->nmem = chains;
    ABC_CU(cudaStreamSynchronize(ctx->stream));
    return ABCORE_OK;
}

// Enqueue the whole batch on the stream (captured into a graph on first use).
static int enqueue_batch(abcore_ctx *ctx, BatchState *b) {
    const Graph &g = ctx->g;
    const int64_t n = g.n();
    if (b->lvl_global) ABC_CU(cudaMemsetAsync(b->lvl, 0xff, (size_t)n * b->lvl_stride, ctx->stream));
    for (size_t wi = 0; wi < b->waves.size(); ++wi) {
        Wave &w = b->waves[wi];
        const int cw = (int)w.chains.size();
        for (int c = 0; c < cw; ++c) {
            ABC_CU(cudaMemsetAsync(b->mem[c].ctl, 0, sizeof(PeelCtl), ctx->stream));
            ABC_CU(cudaMemsetAsync(b->mem[c].bar, 0, 64 * sizeof(unsigned), ctx->stream));
        }
        if (!b->lvl_global) ABC_CU(cudaMemsetAsync(b->lvl, 0xff, (size_t)n * b->lvl_stride, ctx->stream));
        ABC_CU(cudaMemsetAsync(b->flags, 0, sizeof(uint32_t) * (size_t)w.grid * 32, ctx->stream));
        BatchArgs B{};
        B.off = g.off;
        B.adj = g.adj;
        B.nU = g.nU;
        B.nV = g.nV;
        B.chains = w.d_chains;
        B.mem = b->d_mem;
        B.betas = b->d_betas;
        B.pvs = b->d_pvs;
        B.fracs = b->d_fracs;
        B.nchains = cw;
        B.lvl = b->lvl;
        B.lvl_stride = b->lvl_stride;
        B.chunk = std::max(ctx->prm.chunk, 32);
        B.flags = b->flags;
        B.batch_entries = ctx->prm.batch_entries;
        B.packed = batch_packed(ctx) ? 1 : 0;
        // chains keep counts in vertex order: every step scans all of a chain's candidates in
        // order, which the swizzled layout would turn into random sector reads (measured slower)
        B.swz = 0;
        B.flush_steps = ctx->prm.flush_steps < 0 ? FLUSH_STEPS : ctx->prm.flush_steps;
        B.qcap = b->qcap;
        B.timeout_ns = (unsigned long long)ctx->prm.timeout_ms * 1000000ull;
        B.prof = b->prof ? b->prof + wi * MAX_CHAINS_PER_WAVE * PROF_STRIDE : nullptr;
        void *args[] = {&B};
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(w.grid);
        cfg.blockDim = dim3(BATCH_THREADS);
        cfg.stream = ctx->stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        ABC_CU(cudaLaunchKernelExC(&cfg, (const void *)batch_kernel(ctx), args));
        ctx->stats.launches++;
        for (size_t p0 = 0; p0 < w.pairs.size(); p0 += EMIT_PAIRS) {
            const int np = (int)std::min<size_t>(EMIT_PAIRS, w.pairs.size() - p0);
            const size_t shm = sizeof(int32_t) * (4 * cw + 1 + 2 * np);
            // a wave whose chains have the columns 0, 1, ... of rows of at most 16
            const int words = !b->lvl_global && b->lvl_stride <= 16 ? b->lvl_stride / 4 : 0;
            auto *emit = words == 1 ? k_batch_emit<1> : words == 2 ? k_batch_emit<2> : words == 3 ? k_batch_emit<3>
                       : words == 4 ? k_batch_emit<4> : k_batch_emit<0>;
            const int eg = (int)std::min<int64_t>((n + 255) / 256, (int64_t)ctx->num_sms * 8);
            emit<<<std::max(eg, 1), 256, shm, ctx->stream>>>(g.old2new, g.nU, g.nV, b->lvl, b->lvl_stride,
                                                                     w.d_chains, cw, w.d_pairs + p0, w.d_pidx + p0, np, b->d_out);
            ctx->stats.launches++;
        }
        for (int c = 0; c < cw; ++c)
            ABC_CU(cudaMemcpyAsync(b->ctl_host + wi * MAX_CHAINS_PER_WAVE + c, b->mem[c].ctl, sizeof(PeelCtl),
                                   cudaMemcpyDeviceToHost, ctx->stream));
    }
    return ABCORE_OK;
}

// Largest graph whose batch runs a block per pair: every pair's candidates fit a block, and peeling a pair by itself on one
// SM takes less than a chain's steps on their share of the GPU (three group barriers and a cascade's
// start and end each, about 25 us whatever their size). 8 x 8 pairs: 3,500 vertices and 20k edges 84 us against 957
// in chains; 15,010 and 200k 115 against 1,109; 35,000 and 800k 182 against 1,119; 21,000 and 1M 134 against 810.
constexpr int64_t SMALL_BATCH_EDGES = 1 << 20;
// ... and nothing is asked for that only chains have (a parameter of theirs, timed kernels, the timeline).
// Few pairs of very many rows to walk at once are left to the chains too: 4 pairs with 33,000 rows of 30 entries each
// 408 us a block per pair, 190 in chains.
constexpr double SMALL_BATCH_ROWS = 16384;
constexpr int32_t SMALL_BATCH_PAIRS = 32;
static bool small_batch(const abcore_ctx *ctx, int32_t n, const int32_t *alphas, const int32_t *betas) {
    const Params &p = ctx->prm, d;
    if (n < SMALL_BATCH_PAIRS && ctx->g.n() > SMALL_BATCH_ROWS)
        for (int32_t i = 0; i < n; ++i)
            if (first_round_rows(ctx->g, alphas[i], betas[i]) > SMALL_BATCH_ROWS) return false;
    return p.small_peel && ctx->g.n() <= abc::SMALL_MAX && ctx->g.m <= SMALL_BATCH_EDGES && p.timing == 0 && p.log_level < 2 &&
           !kernels_steered(p) && p.batch_plain_below == d.batch_plain_below && p.batch_seed == d.batch_seed &&
           p.packed_counts == d.packed_counts && (p.batch_wave < 0 || p.batch_wave == wave_by_size(ctx));
}

static int batch_small(abcore_ctx *ctx, BatchState *b, int32_t n, const int32_t *alphas, const int32_t *betas, uint8_t *d_masks_u,
                       uint8_t *d_masks_v) {
    const Graph &g = ctx->g;
    if (b->small_cap < n) {
        ctx->release(b->d_queries);
        ctx->host_release(b->h_queries);
        ctx->host_release(b->h_small);
        b->small_cap = 0;
        ABC_TRY(ctx->alloc(&b->d_queries, (size_t)n, "batch queries"));
        ABC_TRY(ctx->host_alloc(&b->h_queries, (size_t)n, "batch queries"));
        ABC_TRY(ctx->host_alloc(&b->h_small, (size_t)n, "batch statistics"));
        b->small_cap = n;
    }
    int64_t most = 0;
    for (int32_t i = 0; i < n; ++i) {
        const int32_t pU = (int32_t)cnt_ge(g.cntU_ge, alphas[i]), pV = (int32_t)cnt_ge(g.cntV_ge, betas[i]);
        b->h_queries[i] = {alphas[i], betas[i], pU, pV, 0, 0};
        most = std::max<int64_t>(most, (int64_t)pU + pV);
    }
    const size_t smem = abc::small_smem(most);
    // (the largest: the limit belongs to the function, which other contexts launch too)
    auto *k = std::max(g.maxdegU, g.maxdegV) > abc::SMALL_LONG ? k_batch_small<true> : k_batch_small<false>;
    ABC_CU(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)abc::small_smem(abc::SMALL_MAX)));
    ABC_CU(cudaMemcpyAsync(b->d_queries, b->h_queries, sizeof(abc::SmallQuery) * n, cudaMemcpyHostToDevice, ctx->stream));
    k<<<n, abc::SMALL_THREADS, smem, ctx->stream>>>({g.off, g.adj, g.old2new, g.nU, g.nV}, b->d_queries, d_masks_u, d_masks_v,
                                                                b->h_small);
    ABC_CU(cudaGetLastError());
    ABC_CU(cudaStreamSynchronize(ctx->stream));
    abcore_stats &s = ctx->stats;
    s.launches++;
    for (int32_t i = 0; i < n; ++i) {
        const abc::SmallStats &t = b->h_small[i];
        s.peels++;
        s.candidates += (int64_t)t.inits;
        s.init_vertices += (int64_t)t.inits;
        s.search_probes += (int64_t)t.probes;
        s.entries += (int64_t)t.entries;
        s.decrements += (int64_t)t.decs;
        s.pushes += (int64_t)t.pushes;
        s.items += (int64_t)t.pushes;
    }
    s.emit_gathered += (int64_t)n * g.n();
    return ABCORE_OK;
}

int batch_compute(abcore_ctx *ctx, int32_t n, const int32_t *alphas, const int32_t *betas, uint8_t *d_masks_u,
                  uint8_t *d_masks_v, bool sync_and_check) {
    const Graph &g = ctx->g;
    if (!ctx->batch) ctx->batch = new BatchState();
    BatchState *b = ctx->batch;
    if (small_batch(ctx, n, alphas, betas)) return batch_small(ctx, b, n, alphas, betas, d_masks_u, d_masks_v);
    if (!b->d_out) ABC_TRY(ctx->alloc(&b->d_out, 2, "batch mask addresses"));
    if (!b->h_out) ABC_TRY(ctx->host_alloc(&b->h_out, 2, "batch mask addresses"));
    const bool same = b->exec && b->key_graph_n == g.n() &&
                      b->key_graph_m == g.m && b->key_chunk == ctx->prm.chunk &&
                      b->key_a == std::vector<int32_t>(alphas, alphas + n) &&
                      b->key_b == std::vector<int32_t>(betas, betas + n);
    if (!same || !b->use_graph) {
        destroy_plan(ctx, b);
        std::map<int32_t, int> na;
        for (int32_t i = 0; i < n; ++i)
            if (alphas[i] >= ctx->prm.batch_plain_below) na[alphas[i]]++;
        int want = std::min<int>((int)na.size(), MAX_CHAINS_PER_WAVE);
        if (batch_wave_of(ctx) > 0) want = std::min(want, batch_wave_of(ctx));
        if (want > 0) {
            ABC_TRY(ensure_memory(ctx, b, want));
            ABC_TRY(make_plan(ctx, b, n, alphas, betas));
        } else {
            b->waves.clear();
        }
        b->key_a.assign(alphas, alphas + n);
        b->key_b.assign(betas, betas + n);
        b->key_graph_n = g.n();
        b->key_graph_m = g.m;
        b->key_chunk = ctx->prm.chunk;
        if (b->use_graph) {
            cudaStreamCaptureStatus cs;
            ABC_CU(cudaStreamIsCapturing(ctx->stream, &cs));
            if (cs == cudaStreamCaptureStatusNone &&
                cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
                const int64_t l0 = ctx->stats.launches;
                int rc = enqueue_batch(ctx, b);
                cudaGraph_t graph = nullptr;
                cudaError_t e = cudaStreamEndCapture(ctx->stream, &graph);
                ctx->stats.launches = l0;
                if (rc == ABCORE_OK && e == cudaSuccess &&
                    cudaGraphInstantiate(&b->exec, graph, 0) == cudaSuccess) {
                    b->graph = graph;
                } else {
                    if (graph) cudaGraphDestroy(graph);
                    cudaGetLastError();
                    b->exec = nullptr;
                    b->use_graph = false;  // capture refused: launch directly from now on
                }
            } else {
                cudaGetLastError();
                b->use_graph = false;
            }
        }
    }
    if (b->q_dirty) {
        for (auto &m : b->mem) ABC_CU(cudaMemsetAsync(m.q, 0xff, sizeof(unsigned long long) * (size_t)b->qcap, ctx->stream));
        b->q_dirty = false;
    }
    // (the previous call has ended: its upload is done)
    b->h_out[0] = d_masks_u;
    b->h_out[1] = d_masks_v;
    ABC_CU(cudaMemcpyAsync(b->d_out, b->h_out, 2 * sizeof(uint8_t *), cudaMemcpyHostToDevice, ctx->stream));
    const bool timed = ctx->prm.timing != 0;
    if (timed) {
        if (!b->ev0) ABC_CU(cudaEventCreate(&b->ev0));
        if (!b->ev1) ABC_CU(cudaEventCreate(&b->ev1));
        ABC_CU(cudaEventRecord(b->ev0, ctx->stream));
    }
    if (b->exec) {
        ABC_CU(cudaGraphLaunch(b->exec, ctx->stream));
        for (auto &w : b->waves) ctx->stats.launches += 1 + (int64_t)((w.pairs.size() + EMIT_PAIRS - 1) / EMIT_PAIRS);
    } else {
        ABC_TRY(enqueue_batch(ctx, b));
    }
    // pairs of small alpha are peeled one at a time by the single peel, always the plain one (the
    // batch stays index-free): there a chain would walk far more rows than the separate peels,
    // whose degree prefixes leave most of them out
    int plain_rc = ABCORE_OK;
    bool plain_any = false;
    for (int32_t i = 0; i < n && !plain_rc; ++i) {
        if (alphas[i] >= ctx->prm.batch_plain_below) continue;
        plain_any = true;
        plain_rc = peel_compute(ctx, alphas[i], betas[i], d_masks_u + (size_t)i * g.nU, d_masks_v + (size_t)i * g.nV,
                                false, false);
    }
    if (timed) ABC_CU(cudaEventRecord(b->ev1, ctx->stream));
    ABC_CU(cudaGetLastError());
    (void)sync_and_check;
    ABC_CU(cudaStreamSynchronize(ctx->stream));
    if (plain_any) {
        const int frc = peel_finish(ctx);
        if (!plain_rc) plain_rc = frc;
    }
    if (plain_rc) return plain_rc;
    int first_err = 0;
    abcore_stats &s = ctx->stats;
    for (size_t wi = 0; wi < b->waves.size(); ++wi)
        for (size_t c = 0; c < b->waves[wi].chains.size(); ++c) {
            const PeelCtl &pc = b->ctl_host[wi * MAX_CHAINS_PER_WAVE + c];
            if (pc.err && !first_err) first_err = pc.err;
            s.peels += (int64_t)pc.st[ST_STEPS];
            s.candidates += b->waves[wi].chains[c].pU0 + b->waves[wi].chains[c].pV0;
            s.init_vertices += (int64_t)pc.st[ST_INIT];
            s.search_probes += (int64_t)pc.st[ST_PROBES];
            s.stream_entries += (int64_t)pc.st[ST_STREAM];
            s.entries += (int64_t)pc.st[ST_ENTRIES];
            s.decrements += (int64_t)pc.st[ST_DECS] + (int64_t)pc.st[ST_SDECS];
            s.stream_decrements += (int64_t)pc.st[ST_SDECS];
            s.pushes += (int64_t)pc.st[ST_PUSHES];
            s.items += (int64_t)pc.st[ST_ITEMS];
        }
    for (auto &w : b->waves) s.emit_gathered += (int64_t)w.pairs.size() * g.n();
    if (b->prof && ctx->prm.log_level >= 2) {
        // per chain: the wave, alpha, and each step's duration in microseconds (step 0 includes
        // the count init and the first round)
        std::vector<unsigned long long> h(b->waves.size() * MAX_CHAINS_PER_WAVE * PROF_STRIDE);
        if (cudaMemcpy(h.data(), b->prof, sizeof(unsigned long long) * h.size(), cudaMemcpyDeviceToHost) == cudaSuccess) {
            for (size_t wi = 0; wi < b->waves.size(); ++wi)
                for (size_t c = 0; c < b->waves[wi].chains.size(); ++c) {
                    const ChainDev &cd = b->waves[wi].chains[c];
                    const unsigned long long *t = h.data() + (wi * MAX_CHAINS_PER_WAVE + c) * PROF_STRIDE;
                    std::string line;
                    char tmp[64];
                    unsigned long long prev = t[0];
                    for (int j = 0; j < cd.nsteps; ++j) {
                        const unsigned long long a0 = t[prof_at(j, 0)], a1 = t[prof_at(j, 1)], a2 = t[prof_at(j, 2)];
                        snprintf(tmp, sizeof(tmp), " %.0f/%.0f/%.0f", (double)(a0 - prev) / 1e3, (double)(a1 - a0) / 1e3,
                                 (double)(a2 - a1) / 1e3);
                        line += tmp;
                        prev = a2;
                    }
                    ctx->log(2, "batch wave %zu chain alpha=%d blocks=%d total %.1f us; steps (walk/scan/cascade us):%s", wi,
                             cd.alpha, cd.nblocks, (double)(t[prof_at(cd.nsteps - 1, 2)] - t[0]) / 1e3, line.c_str());
                }
        }
    }
    if (timed) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, b->ev0, b->ev1) == cudaSuccess) {
            s.kernel_ms[ABCORE_K_BATCH] += ms;
            s.kernel_launches[ABCORE_K_BATCH]++;
        }
    }
    if (first_err) {
        b->q_dirty = true;
        if (first_err == ABCORE_ETIMEDOUT)
            return ctx->fail(ABCORE_ETIMEDOUT, "batch: a bounded device wait expired (limit %lld ms)",
                             (long long)ctx->prm.timeout_ms);
        return ctx->fail(first_err, "batch: device reported error %d", first_err);
    }
    return ABCORE_OK;
}
