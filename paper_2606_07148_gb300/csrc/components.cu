// Connected components of the bipartite graph: the labels GFQ computes in its preprocessing and
// maintains under updates to scope each re-peel to the updated edge's component (Section 5).
//
// Lock-free union-find (cc_core.cuh), in the sampled form of Sutton, Ben-Nun and Barak ("Optimizing
// parallel graph connectivity computation via subgraph sampling"): most edges of a graph with one
// big component join vertices that are already together, so few are looked at.
//  1. seed: every vertex is joined with its row's first edge. Rows are ascending in degree order, so
//     that is its highest-degree neighbour and the chains of such neighbours end at the hubs:
//     one edge a vertex leaves nearly every vertex in the hubs' tree.
//     A hub that is its best neighbour's best neighbour roots a tree of its own: such roots' rows
//     are walked until they are joined too, which brings their whole trees.
//  2. U rows whose vertex is not in the tree of `c`, the first (highest-degree) U vertex, are
//     walked in full. c is the smallest id that can be in its tree, so it is that tree's root from
//     the start and "in c's tree" is "root == c".
//  3. The edges not seen then belong to U rows that were in c's tree: a V vertex outside it that has
//     such a neighbour joins it (one such edge is enough).
// Rows are walked by a block (>= 1024 entries), a warp (>= 32) or a thread each: layers are
// numbered by non-increasing degree, so the classes are id ranges, all in one launch.
//
// Bound: one random 32-byte sector a row in the seed, and the latency of its tree walks. Looking at
// every edge instead was bound by its random parent reads. A final pass compresses every path and names each
// component by the smallest caller id in it (U vertex u is u, V vertex v is nU + v), so labels do
// not depend on the internal numbering or on the order in which the unions happened.
#include <algorithm>

#include "cc_core.cuh"
#include "device.cuh"
#include "internal.h"

namespace {

constexpr int CC_HUB = 1024;    // rows at least this long: one block each
constexpr int CC_MEDIUM = 32;   // rows at least this long: one warp each

__device__ __forceinline__ bool slot_deleted(const uint32_t *tomb, int64_t p) {
    return tomb != nullptr && ((__ldg(&tomb[p >> 5]) >> (p & 31)) & 1u);
}

// An edge counts if its slot is not deleted and, with a `keep` mask, both endpoints are kept.
__device__ __forceinline__ bool edge_kept(const uint32_t *tomb, const uint8_t *keep, int64_t p, int32_t x, int32_t y) {
    return !slot_deleted(tomb, p) && (keep == nullptr || (__ldg(&keep[x]) && __ldg(&keep[y])));
}

// The first kept edge among a row's first CC_SEED entries, as its other end, or -1. (A bound on the
// look keeps long runs of deleted entries from one thread; a vertex it leaves alone is walked later.)
constexpr int CC_SEED = 4;
__device__ __forceinline__ int32_t first_neighbour(const int64_t *off, const int32_t *adj, const uint32_t *tomb,
                                                   const uint8_t *keep, int32_t x) {
    if (keep != nullptr && !__ldg(&keep[x])) return -1;
    const int64_t s = __ldg(&off[x]), e = min(__ldg(&off[x + 1]), s + CC_SEED);
    for (int64_t p = s; p < e; ++p) {
        const int32_t y = __ldg(&adj[p]);
        if (!slot_deleted(tomb, p) && (keep == nullptr || __ldg(&keep[y]))) return y;
    }
    return -1;
}

// A new forest: U vertices are roots, and a V vertex starts under its first neighbour (a U
// vertex, so a smaller id), which needs no atomic.
__global__ void __launch_bounds__(256) k_cc_init(const int64_t *off, const int32_t *adj, const uint32_t *tomb, const uint8_t *keep,
                                                 int32_t *parent, int32_t nU, int64_t n) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        const int32_t f = x < nU ? -1 : first_neighbour(off, adj, tomb, keep, (int32_t)x);
        parent[x] = f >= 0 ? f : (int32_t)x;
    }
}

// Vertices [0, n) joined with their first neighbours. The first try reads the neighbour's parent
// through L1 and hooks below it without looking for its root: parents of the hubs are read by
// nearly every vertex, and all those reads meeting in one L2 line took 0.36 ms for 4M vertices
// (now 0.04). A parent that has moved on meanwhile is still in the same tree, and the
// atomicCAS makes sure that what is hooked was a root.
__global__ void __launch_bounds__(256) k_cc_seed(const int64_t *off, const int32_t *adj, const uint32_t *tomb, const uint8_t *keep,
                                                 int32_t *parent, int64_t n) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        const int32_t f = first_neighbour(off, adj, tomb, keep, (int32_t)x);
        if (f < 0) continue;
        const int32_t t = parent[f];
        if (t < x && atomicCAS(&parent[x], (int32_t)x, t) == x) continue;
        if (t != x) abc::cc_unite(parent, (int32_t)x, f);
    }
}

// Whether x is in the tree of c, the smallest id that can be in it. Never reads c's own word (every
// vertex of a big component would), reads through L1, and leaves x just below c. A parent that another thread has
// moved meanwhile is read old or new: both lead on in the same tree, so "yes" is always right, and a
// vertex that was in the tree when the launch began always gets it.
__device__ __forceinline__ bool cc_in(int32_t *parent, int32_t x, int32_t c) {
    if (x == c) return true;
    int32_t y = x, p = parent[x];
    const int32_t p0 = p;
    while (p != c) {
        if (p == y) return false;
        y = p;
        p = parent[y];
    }
    if (p0 != c) parent[x] = c;
    return true;
}

// The vertex whose tree the walks leave out: the first U vertex, with `keep` the first kept one
// (looked for among the first CC_LOOK; if none is there, U vertex 0, whose tree then holds nothing
// kept). The same in every block. Block-collective.
constexpr int CC_LOOK = 4096;
__device__ __forceinline__ int32_t big_tree(const uint8_t *keep, int32_t nU) {
    if (keep == nullptr) return 0;
    __shared__ int first_s;
    if (threadIdx.x == 0) first_s = CC_LOOK;
    __syncthreads();
    for (int b = 0; b < min(nU, CC_LOOK); b += blockDim.x) {
        const int x = b + threadIdx.x;
        if (x < min(nU, CC_LOOK) && keep[x]) atomicMin(&first_s, x);
        if (__syncthreads_or(first_s < CC_LOOK)) break;
    }
    const int32_t c = first_s;
    __syncthreads();
    return c < CC_LOOK ? c : 0;
}

// Row x, entries s + lane, s + lane + step, ...: step 2 for a U row, step 3 for a V row (see the header).
// With ROOTS (U rows), only a row whose vertex is a root, and only until it is in c's tree.
template <bool UPPER, bool ROOTS>
__device__ __forceinline__ void cc_row(const int64_t *off, const int32_t *adj, const uint32_t *tomb, const uint8_t *keep,
                                       int32_t *parent, int32_t c, int32_t x, int lane, int step) {
    if (keep != nullptr && !__ldg(&keep[x])) return;
    if (ROOTS ? x == c || __ldcg(&parent[x]) != x : cc_in(parent, x, c)) return;
    const int64_t s = __ldg(&off[x]), e = __ldg(&off[x + 1]);
    for (int64_t p = s + lane; p < e; p += step) {
        const int32_t y = __ldg(&adj[p]);
        if (!edge_kept(tomb, keep, p, x, y)) continue;
        if (UPPER) {
            abc::cc_unite(parent, x, y);
            if (ROOTS && abc::cc_find(parent, x) == c) return;
        } else if (cc_in(parent, y, c)) {
            abc::cc_unite(parent, x, c);
            return;
        }
    }
}

// Rows base + [0, h) by blocks [0, bh), base + [h, w) by the warps of blocks [bh, bh + bw), base + [w, nl) by
// the threads of the rest. Each thread decides alone whether its row is in c's tree: one that is
// left out because another thread has just joined it is a row in c's tree like any other.
template <bool UPPER, bool ROOTS>
__global__ void __launch_bounds__(256) k_cc_walk(const int64_t *off, const int32_t *adj, const uint32_t *tomb, const uint8_t *keep,
                                                 int32_t *parent, int32_t nU, int32_t base, int32_t h, int32_t w, int32_t nl, int bh, int bw,
                                                 bool whole) {
    const int32_t c = whole ? -1 : big_tree(keep, nU);  // (no vertex is in the tree of -1)
    const int b = (int)blockIdx.x;
    if (b < bh) {
        for (int64_t x = b; x < h; x += bh) cc_row<UPPER, ROOTS>(off, adj, tomb, keep, parent, c, (int32_t)(base + x), threadIdx.x, blockDim.x);
    } else if (b < bh + bw) {
        const int nw = blockDim.x >> 5;
        for (int64_t x = h + (int64_t)(b - bh) * nw + (threadIdx.x >> 5); x < w; x += (int64_t)bw * nw)
            cc_row<UPPER, ROOTS>(off, adj, tomb, keep, parent, c, (int32_t)(base + x), threadIdx.x & 31, 32);
    } else {
        for (int64_t x = w + (int64_t)(b - bh - bw) * blockDim.x + threadIdx.x; x < nl; x += (int64_t)(gridDim.x - bh - bw) * blockDim.x)
            cc_row<UPPER, ROOTS>(off, adj, tomb, keep, parent, c, (int32_t)(base + x), 0, 1);
    }
}

// Compress every path (parent[x] = root) and record, per root, the smallest caller id. A big
// component's root would draw an atomic from every vertex, one after another (6M vertices in one
// component: 3.7 ms). Vertices under root 0, the first U vertex's, only lower a register, one
// atomic a block; of the others, the lanes that share a root with the first of them send one, and an id
// that does not lower what is already there sends none.
__global__ void __launch_bounds__(256) k_cc_roots(int32_t *parent, const int32_t *new2old, int32_t nU, int64_t n, int32_t *minc,
                                                  unsigned long long *ncomp) {
    __shared__ int32_t least_s;
    if (threadIdx.x == 0) least_s = INT32_MAX;
    __syncthreads();
    unsigned long long roots = 0;
    int32_t least0 = INT32_MAX;
    const int lane = threadIdx.x & 31;
    for (int64_t x0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x0 - lane < n; x0 += (int64_t)gridDim.x * blockDim.x) {
        const bool in = x0 < n;
        const int32_t x = (int32_t)(in ? x0 : n - 1);
        int32_t caller = __ldg(&new2old[x]) + (x >= nU ? nU : 0);
        const int32_t r = cc_in(parent, x, 0) ? 0 : abc::cc_find(parent, x);
        if (r == 0) {
            least0 = min(least0, caller);
        } else if (in) {
            parent[x] = r;
            roots += r == x ? 1 : 0;
        }
        const unsigned rest = __ballot_sync(ABC_FULL, r != 0);
        if (rest == 0) continue;
        const int first = __ffs(rest) - 1;
        const bool same = r == __shfl_sync(ABC_FULL, r, first);
        const int32_t least = __reduce_min_sync(ABC_FULL, same ? caller : INT32_MAX);
        if (same) caller = least;
        if (r != 0 && (!same || lane == first) && caller < __ldcg(&minc[r])) atomicMin(&minc[r], caller);
    }
    least0 = __reduce_min_sync(ABC_FULL, least0);
    if (lane == 0) atomicMin(&least_s, least0);
    __syncthreads();
    if (threadIdx.x == 0 && least_s != INT32_MAX) atomicMin(&minc[0], least_s);
    if (blockIdx.x == 0 && threadIdx.x == 0) roots++;  // root 0
    const unsigned long long v[1] = {roots};
    unsigned long long *const d[1] = {ncomp};
    abc::block_add<1>(v, d);
}

// Labels in the caller's order.
__global__ void k_cc_emit(const int32_t *old2new, const int32_t *parent, const int32_t *minc, int32_t nU, int32_t nV,
                          int32_t *lab_u, int32_t *lab_v) {
    const int64_t n = (int64_t)nU + nV;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t l = __ldg(&minc[__ldg(&parent[__ldg(&old2new[i])])]);
        if (i < nU) lab_u[i] = l;
        else lab_v[i - nU] = l;
    }
}

// Community of vertex q: members of the core (alive[x]) in q's component of the core.
__global__ void k_community(const int32_t *old2new, const int32_t *parent, const uint8_t *alive, int32_t q_internal,
                            int32_t nU, int32_t nV, uint8_t *mask_u, uint8_t *mask_v, unsigned long long *size) {
    const int64_t n = (int64_t)nU + nV;
    const int32_t rq = abc::cc_find(const_cast<int32_t *>(parent), q_internal);
    const bool qin = __ldg(&alive[q_internal]) != 0;
    unsigned long long c = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t x = __ldg(&old2new[i]);
        const uint8_t in = (qin && __ldg(&alive[x]) && abc::cc_find(const_cast<int32_t *>(parent), x) == rq) ? 1 : 0;
        if (i < nU) mask_u[i] = in;
        else mask_v[i - nU] = in;
        c += in;
    }
    const unsigned long long v[1] = {c};
    unsigned long long *const d[1] = {size};
    abc::block_add<1>(v, d);
}

}  // namespace

// Sparse graphs, of up to this many edges and two a vertex, unite all of them in one launch: there is little to leave out,
// and the seed and the other walks are four launches. Labels, in walks / in one: 1,000 components of four edges 78 / 56 us, 30,000
// 83 / 64, a path of 20,000 vertices 124 / 83, a 100 x 100 grid 136 / 94; but 3.3 edges a vertex, 20,000 edges 71 / 84.
constexpr int64_t CC_WHOLE = 1 << 17;

// The seed over vertices [0, nseed), then both walks.
static int cc_unions(abcore_ctx *ctx, int32_t *parent, const uint32_t *tomb, cudaStream_t st, const uint8_t *keep,
                     int64_t nseed) {
    const Graph &g = ctx->g;
    const int64_t cap = (int64_t)ctx->num_sms * 8;
    const bool whole = g.m <= CC_WHOLE && g.m <= 2 * (cnt_ge(g.cntU_ge, 1) + cnt_ge(g.cntV_ge, 1));
    if (nseed > 0 && !whole) {
        k_cc_seed<<<(unsigned)std::min<int64_t>((nseed + 255) / 256, 2 * cap), 256, 0, st>>>(g.off, g.adj, tomb, keep, parent, nseed);
        ctx->stats.launches++;
    }
    for (int pass = 0; pass < 3; ++pass) {  // U rows of roots, U rows, V rows
        if (whole && pass != 1) continue;
        const int layer = pass == 2 ? 1 : 0;
        const int32_t nl = layer == 0 ? g.nU : g.nV;
        const std::vector<int64_t> &cnt = layer == 0 ? g.cntU_ge : g.cntV_ge;
        const int32_t h = (int32_t)std::min<int64_t>(cnt_ge(cnt, CC_HUB), nl);
        const int32_t w = (int32_t)std::min<int64_t>(cnt_ge(cnt, CC_MEDIUM), nl);
        const int32_t nz = (int32_t)std::min<int64_t>(cnt_ge(cnt, 1), nl);  // (isolated vertices have no row)
        const int64_t bh = std::min<int64_t>(h, cap), bw = std::min<int64_t>(((int64_t)(w - h) + 7) / 8, cap);
        const int64_t bt = std::min<int64_t>(((int64_t)(nz - w) + 255) / 256, cap);
        if (bh + bw + bt == 0) continue;
        auto *k = pass == 0 ? k_cc_walk<true, true> : pass == 1 ? k_cc_walk<true, false> : k_cc_walk<false, false>;
        k<<<(unsigned)(bh + bw + bt), 256, 0, st>>>(g.off, g.adj, tomb, keep, parent, g.nU, layer == 0 ? 0 : g.nU, h, w, nz,
                                                    (int)bh, (int)bw, whole);
        ctx->stats.launches++;
    }
    ABC_CU(cudaGetLastError());
    return ABCORE_OK;
}

int community_compute(abcore_ctx *ctx, const uint8_t *d_alive, int32_t q_internal, uint8_t *d_mask_u,
                      uint8_t *d_mask_v, int64_t *size) {
    const Graph &g = ctx->g;
    const int64_t n = g.n();
    int32_t *parent = nullptr;
    unsigned long long *cnt = nullptr;
    ABC_TRY(ctx->alloc(&parent, (size_t)std::max<int64_t>(n, 1), "community forest"));
    int rc = ctx->alloc(&cnt, 1, "community size");
    if (!rc) rc = cc_hook_base(ctx, parent, nullptr, ctx->stream, d_alive);
    unsigned long long h = 0;
    if (!rc) {
        const unsigned gi = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)ctx->num_sms * 16));
        cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), ctx->stream);
        k_community<<<gi, 256, 0, ctx->stream>>>(g.old2new, parent, d_alive, q_internal, g.nU, g.nV, d_mask_u, d_mask_v, cnt);
        ctx->stats.launches++;
        cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream);
        const cudaError_t e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) rc = ctx->cuda_fail(e, "community");
    }
    ctx->release(parent);
    ctx->release(cnt);
    if (!rc && size) *size = (int64_t)h;
    return rc;
}

// 80M edges, 6M vertices: init 36 us, seed 42, roots' rows 29, U rows 31, V rows 40 (then 25 for the roots'
// names and 18 for the labels), where uniting every edge took 1,770 and the names 3,700. Each of
// these reads the 48 MB of offsets or the 24 MB of parents once, and the first two one random
// 32-byte sector a row (190 MB).
int cc_hook_base(abcore_ctx *ctx, int32_t *parent, const uint32_t *tomb, cudaStream_t st, const uint8_t *keep) {
    const Graph &g = ctx->g;
    const int64_t n = g.n();
    const unsigned gi = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)ctx->num_sms * 16));
    k_cc_init<<<gi, 256, 0, st>>>(g.off, g.adj, tomb, keep, parent, g.nU, n);
    ctx->stats.launches++;
    return cc_unions(ctx, parent, tomb, st, keep, g.nU);
}

int cc_hook_rows(abcore_ctx *ctx, int32_t *parent, const uint32_t *tomb, cudaStream_t st, const uint8_t *keep) {
    return cc_unions(ctx, parent, tomb, st, keep, ctx->g.n());
}

int cc_emit(abcore_ctx *ctx, int32_t *parent, int32_t *d_lab_u, int32_t *d_lab_v, int64_t *ncomp, cudaStream_t st) {
    const Graph &g = ctx->g;
    const int64_t n = g.n();
    int32_t *minc = nullptr;
    unsigned long long *cnt = nullptr;
    ABC_TRY(ctx->alloc(&minc, (size_t)std::max<int64_t>(n, 1), "component labels"));
    int rc = ctx->alloc(&cnt, 1, "component count");
    unsigned long long h = 0;
    if (!rc) {
        const unsigned gi = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)ctx->num_sms * 16));
        cudaMemsetAsync(minc, 0x7f, sizeof(int32_t) * (size_t)std::max<int64_t>(n, 1), st);
        cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), st);
        k_cc_roots<<<gi, 256, 0, st>>>(parent, g.new2old, g.nU, n, minc, cnt);
        if (n > 0) k_cc_emit<<<gi, 256, 0, st>>>(g.old2new, parent, minc, g.nU, g.nV, d_lab_u, d_lab_v);
        ctx->stats.launches += 2;
        cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, st);
        const cudaError_t e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = ctx->cuda_fail(e, "components");
    }
    ctx->release(minc);
    ctx->release(cnt);
    if (!rc && ncomp) *ncomp = (int64_t)h;
    return rc;
}

int components_compute(abcore_ctx *ctx, int32_t *d_lab_u, int32_t *d_lab_v, int64_t *ncomp) {
    int32_t *parent = nullptr;
    ABC_TRY(ctx->alloc(&parent, (size_t)std::max<int64_t>(ctx->g.n(), 1), "component forest"));
    int rc = cc_hook_base(ctx, parent, nullptr, ctx->stream);
    if (!rc) rc = cc_emit(ctx, parent, d_lab_u, d_lab_v, ncomp, ctx->stream);
    ctx->release(parent);
    return rc;
}
