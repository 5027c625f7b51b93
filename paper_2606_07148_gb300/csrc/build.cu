// Device CSR builder for both layers (Section 3: CSR storage; Section 4.1: flat continuous ids).
//
// From m distinct edges (u, v) it builds, entirely on the GPU:
//   * a renumbering of each layer by non-increasing degree (ties by caller id), so that for any
//     threshold t the vertices of a layer with degree >= t form a prefix of its id range;
//   * unified internal ids: U vertex i is i, V vertex j is nU + j;
//   * off[n+1] (int64) and adj[2m] (int32, unified ids): rows 0..nU-1 list V neighbours, rows
//     nU..n-1 list U neighbours, every row ascending (so also by non-increasing degree);
//   * new2old / old2new permutations, and host tables of vertex and edge counts per threshold.
// Vertices are ordered by a stable least-significant-digit radix sort over 64-bit keys written for this
// library: 8-bit digits, a fixed grid whose blocks own contiguous key ranges, per-block digit
// histograms, one scan per digit, and a scatter whose in-warp ranks come from match.any. Edges are
// split into row ranges that fit a block's shared memory and sorted there ("edges into rows" below).
#include <algorithm>
#include <cstring>

#include "device.cuh"
#include "internal.h"

namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_IPT = 16;
constexpr int RS_TILE = RS_THREADS * RS_IPT;
constexpr int RS_RADIX = 256;

__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const uint64_t *__restrict__ keys, int64_t N,
                                                        int shift, int64_t tiles_per_block,
                                                        unsigned *__restrict__ hist, int G) {
    __shared__ unsigned h[RS_WARPS][RS_RADIX];
    const int w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < RS_WARPS * RS_RADIX; i += RS_THREADS) (&h[0][0])[i] = 0;
    __syncthreads();
    int64_t start = (int64_t)blockIdx.x * tiles_per_block * RS_TILE;
    int64_t end = min(start + tiles_per_block * RS_TILE, N);
    for (int64_t i = start + threadIdx.x; i < end; i += RS_THREADS) {
        unsigned d = (unsigned)(keys[i] >> shift) & 255u;
        atomicAdd(&h[w][d], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < RS_RADIX; d += RS_THREADS) {
        unsigned s = 0;
        for (int k = 0; k < RS_WARPS; ++k) s += h[k][d];
        hist[(int64_t)d * G + blockIdx.x] = s;
    }
}

// One block per digit: the digit's counts in the blocks before each block, and its total. (One block
// over all 256 G counts took 145 us a pass at full size, a fifth of the pass.)
__global__ void __launch_bounds__(RS_THREADS) k_rs_scan(const unsigned *__restrict__ hist, int G, unsigned *__restrict__ offs,
                                                        unsigned long long *__restrict__ total) {
    __shared__ unsigned wsum[RS_WARPS];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t row = (int64_t)blockIdx.x * G;
    unsigned run = 0;
    for (int b0 = 0; b0 < G; b0 += RS_THREADS) {
        const int b = b0 + threadIdx.x;
        const unsigned c = b < G ? hist[row + b] : 0u;
        const unsigned inc = (unsigned)abc::warp_incl_scan((int)c);
        if (lane == 31) wsum[w] = inc;
        __syncthreads();
        unsigned before = 0, all = 0;
#pragma unroll
        for (int q = 0; q < RS_WARPS; ++q) {
            before += q < w ? wsum[q] : 0u;
            all += wsum[q];
        }
        if (b < G) offs[row + b] = run + before + inc - c;
        run += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = run;
}

__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(const uint64_t *__restrict__ in,
                                                           uint64_t *__restrict__ out, int64_t N,
                                                           int shift, int64_t tiles_per_block,
                                                           const unsigned *__restrict__ offs,
                                                           const unsigned long long *__restrict__ total, int G) {
    __shared__ unsigned long long base[RS_RADIX];
    __shared__ unsigned long long dsum[RS_WARPS];
    __shared__ unsigned wcnt[RS_WARPS][RS_RADIX];
    __shared__ unsigned woff[RS_WARPS][RS_RADIX];
    __shared__ unsigned tcnt[RS_RADIX];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    {  // digit d's keys start after those of the digits below it
        const unsigned long long mine = total[threadIdx.x];
        unsigned long long inc = (unsigned long long)abc::warp_incl_scan64((long long)mine);
        if (lane == 31) dsum[w] = inc;
        __syncthreads();
        for (int q = 0; q < w; ++q) inc += dsum[q];
        base[threadIdx.x] = inc - mine + offs[(int64_t)threadIdx.x * G + blockIdx.x];
    }
    const int64_t t0 = (int64_t)blockIdx.x * tiles_per_block;
    const int64_t total_tiles = (N + RS_TILE - 1) / RS_TILE;
    const int64_t t1 = min(t0 + tiles_per_block, total_tiles);
    const unsigned lt = abc::lanemask_lt();
    for (int64_t tile = t0; tile < t1; ++tile) {
        for (int i = threadIdx.x; i < RS_WARPS * RS_RADIX; i += RS_THREADS) (&wcnt[0][0])[i] = 0;
        __syncthreads();
        const int64_t seg = tile * RS_TILE + (int64_t)w * 32 * RS_IPT;
        uint64_t k[RS_IPT];
        unsigned r[RS_IPT];
#pragma unroll
        for (int it = 0; it < RS_IPT; ++it) {
            const int64_t idx = seg + it * 32 + lane;
            const bool valid = idx < N;
            k[it] = valid ? in[idx] : 0ull;
        }
#pragma unroll
        for (int it = 0; it < RS_IPT; ++it) {
            const int64_t idx = seg + it * 32 + lane;
            const bool valid = idx < N;
            const unsigned act = __ballot_sync(ABC_FULL, valid);
            r[it] = 0;
            if (valid) {
                const unsigned d = (unsigned)(k[it] >> shift) & 255u;
                const unsigned peers = __match_any_sync(act, d);
                const unsigned before = __popc(peers & lt);
                const unsigned prev = wcnt[w][d];
                __syncwarp(act);
                if (before == 0) wcnt[w][d] = prev + __popc(peers);
                __syncwarp(act);
                r[it] = prev + before;
            }
        }
        __syncthreads();
        {
            const int d = threadIdx.x;
            unsigned s = 0;
#pragma unroll
            for (int q = 0; q < RS_WARPS; ++q) {
                woff[q][d] = s;
                s += wcnt[q][d];
            }
            tcnt[d] = s;
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < RS_IPT; ++it) {
            const int64_t idx = seg + it * 32 + lane;
            if (idx < N) {
                const unsigned d = (unsigned)(k[it] >> shift) & 255u;
                out[base[d] + woff[w][d] + r[it]] = k[it];
            }
        }
        __syncthreads();
        base[threadIdx.x] += tcnt[threadIdx.x];
        __syncthreads();
    }
}

// Sort N keys on bits [bit_lo, bit_hi); bits outside that range ride along. *result is a or b.
int radix_sort_u64(abcore_ctx *ctx, uint64_t *a, uint64_t *b, int64_t N, int bit_lo, int bit_hi,
                   uint64_t **result) {
    *result = a;
    if (N <= 1 || bit_hi <= bit_lo) return ABCORE_OK;
    const int64_t tiles = (N + RS_TILE - 1) / RS_TILE;
    int G = (int)std::min<int64_t>(tiles, (int64_t)ctx->num_sms * 4);
    const int64_t tpb = (tiles + G - 1) / G;
    G = (int)((tiles + tpb - 1) / tpb);
    unsigned *hist = nullptr, *offs = nullptr;
    unsigned long long *total = nullptr;
    int rc = ctx->alloc(&hist, (size_t)RS_RADIX * G, "radix histogram");
    if (!rc) rc = ctx->alloc(&offs, (size_t)RS_RADIX * G, "radix offsets");
    if (!rc) rc = ctx->alloc(&total, RS_RADIX, "radix totals");
    if (rc) {
        ctx->release(hist);
        ctx->release(offs);
        return rc;
    }
    uint64_t *src = a, *dst = b;
    for (int shift = bit_lo; shift < bit_hi; shift += 8) {
        k_rs_hist<<<G, RS_THREADS, 0, ctx->stream>>>(src, N, shift, tpb, hist, G);
        k_rs_scan<<<RS_RADIX, RS_THREADS, 0, ctx->stream>>>(hist, G, offs, total);
        k_rs_scatter<<<G, RS_THREADS, 0, ctx->stream>>>(src, dst, N, shift, tpb, offs, total, G);
        std::swap(src, dst);
    }
    cudaError_t e = cudaGetLastError();
    ctx->release(hist);
    ctx->release(offs);
    ctx->release(total);
    if (e != cudaSuccess) return ctx->cuda_fail(e, "radix sort launch");
    *result = src;
    return ABCORE_OK;
}

// ---- exclusive scan of int32 counts into int64 offsets (out[N] = total) -------------------
constexpr int SC_THREADS = 256, SC_IPT = 16, SC_TILE = SC_THREADS * SC_IPT;

__device__ long long block_excl_scan(long long v, long long *total) {
    __shared__ long long wsum[SC_THREADS / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    long long inc = abc::warp_incl_scan64(v);
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
        long long x = lane < SC_THREADS / 32 ? wsum[lane] : 0;
        long long xi = abc::warp_incl_scan64(x);
        if (lane < SC_THREADS / 32) wsum[lane] = xi - x;
        if (lane == SC_THREADS / 32 - 1) *total = xi;
    }
    __syncthreads();
    long long r = inc - v + wsum[w];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(SC_THREADS) k_scan_part(const int32_t *__restrict__ in, int64_t N,
                                                          long long *__restrict__ part) {
    __shared__ long long tot;
    const int64_t b = (int64_t)blockIdx.x * SC_TILE + (int64_t)threadIdx.x * SC_IPT;
    long long s = 0;
    for (int i = 0; i < SC_IPT; ++i)
        if (b + i < N) s += in[b + i];
    block_excl_scan(s, &tot);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) k_scan_top(long long *part, int64_t nb, int64_t *out_total) {
    __shared__ long long sh[1024];
    const int t = threadIdx.x;
    const int64_t per = (nb + 1023) / 1024;
    const int64_t b = t * per, e = min(b + per, nb);
    long long s = 0;
    for (int64_t i = b; i < e; ++i) s += part[i];
    sh[t] = s;
    __syncthreads();
    for (int d = 1; d < 1024; d <<= 1) {
        long long v = t >= d ? sh[t - d] : 0;
        __syncthreads();
        sh[t] += v;
        __syncthreads();
    }
    long long run = sh[t] - s;
    for (int64_t i = b; i < e; ++i) {
        long long x = part[i];
        part[i] = run;
        run += x;
    }
    if (t == 1023) *out_total = sh[1023];
}

__global__ void __launch_bounds__(SC_THREADS) k_scan_final(const int32_t *__restrict__ in, int64_t N,
                                                           const long long *__restrict__ part,
                                                           int64_t *__restrict__ out) {
    __shared__ long long tot;
    const int64_t b = (int64_t)blockIdx.x * SC_TILE + (int64_t)threadIdx.x * SC_IPT;
    int32_t v[SC_IPT];
    long long s = 0;
    for (int i = 0; i < SC_IPT; ++i) {
        v[i] = b + i < N ? in[b + i] : 0;
        s += v[i];
    }
    long long run = block_excl_scan(s, &tot) + part[blockIdx.x];
    for (int i = 0; i < SC_IPT; ++i)
        if (b + i < N) {
            out[b + i] = run;
            run += v[i];
        }
}

int exclusive_scan_i32(abcore_ctx *ctx, const int32_t *in, int64_t N, int64_t *out) {
    if (N == 0) {
        ABC_CU(cudaMemsetAsync(out, 0, sizeof(int64_t), ctx->stream));
        return ABCORE_OK;
    }
    const int64_t nb = (N + SC_TILE - 1) / SC_TILE;
    long long *part = nullptr;
    ABC_TRY(ctx->alloc(&part, (size_t)nb, "scan partials"));
    k_scan_part<<<(unsigned)nb, SC_THREADS, 0, ctx->stream>>>(in, N, part);
    k_scan_top<<<1, 1024, 0, ctx->stream>>>(part, nb, out + N);
    k_scan_final<<<(unsigned)nb, SC_THREADS, 0, ctx->stream>>>(in, N, part, out);
    cudaError_t e = cudaGetLastError();
    ctx->release(part);
    if (e != cudaSuccess) return ctx->cuda_fail(e, "scan launch");
    return ABCORE_OK;
}

// ---- builder kernels --------------------------------------------------------------------
__global__ void k_count_deg(const int32_t *__restrict__ eu, const int32_t *__restrict__ ev, int64_t m,
                            int32_t nU, int32_t nV, int32_t *__restrict__ degU,
                            int32_t *__restrict__ degV, int *err) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = eu[i], v = ev[i];
        if (u < 0 || u >= nU || v < 0 || v >= nV) {
            abc::set_error(err, ABCORE_EINVAL);
            continue;
        }
        atomicAdd(&degU[u], 1);
        atomicAdd(&degV[v], 1);
    }
}

// Largest degree of each layer, out[0] and out[1].
__global__ void __launch_bounds__(256) k_max(const int32_t *__restrict__ deg, int32_t nU, int64_t n, int *out) {
    __shared__ int s_max[2];
    if (threadIdx.x < 2) s_max[threadIdx.x] = 0;
    __syncthreads();
    int mu = 0, mv = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (i < nU) mu = max(mu, deg[i]);
        else mv = max(mv, deg[i]);
    }
    mu = __reduce_max_sync(ABC_FULL, mu);
    mv = __reduce_max_sync(ABC_FULL, mv);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&s_max[0], mu);
        atomicMax(&s_max[1], mv);
    }
    __syncthreads();
    if (threadIdx.x < 2 && s_max[threadIdx.x] > 0) atomicMax(&out[threadIdx.x], s_max[threadIdx.x]);
}

// Sort keys of all vertices by (layer, non-increasing degree): (layer << dbits | layer's maximum - degree) << 32 |
// unified caller id. Both layers go through one sort.
__global__ void k_relabel_keys(const int32_t *__restrict__ deg, int32_t nU, int64_t n, int32_t mdU, int32_t mdV, int dbits,
                               uint64_t *__restrict__ keys) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t hi = i < nU ? (uint32_t)(mdU - deg[i]) : ((uint32_t)1 << dbits) | (uint32_t)(mdV - deg[i]);
        keys[i] = ((uint64_t)hi << 32) | (uint64_t)i;
    }
}

__device__ __forceinline__ int32_t key_degree(uint64_t k, bool lower, int32_t mdU, int32_t mdV, int dbits) {
    const int32_t below = (int32_t)((uint32_t)(k >> 32) & (((uint32_t)1 << dbits) - 1u));
    return (lower ? mdV : mdU) - below;
}

__global__ void k_relabel_finish(const uint64_t *__restrict__ keys, int32_t nU, int64_t n, int32_t mdU, int32_t mdV, int dbits,
                                 int32_t *__restrict__ new2old, int32_t *__restrict__ old2new, int32_t *__restrict__ degnew) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = keys[p];
        const int32_t i = (int32_t)(k & 0xffffffffu);
        new2old[p] = i < nU ? i : i - nU;
        old2new[i] = (int32_t)p;
        degnew[p] = key_degree(k, i >= nU, mdU, mdV, dbits);
    }
}

// Row-major edge keys: (row rank << cbits) | column rank, both in internal per-layer ranks.
__global__ void k_edge_keys(const int32_t *__restrict__ eu, const int32_t *__restrict__ ev, int64_t m,
                            const int32_t *__restrict__ old2new, int32_t nU, int upper_rows,
                            int cbits, uint64_t *__restrict__ keys) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t ru = (uint64_t)old2new[eu[i]];
        const uint64_t rv = (uint64_t)(old2new[nU + ev[i]] - nU);
        keys[i] = upper_rows ? ((ru << cbits) | rv) : ((rv << cbits) | ru);
    }
}

__global__ void k_extract(const uint64_t *__restrict__ keys, int64_t m, uint64_t cmask, int32_t add,
                          int32_t *__restrict__ adj, int *err) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = keys[i];
        if (i > 0 && keys[i - 1] == k) abc::set_error(err, ABCORE_EEXIST);
        adj[i] = (int32_t)(k & cmask) + add;
    }
}

// Second ordering pass (build with a rank): position p of the degree order gets the key
// (layer << rbits | maxrank - rank) << 32 | p, so a stable sort orders each layer by non-increasing rank, ties by
// degree order.
__global__ void k_rank_keys(const uint64_t *__restrict__ by_degree, int32_t nU, int64_t n, const int32_t *__restrict__ rank,
                            int32_t maxrank, int rbits, uint64_t *__restrict__ keys) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t i = (int32_t)(by_degree[p] & 0xffffffffu);
        const uint32_t hi = (uint32_t)(maxrank - rank[i]) | (i < nU ? 0u : (uint32_t)1 << rbits);
        keys[p] = ((uint64_t)hi << 32) | (uint64_t)p;
    }
}

__global__ void k_rank_finish(const uint64_t *__restrict__ by_rank, const uint64_t *__restrict__ by_degree, int32_t nU, int64_t n,
                              int32_t mdU, int32_t mdV, int dbits, int32_t *__restrict__ new2old,
                              int32_t *__restrict__ old2new, int32_t *__restrict__ degnew) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = by_degree[by_rank[q] & 0xffffffffu];
        const int32_t i = (int32_t)(k & 0xffffffffu);
        new2old[q] = i < nU ? i : i - nU;
        old2new[i] = (int32_t)q;
        degnew[q] = key_degree(k, i >= nU, mdU, mdV, dbits);
    }
}

// Caller-id edges of a CSR's U rows: (new2old[row], new2old[column]).
__global__ void k_edges_of(const int32_t *__restrict__ rowid, const int32_t *__restrict__ adj, int64_t m,
                           const int32_t *__restrict__ new2old, int32_t *__restrict__ eu, int32_t *__restrict__ ev) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        eu[i] = new2old[rowid[i]];
        ev[i] = new2old[adj[i]];
    }
}

// cnt_ge[t] for t in [0, maxdeg + 1] of a layer whose rows are in non-increasing length (blockIdx.y: the layer).
struct DegTables {
    int64_t *cnt[2], *edges[2];
    int32_t md[2];
};
__global__ void k_cnt_ge(const int64_t *__restrict__ off, int32_t nU, int32_t nV, DegTables T) {
    const int l = blockIdx.y;
    const int64_t base = l ? nU : 0, nl = l ? nV : nU;
    int64_t *cnt_ge = T.cnt[l];
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nl;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t d = (int32_t)(off[base + p + 1] - off[base + p]);
        const int32_t dn = p + 1 < nl ? (int32_t)(off[base + p + 2] - off[base + p + 1]) : -1;
        for (int32_t t = dn + 1; t <= d; ++t) cnt_ge[t] = p + 1;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        cnt_ge[T.md[l] + 1] = 0;
        if (nl == 0) cnt_ge[0] = 0;
    }
}

__global__ void k_edges_ge(const int64_t *__restrict__ off, int32_t nU, DegTables T) {
    const int l = blockIdx.y;
    const int64_t base = l ? nU : 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t <= (int64_t)T.md[l] + 1;
         t += (int64_t)gridDim.x * blockDim.x)
        T.edges[l][t] = off[base + T.cnt[l][t]] - off[base];
}

// ---- edges into rows ------------------------------------------------------------------------
// Both layers' rows, each ascending, from the edge list. Every row's place is known from the degrees,
// so the edges only have to be brought near it and then ordered where they can be held on chip:
//   bins    the rows of a layer are cut into bins of about BIN_EDGES edges (row r is in bin off[r] / BIN_EDGES);
//   k_split every edge goes to the region of its row's bin, in both layers at once (with more than
//           SPLIT_BINS bins: of a group of bins, and k_regroup then moves it to its bin's region);
//   k_rows  one block a bin: counts the edges into their rows in shared memory, sorts each row and
//           writes its column ids.
// None of this keeps an order, so ranks inside a bin come from shared-memory atomics and a region's next
// free place from one global atomic per tile and bin. (Sorting (row, column) keys by 8-bit digits,
// one layer after the other, moved every edge twelve times for 22-bit ids: 17 ms for 80M edges with
// its histograms and scans.) 80M edges now: split 1.19 ms, bound by its 160M random reads of vertex
// records through L1 (one sector each); regroup 0.39 a layer, its shared-memory staging; rows
// 0.88 and 1.00 for the two layers, instruction issue (about 230 a 32 edges, 60 % of the issue slots).
constexpr int BIN_SHIFT = 12;
constexpr int64_t BIN_EDGES = 1 << BIN_SHIFT;
constexpr int SPLIT_BINS = 1024;       // bins k_split can tell apart (its shared counters)
constexpr int GROUPS = 256;            // groups of bins it splits into when there are more
constexpr int SPLIT_THREADS = 512, SPLIT_IPT = 8, SPLIT_TILE = SPLIT_THREADS * SPLIT_IPT;
constexpr int ROWS_CAP = 6144;         // edges of a bin k_rows holds with 256 threads (four blocks an SM) ...
constexpr int ROWS_CAP_MID = 13312;    // ... with 512 (two an SM), bins whose last row is long ...
constexpr int ROWS_CAP_BIG = 24576;    // ... and with 1024 (one an SM)
constexpr int WARP_ROW = 1024;         // rows up to this length are sorted by one warp in registers
constexpr int SHORT_ROW = 32;          // bins of rows up to this length are sorted by counting smaller entries

// Per layer: the bins' first edge positions and rows (bin b: edges [start[b], start[b + 1]) of the layer, rows
// [row[b], row[b + 1])), and the vertex records by caller id: {row, bin}. A key is the column in its low cbits,
// the row above it and the bin's number in its group above that.
struct LayerBins {
    int64_t *start;
    int32_t *row;
    unsigned long long *cur1, *cur2;  // next free place per group / per bin
    int32_t nb, shift;                // bins; bins per group = 1 << shift
    int32_t rbits, cbits;
    __device__ __forceinline__ int32_t key_row(uint64_t k) const { return (int32_t)((k >> cbits) & (((uint64_t)1 << rbits) - 1)); }
    __device__ __forceinline__ int32_t key_col(uint64_t k) const { return (int32_t)(k & (((uint64_t)1 << cbits) - 1)); }
};
struct Bins {
    LayerBins u, v;
    int2 *rec;                        // [n], U then V
};

__global__ void __launch_bounds__(256) k_bins(const int64_t *__restrict__ off, const int32_t *__restrict__ new2old, int32_t nU,
                                              int64_t n, int64_t m, Bins B) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        const int l = x >= nU;
        const LayerBins &L = l ? B.v : B.u;
        const int64_t vb = l ? nU : 0, eb = l ? m : 0;
        const int64_t o = off[x] - eb, o2 = off[x + 1] - eb;
        const int64_t b = o >> BIN_SHIFT;
        B.rec[vb + new2old[x]] = make_int2((int32_t)(x - vb), (int32_t)b);
        if (o2 == o) continue;  // (vertices without edges come last in either order)
        const int64_t bp = x > vb ? (off[x - 1] - eb) >> BIN_SHIFT : -1;
        for (int64_t t = bp + 1; t <= b; ++t) {
            L.start[t] = o;
            L.row[t] = (int32_t)(x - vb);
        }
        if (o2 == m)
            for (int64_t t = b + 1; t <= L.nb; ++t) {
                L.start[t] = m;
                L.row[t] = (int32_t)(x - vb) + 1;
            }
    }
}

__global__ void __launch_bounds__(256) k_cursors(Bins B) {
    const LayerBins &L = blockIdx.y ? B.v : B.u;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < L.nb; t += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long s = (unsigned long long)L.start[t];
        L.cur2[t] = s;
        if ((t & ((1 << L.shift) - 1)) == 0) L.cur1[t >> L.shift] = s;
    }
}

// Block-collective: each of nb counters cnt[b] becomes the sum of those before it, and place[b] the tile's
// reservation in bin b's region (next free place cur[b]) less that sum, so that the tile's i-th key in
// bin order goes to place[its bin] + i.
template <int THREADS>
__device__ __forceinline__ void tile_offsets(unsigned *cnt, unsigned long long *place, unsigned long long *cur, int nb) {
    __shared__ unsigned wsum[THREADS / 32];
    __shared__ unsigned carry_s;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry_s = 0;
    for (int b0 = 0; b0 < nb; b0 += THREADS) {
        const int b = b0 + threadIdx.x;
        const unsigned c = b < nb ? cnt[b] : 0u;
        unsigned long long g = 0;
        if (c) g = atomicAdd(&cur[b], (unsigned long long)c);
        const unsigned inc = (unsigned)abc::warp_incl_scan((int)c);
        if (lane == 31) wsum[w] = inc;
        __syncthreads();
        if (w == 0) {
            const unsigned x = lane < THREADS / 32 ? wsum[lane] : 0u;
            const unsigned xi = (unsigned)abc::warp_incl_scan((int)x);
            if (lane < THREADS / 32) wsum[lane] = xi - x + carry_s;
            __syncwarp();
            if (lane == THREADS / 32 - 1) carry_s += xi;
        }
        __syncthreads();
        if (b < nb) {
            const unsigned ex = inc - c + wsum[w];
            cnt[b] = ex;
            place[b] = g - ex;
        }
        __syncthreads();
    }
}

// Edges [tile] of the list to the regions of their rows' groups in both layers, as keys. A tile's edge remembers
// its rank among the tile's edges of its group (12 bits), the group (10) and its bin's number in the group (10).
__global__ void __launch_bounds__(SPLIT_THREADS, 2) k_split(const int32_t *__restrict__ eu, const int32_t *__restrict__ ev,
                                                            int64_t m, int32_t nU, Bins B, int ngroups, uint64_t *__restrict__ outU,
                                                            uint64_t *__restrict__ outV) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    uint64_t *stage = reinterpret_cast<uint64_t *>(sm_raw);
    unsigned long long *place = reinterpret_cast<unsigned long long *>(stage + SPLIT_TILE);
    unsigned *cnt = reinterpret_cast<unsigned *>(place + ngroups);  // [2][ngroups]
    unsigned short *sbin = reinterpret_cast<unsigned short *>(cnt + 2 * ngroups);
    const int t = threadIdx.x;
    const int64_t e0 = (int64_t)blockIdx.x * SPLIT_TILE;
    const int ne = (int)min((int64_t)SPLIT_TILE, m - e0);
    const int shift = B.u.shift;  // (the layers have as many edges: the same bins and groups)
    const unsigned in_group = (1u << shift) - 1u;
    for (int i = t; i < 2 * ngroups; i += SPLIT_THREADS) cnt[i] = 0;
    int32_t u[SPLIT_IPT], v[SPLIT_IPT];
    unsigned ru[SPLIT_IPT], rv[SPLIT_IPT];
#pragma unroll
    for (int k = 0; k < SPLIT_IPT; ++k) {
        const int i = k * SPLIT_THREADS + t;
        u[k] = i < ne ? __ldcs(&eu[e0 + i]) : 0;
        v[k] = i < ne ? __ldcs(&ev[e0 + i]) : 0;
    }
#pragma unroll
    for (int k = 0; k < SPLIT_IPT; ++k) {
        if (k * SPLIT_THREADS + t < ne) {
            const int2 a = __ldg(&B.rec[u[k]]), b = __ldg(&B.rec[(int64_t)nU + v[k]]);
            u[k] = a.x;
            v[k] = b.x;
            ru[k] = ((unsigned)a.y >> shift) << 12 | ((unsigned)a.y & in_group) << 22;
            rv[k] = ((unsigned)b.y >> shift) << 12 | ((unsigned)b.y & in_group) << 22;
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < SPLIT_IPT; ++k) {
        if (k * SPLIT_THREADS + t < ne) {
            ru[k] |= atomicAdd(&cnt[(ru[k] >> 12) & 1023u], 1u);
            rv[k] |= atomicAdd(&cnt[ngroups + ((rv[k] >> 12) & 1023u)], 1u);
        }
    }
    __syncthreads();
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        uint64_t *out = l ? outV : outU;
        if (out == nullptr) continue;
        const LayerBins &L = l ? B.v : B.u;
        tile_offsets<SPLIT_THREADS>(cnt + l * ngroups, place, L.cur1, ngroups);
#pragma unroll
        for (int k = 0; k < SPLIT_IPT; ++k) {
            if (k * SPLIT_THREADS + t < ne) {
                const unsigned r = l ? rv[k] : ru[k], g = (r >> 12) & 1023u;
                const unsigned p = cnt[l * ngroups + g] + (r & 4095u);
                stage[p] = ((uint64_t)(r >> 22) << L.rbits | (uint64_t)(uint32_t)(l ? v[k] : u[k])) << L.cbits |
                           (uint64_t)(uint32_t)(l ? u[k] : v[k]);
                sbin[p] = (unsigned short)g;
            }
        }
        __syncthreads();
        for (int i = t; i < ne; i += SPLIT_THREADS) out[place[sbin[i]] + (unsigned)i] = stage[i];
        __syncthreads();
    }
}

// Keys in their groups' regions to their bins' regions. A block takes one tile of one group.
__global__ void __launch_bounds__(SPLIT_THREADS, 3) k_regroup(const uint64_t *__restrict__ in, uint64_t *__restrict__ out, LayerBins L,
                                                              int ngroups) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int F = 1 << L.shift;
    uint64_t *stage = reinterpret_cast<uint64_t *>(sm_raw);
    unsigned long long *place = reinterpret_cast<unsigned long long *>(stage + SPLIT_TILE);
    unsigned *cnt = reinterpret_cast<unsigned *>(place + F);
    unsigned short *sbin = reinterpret_cast<unsigned short *>(cnt + F);
    __shared__ int64_t s_lo, s_hi;
    __shared__ int s_group;
    const int t = threadIdx.x;
    if (t < 32) {  // the group and place of this block's tile: groups hold ceil(edges / tile) tiles each
        int64_t left = blockIdx.x;
        if (t == 0) s_group = -1;
        __syncwarp();
        for (int g0 = 0; g0 < ngroups; g0 += 32) {
            const int g = g0 + t;
            int64_t a = 0, b = 0;
            if (g < ngroups) {
                a = L.start[(int64_t)g << L.shift];
                b = L.start[min((int64_t)(g + 1) << L.shift, (int64_t)L.nb)];
            }
            const long long nt = (b - a + SPLIT_TILE - 1) / SPLIT_TILE;
            const long long inc = abc::warp_incl_scan64(nt);
            const unsigned mine = __ballot_sync(ABC_FULL, left < inc);
            if (mine) {
                if (t == __ffs(mine) - 1) {
                    s_group = g;
                    s_lo = a + (left - (inc - nt)) * SPLIT_TILE;
                    s_hi = min(b, s_lo + SPLIT_TILE);
                }
                break;
            }
            left -= __shfl_sync(ABC_FULL, inc, 31);
        }
    }
    for (int i = t; i < F; i += SPLIT_THREADS) cnt[i] = 0;
    __syncthreads();
    if (s_group < 0) return;  // (the grid is an upper bound)
    const int64_t b0 = (int64_t)s_group << L.shift;
    const int nbin = (int)min((int64_t)F, (int64_t)L.nb - b0);
    const int64_t lo = s_lo;
    const int ne = (int)(s_hi - lo);
    uint64_t k[SPLIT_IPT];
    unsigned r[SPLIT_IPT];
#pragma unroll
    for (int q = 0; q < SPLIT_IPT; ++q) {
        const int i = q * SPLIT_THREADS + t;
        k[q] = i < ne ? __ldcs(&in[lo + i]) : 0;
    }
#pragma unroll
    for (int q = 0; q < SPLIT_IPT; ++q) {
        if (q * SPLIT_THREADS + t < ne) {
            const unsigned a = (unsigned)(k[q] >> (L.rbits + L.cbits));
            r[q] = (a << 16) | atomicAdd(&cnt[a], 1u);
        }
    }
    __syncthreads();
    tile_offsets<SPLIT_THREADS>(cnt, place, L.cur2 + b0, nbin);
#pragma unroll
    for (int q = 0; q < SPLIT_IPT; ++q) {
        if (q * SPLIT_THREADS + t < ne) {
            const unsigned p = cnt[r[q] >> 16] + (r[q] & 0xffffu);
            stage[p] = k[q];
            sbin[p] = (unsigned short)(r[q] >> 16);
        }
    }
    __syncthreads();
    for (int i = t; i < ne; i += SPLIT_THREADS) out[place[sbin[i]] + (unsigned)i] = stage[i];
}

// Place of a row's e-th sorted entry in its shared-memory room: inside each full run of 32 the low five
// bits are mixed with the run's number, so that lanes holding consecutive entries in registers store
// them without bank conflicts.
__device__ __forceinline__ int mixed(int e, int len) { return (e | 31) < len ? e ^ ((e >> 5) & 31) : e; }

// One warp sorts len <= 32 K entries of room[0, len) ascending by a bitonic network, lane l holding
// entries l K ... l K + K - 1: distances below K stay in the lane's registers. The sorted entries
// go back to room at mixed(e).
template <int K>
__device__ __forceinline__ void warp_sort(int32_t *room, int len, int whole) {
    const int lane = threadIdx.x & 31;
    int32_t v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = k * 32 + lane < len ? room[k * 32 + lane] : INT32_MAX;
#pragma unroll
    for (int size = 2; size <= 32 * K; size <<= 1) {
#pragma unroll
        for (int dist = size >> 1; dist >= 1; dist >>= 1) {
            if (dist < K) {
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const int o = k ^ dist;
                    if (o > k) {
                        const bool up = size < K ? (k & size) == 0 : (size == 32 * K || (lane & (size / K)) == 0);
                        const int32_t a = min(v[k], v[o]), b = max(v[k], v[o]);
                        v[k] = up ? a : b;
                        v[o] = up ? b : a;
                    }
                }
            } else {
                const int dl = dist / K;
                const bool up = size == 32 * K || (lane & (size / K)) == 0;
                const bool keep_min = ((lane & dl) == 0) == up;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const int32_t o = __shfl_xor_sync(ABC_FULL, v[k], dl);
                    v[k] = keep_min ? min(v[k], o) : max(v[k], o);
                }
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int e = lane * K + k;
        if (e < len) room[mixed(e, whole)] = v[k];
    }
    __syncwarp();
}

__device__ __forceinline__ void warp_sort_any(int32_t *room, int len, int whole) {
    if (len <= 64) warp_sort<2>(room, len, whole);
    else if (len <= 128) warp_sort<4>(room, len, whole);
    else if (len <= 256) warp_sort<8>(room, len, whole);
    else if (len <= 512) warp_sort<16>(room, len, whole);
    else warp_sort<32>(room, len, whole);
}

// A warp a row: up to 32 entries by a network over the lanes, up to WARP_ROW by warp_sort (longer rows are left).
// `end[i]` is row i's end in `room`. Returns whether a row holds an entry twice.
__device__ __forceinline__ bool sort_rows(int32_t *room, const unsigned short *end, int nr, int32_t add, int32_t *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    bool twice = false;
    for (int i = threadIdx.x >> 5; i < nr; i += blockDim.x >> 5) {
        const int s = i > 0 ? end[i - 1] : 0, len = end[i] - s;
        if (len > WARP_ROW) continue;
        if (len > 32) warp_sort_any(room + s, len, len);
        int32_t last = -1;
        for (int e = lane; e - lane < len; e += 32) {
            int32_t v = e < len ? room[s + (len > 32 ? mixed(e, len) : e)] : INT32_MAX;
            if (len <= 32) {
#pragma unroll
                for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
                    for (int d = size >> 1; d >= 1; d >>= 1) {
                        const int32_t o = __shfl_xor_sync(ABC_FULL, v, d);
                        v = (((lane & d) == 0) == ((lane & size) == 0 || size == 32)) ? min(v, o) : max(v, o);
                    }
                }
            }
            const int32_t up = __shfl_up_sync(ABC_FULL, v, 1);
            const int32_t before = lane == 0 ? last : up;
            if (e < len) {
                twice |= before == v;
                out[s + e] = v + add;
            }
            last = __shfl_sync(ABC_FULL, v, 31);
        }
        __syncwarp();
    }
    return twice;
}

// The rows of one bin of a layer holding more than `above` and at most CAP edges (see the section's header).
// Three ways by row length: bins of short rows, where every entry counts the smaller ones of its row (a
// network over 32 lanes idles on rows of 20: 160 instructions per 32 entries against 95); rows up to
// WARP_ROW, a warp each; longer ones by the whole block, runs of WARP_ROW by its warps and then merged
// pairwise, each thread finding where its share of the output starts in both runs and merging on.
// 256 threads and four blocks an SM: a bin of 4,096 edges has few rows where rows are long, and with
// twice the warps in half the blocks more of them idled.
template <int CAP, int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) k_rows(const uint64_t *__restrict__ keys, LayerBins L, const int64_t *__restrict__ off,
                                                        int64_t obase, int above, int32_t add, int32_t *__restrict__ adj, int *err) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    int32_t *room = reinterpret_cast<int32_t *>(sm_raw);           // [CAP] the bin's columns, row by row
    unsigned *cur = reinterpret_cast<unsigned *>(room + CAP);      // [CAP / 2 + 1] 16-bit next places, two rows a word
    unsigned short *rowof = reinterpret_cast<unsigned short *>(cur + CAP / 2 + 1);  // [CAP] an entry's row (short rows)
    __shared__ int s_max, s_nbig, s_sum;
    __shared__ int s_big[CAP / WARP_ROW + 1];
    constexpr int PER = CAP / THREADS;
    const int t = threadIdx.x;
    const int64_t s = L.start[blockIdx.x];
    const int64_t c64 = L.start[blockIdx.x + 1] - s;
    if (c64 <= above || c64 > CAP) return;
    const int c = (int)c64;
    const int32_t r0 = L.row[blockIdx.x];
    const int nr = L.row[blockIdx.x + 1] - r0;
    if (t == 0) s_max = s_nbig = s_sum = 0;
    __syncthreads();
    const int64_t *o = off + r0;  // this layer's offsets, less obase
    int mx = 0;
    for (int w = t; 2 * w < nr; w += THREADS) {
        const int64_t a = o[2 * w], b = o[2 * w + 1], e = 2 * w + 2 <= nr ? o[2 * w + 2] : b;
        const int la = (int)(b - a), lb = (int)(e - b);
        cur[w] = (unsigned)(a - obase - s) | ((unsigned)(b - obase - s) << 16);
        mx = max(mx, max(la, lb));
        if (la > WARP_ROW) s_big[atomicAdd(&s_nbig, 1)] = 2 * w;
        if (lb > WARP_ROW) s_big[atomicAdd(&s_nbig, 1)] = 2 * w + 1;
    }
    mx = __reduce_max_sync(ABC_FULL, mx);
    if ((t & 31) == 0 && mx) atomicMax(&s_max, mx);
    __syncthreads();
    const bool short_rows = s_max <= SHORT_ROW;
    constexpr int KILP = 4;
    for (int i = t; i < c; i += THREADS * KILP) {
        uint64_t k[KILP];
#pragma unroll
        for (int q = 0; q < KILP; ++q)
            if (i + q * THREADS < c) k[q] = __ldcs(&keys[s + i + q * THREADS]);
#pragma unroll
        for (int q = 0; q < KILP; ++q)
            if (i + q * THREADS < c) {
                const int r = L.key_row(k[q]) - r0, sh = (r & 1) << 4;
                const unsigned old = atomicAdd(&cur[r >> 1], 1u << sh);
                const int at = (int)((old >> sh) & 0xffffu);
                room[at] = L.key_col(k[q]);
                if (short_rows) rowof[at] = (unsigned short)r;
            }
    }
    __syncthreads();
    // every cursor has reached its row's end
    const unsigned short *end = reinterpret_cast<const unsigned short *>(cur);
    int32_t *out = adj + s;
    bool twice = false;
    if (short_rows) {
        // distinct entries of a row rank 0, 1, ..., as many as their places do; an entry given twice makes the ranks'
        // sum smaller
        int sum = 0;
        for (int e = t; e < c; e += THREADS) {
            const int r = rowof[e], b = r > 0 ? end[r - 1] : 0, f = end[r];
            const int32_t v = room[e];
            int rank = 0;
            for (int j = b; j < f; ++j) rank += room[j] < v ? 1 : 0;
            out[b + rank] = v + add;
            sum += rank - (e - b);
        }
        sum = __reduce_add_sync(ABC_FULL, sum);
        if ((t & 31) == 0 && sum) atomicAdd(&s_sum, sum);
        __syncthreads();
        twice = s_sum != 0;
    } else {
        twice = sort_rows(room, end, nr, add, out);
    }
    for (int q = 0; q < s_nbig; ++q) {
        const int i = s_big[q];
        const int b = i > 0 ? end[i - 1] : 0, len = end[i] - b;
        int32_t *row = room + b;
        for (int e = (t >> 5) * WARP_ROW; e < len; e += (THREADS / 32) * WARP_ROW)
            warp_sort_any(row + e, min(WARP_ROW, len - e), min(WARP_ROW, len - e));
        __syncthreads();
        auto at = [&](int e) { return row[mixed(e, len)]; };
        const int per = (len + THREADS - 1) / THREADS, d0 = min(t * per, len), d1 = min(d0 + per, len);
        for (int w = WARP_ROW; w < len; w <<= 1) {
            // outputs [d0, d1): from the pair of runs [a0, a0 + an), [b0, b0 + bn) they start in, and on into the next
            int a0 = d0 / (2 * w) * (2 * w), an = min(w, len - a0), b0 = a0 + an, bn = min(w, len - b0);
            const int k = d0 - a0;
            int lo = max(0, k - bn), hi = min(k, an);
            while (lo < hi) {
                const int h = (lo + hi) >> 1;
                if (at(a0 + h) <= at(b0 + k - 1 - h)) lo = h + 1;
                else hi = h;
            }
            int x = lo, y = k - lo;
            int32_t va = x < an && d0 < d1 ? at(a0 + x) : INT32_MAX, vb = y < bn && d0 < d1 ? at(b0 + y) : INT32_MAX;
            int32_t v[PER];
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                v[j] = 0;
                if (d0 + j < d1) {
                    if (x == an && y == bn) {
                        a0 = b0 + bn;
                        an = min(w, len - a0);
                        b0 = a0 + an;
                        bn = min(w, len - b0);
                        x = y = 0;
                        va = at(a0);
                        vb = bn > 0 ? at(b0) : INT32_MAX;
                    }
                    const bool first = va <= vb;
                    v[j] = first ? va : vb;
                    if (first) {
                        ++x;
                        va = x < an ? at(a0 + x) : INT32_MAX;
                    } else {
                        ++y;
                        vb = y < bn ? at(b0 + y) : INT32_MAX;
                    }
                }
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (d0 + j < d1) row[mixed(d0 + j, len)] = v[j];
            __syncthreads();
        }
        for (int e = t; e < len; e += THREADS) {
            const int32_t v = at(e);
            twice |= e > 0 && at(e - 1) == v;
            out[b + e] = v + add;
        }
    }
    if (__any_sync(ABC_FULL, twice) && (t & 31) == 0) abc::set_error(err, ABCORE_EEXIST);
}
constexpr size_t rows_smem(int cap) { return (size_t)cap * 4 + (size_t)(cap / 2 + 1) * 4 + (size_t)cap * 2; }

// Bins above ROWS_CAP_BIG (a row of more than 20,000 edges starts there): listed with the positions their edges get in a
// list of their own, which is radix-sorted by (row, column). res: {bins, edges, rows up to the last of them}.
__global__ void __launch_bounds__(1024) k_over_list(LayerBins L, int32_t *obin, int64_t *oofs, int64_t *res) {
    __shared__ long long s_n[1024], s_e[1024];
    const int t = threadIdx.x;
    const int64_t per = ((int64_t)L.nb + 1023) / 1024, b0 = t * per, b1 = min(b0 + per, (int64_t)L.nb);
    long long cn = 0, ce = 0, last = 0;
    for (int64_t b = b0; b < b1; ++b) {
        const int64_t c = L.start[b + 1] - L.start[b];
        if (c > ROWS_CAP_BIG) {
            ++cn;
            ce += c;
            last = L.row[b + 1];
        }
    }
    s_n[t] = cn;
    s_e[t] = ce;
    __syncthreads();
    for (int d = 1; d < 1024; d <<= 1) {
        const long long a = t >= d ? s_n[t - d] : 0, b = t >= d ? s_e[t - d] : 0;
        __syncthreads();
        s_n[t] += a;
        s_e[t] += b;
        __syncthreads();
    }
    long long in = s_n[t] - cn, ie = s_e[t] - ce;
    for (int64_t b = b0; b < b1; ++b) {
        const int64_t c = L.start[b + 1] - L.start[b];
        if (c > ROWS_CAP_BIG) {
            obin[in] = (int32_t)b;
            oofs[in] = ie;
            ++in;
            ie += c;
        }
    }
    if (t == 1023) {
        res[0] = s_n[1023];
        res[1] = s_e[1023];
        oofs[s_n[1023]] = s_e[1023];
    }
    if (last) atomicMax((long long *)&res[2], last);
}

// The listed bins' keys without their bins' numbers (blockIdx.y: the bin).
__global__ void __launch_bounds__(256) k_over_take(const uint64_t *__restrict__ keys, LayerBins L, const int32_t *__restrict__ obin,
                                                   const int64_t *__restrict__ oofs, int64_t nover, uint64_t *__restrict__ list) {
    for (int64_t q = blockIdx.y; q < nover; q += gridDim.y) {
        const int64_t s = L.start[obin[q]], c = oofs[q + 1] - oofs[q];
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < c; i += (int64_t)gridDim.x * blockDim.x) {
            list[oofs[q] + i] = keys[s + i] & (((uint64_t)1 << (L.rbits + L.cbits)) - 1);
        }
    }
}

// ... and back, sorted: a bin's edges lie together in the list, in the order of its rows.
__global__ void __launch_bounds__(256) k_over_put(const uint64_t *__restrict__ list, LayerBins L, const int32_t *__restrict__ obin,
                                                  const int64_t *__restrict__ oofs, int64_t nover, uint64_t cmask, int32_t add,
                                                  int32_t *__restrict__ adj, int *err) {
    for (int64_t q = blockIdx.y; q < nover; q += gridDim.y) {
        const int64_t s = L.start[obin[q]], f = oofs[q], c = oofs[q + 1] - f;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < c; i += (int64_t)gridDim.x * blockDim.x) {
            const uint64_t k = list[f + i];
            if (i > 0 && list[f + i - 1] == k) abc::set_error(err, ABCORE_EEXIST);
            adj[s + i] = (int32_t)(k & cmask) + add;
        }
    }
}
// Expand a CSR into the row id of every entry: one warp per row.
__global__ void k_expand_rows(const int64_t *__restrict__ off, int32_t nrows, int32_t *__restrict__ rowid) {
    const int lane = threadIdx.x & 31;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < nrows;
         r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t s = off[r], e = off[r + 1];
        for (int64_t j = s + lane; j < e; j += 32) rowid[j] = (int32_t)r;
    }
}

__global__ void k_check_off(const int64_t *__restrict__ off, int32_t nrows, int64_t m, int *err) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrows;
         r += (int64_t)gridDim.x * blockDim.x) {
        if (off[r + 1] < off[r]) abc::set_error(err, ABCORE_EINVAL);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && (off[0] != 0 || off[nrows] != m))
        abc::set_error(err, ABCORE_EINVAL);
}

__global__ void k_pair_keys(const int32_t *__restrict__ a, const int32_t *__restrict__ b, int64_t m,
                            int32_t nb, uint64_t *__restrict__ keys) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x)
        keys[i] = (uint64_t)a[i] * (uint64_t)nb + (uint64_t)b[i];
}

__global__ void k_diff(const uint64_t *__restrict__ a, const uint64_t *__restrict__ b, int64_t m, int *err) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x)
        if (a[i] != b[i]) abc::set_error(err, ABCORE_EINVAL);
}

int bits_for(int64_t n) {  // bits needed to hold values 0..n-1 (at least 1)
    int b = 1;
    while (b < 63 && ((int64_t)1 << b) < n) ++b;
    return b;
}

unsigned grid_for(abcore_ctx *ctx, int64_t n, int threads = 256) {
    int64_t g = (n + threads - 1) / threads;
    int64_t cap = (int64_t)ctx->num_sms * 16;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (unsigned)g;
}

int read_err(abcore_ctx *ctx, int *d_err, int *h_err) {
    ABC_CU(cudaMemcpyAsync(h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    ABC_CU(cudaStreamSynchronize(ctx->stream));
    return ABCORE_OK;
}

}  // namespace

void free_graph_of(abcore_ctx *ctx, Graph &g) {
    ctx->release(g.off);
    ctx->release(g.adj);
    ctx->release(g.new2old);
    ctx->release(g.old2new);
    g.cntU_ge.clear(); g.edgesU_ge.clear(); g.cntV_ge.clear(); g.edgesV_ge.clear();
    g.loaded = false;
    g.nU = g.nV = 0;
    g.m = 0;
}

void free_graph(abcore_ctx *ctx) {
    free_pruning(ctx);
    free_graph_of(ctx, ctx->g);
}

int check_csr_offsets(abcore_ctx *ctx, int32_t nrows, const int64_t *d_off, int64_t m) {
    int *d_err = nullptr;
    ABC_TRY(ctx->alloc(&d_err, 1, "error word"));
    int h_err = 0;
    cudaMemsetAsync(d_err, 0, sizeof(int), ctx->stream);
    k_check_off<<<grid_for(ctx, nrows), 256, 0, ctx->stream>>>(d_off, nrows, m, d_err);
    int rc = read_err(ctx, d_err, &h_err);
    ctx->release(d_err);
    if (rc) return rc;
    if (h_err) return ctx->fail(ABCORE_EINVAL, "CSR offsets must start at 0, be non-decreasing and end at m");
    return ABCORE_OK;
}

int expand_csr_to_edges(abcore_ctx *ctx, int32_t nrows, const int64_t *d_off, const int32_t *d_adj,
                        int64_t m, int32_t *d_rowid) {
    (void)d_adj;
    (void)m;
    if (nrows > 0)
        k_expand_rows<<<grid_for(ctx, (int64_t)nrows * 32), 256, 0, ctx->stream>>>(d_off, nrows, d_rowid);
    ABC_CU(cudaGetLastError());
    return ABCORE_OK;
}

// Compare two edge lists as sets (both distinct): EINVAL if they differ.
int compare_edge_sets(abcore_ctx *ctx, int32_t nV, int64_t m, const int32_t *eu1, const int32_t *ev1,
                      const int32_t *eu2, const int32_t *ev2) {
    uint64_t *a = nullptr, *b = nullptr, *c = nullptr, *d = nullptr;
    int *d_err = nullptr;
    int rc = ctx->alloc(&a, (size_t)m, "validate keys");
    if (!rc) rc = ctx->alloc(&b, (size_t)m, "validate keys");
    if (!rc) rc = ctx->alloc(&c, (size_t)m, "validate keys");
    if (!rc) rc = ctx->alloc(&d, (size_t)m, "validate keys");
    if (!rc) rc = ctx->alloc(&d_err, 1, "error word");
    int h_err = 0;
    if (!rc) {
        cudaMemsetAsync(d_err, 0, sizeof(int), ctx->stream);
        k_pair_keys<<<grid_for(ctx, m), 256, 0, ctx->stream>>>(eu1, ev1, m, nV, a);
        k_pair_keys<<<grid_for(ctx, m), 256, 0, ctx->stream>>>(eu2, ev2, m, nV, c);
        int64_t maxkey = (int64_t)ctx->g.nU * nV;
        int bits = bits_for(maxkey > 1 ? maxkey : 2);
        uint64_t *r1, *r2;
        rc = radix_sort_u64(ctx, a, b, m, 0, bits, &r1);
        if (!rc) rc = radix_sort_u64(ctx, c, d, m, 0, bits, &r2);
        if (!rc) {
            k_diff<<<grid_for(ctx, m), 256, 0, ctx->stream>>>(r1, r2, m, d_err);
            rc = read_err(ctx, d_err, &h_err);
        }
    }
    ctx->release(a); ctx->release(b); ctx->release(c); ctx->release(d); ctx->release(d_err);
    if (rc) return rc;
    if (h_err) return ctx->fail(ABCORE_EINVAL, "the two CSR layers describe different edge sets");
    return ABCORE_OK;
}

int build_graph_from_device_edges(abcore_ctx *ctx, int32_t nU, int32_t nV, int64_t m,
                                  const int32_t *d_eu, const int32_t *d_ev) {
    free_graph(ctx);
    return build_graph(ctx, ctx->g, nU, nV, m, d_eu, d_ev, nullptr, 0);
}

int csr_edges(abcore_ctx *ctx, const Graph &g, int32_t *d_eu, int32_t *d_ev) {
    int32_t *rowid = nullptr;
    ABC_TRY(ctx->alloc(&rowid, (size_t)std::max<int64_t>(g.m, 1), "edge rows"));
    int rc = expand_csr_to_edges(ctx, g.nU, g.off, g.adj, g.m, rowid);
    if (!rc && g.m > 0) {
        k_edges_of<<<grid_for(ctx, g.m), 256, 0, ctx->stream>>>(rowid, g.adj, g.m, g.new2old, d_eu, d_ev);
        const cudaError_t e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) rc = ctx->cuda_fail(e, "edge list");
    }
    ctx->release(rowid);
    return rc;
}

// One layer's rows from its keys in bin order: rows of at most ROWS_CAP_BIG edges in shared memory, the rest by radix
// sort of their bins' keys (over: {bins, edges, rows}; la, lb: room for those edges).
static int layer_rows(abcore_ctx *ctx, const Graph &g, const LayerBins &L, int l, int32_t nU, int64_t m, int maxdeg, const uint64_t *keys,
                      int32_t *out, const int64_t *over, const int32_t *obin, const int64_t *oofs, uint64_t *la,
                      uint64_t *lb, int *d_err) {
    const int32_t add = l ? 0 : nU;
    const int64_t obase = l ? m : 0;
    const int64_t *off = g.off + (l ? nU : 0);
    // (a bin holds less than BIN_EDGES edges besides its last row's)
#define ROWS(cap, threads, minb, above)                                                                                        \
    if (above == 0 || maxdeg > above - BIN_EDGES) {                                                                            \
        ABC_CU(cudaFuncSetAttribute(k_rows<cap, threads, minb>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rows_smem(cap))); \
        k_rows<cap, threads, minb><<<(unsigned)L.nb, threads, rows_smem(cap), ctx->stream>>>(keys, L, off, obase, above, add, out, d_err); \
    }
    ROWS(ROWS_CAP, 256, 4, 0)
    ROWS(ROWS_CAP_MID, 512, 2, ROWS_CAP)
    ROWS(ROWS_CAP_BIG, 1024, 1, ROWS_CAP_MID)
#undef ROWS
    if (over[1] > 0) {
        const dim3 grid((unsigned)std::min<int64_t>((over[1] / over[0] + 255) / 256 + 1, 64), (unsigned)std::min<int64_t>(over[0], 16384));
        k_over_take<<<grid, 256, 0, ctx->stream>>>(keys, L, obin, oofs, over[0], la);
        uint64_t *sorted;
        ABC_TRY(radix_sort_u64(ctx, la, lb, over[1], 0, L.cbits + bits_for(over[2]), &sorted));
        k_over_put<<<grid, 256, 0, ctx->stream>>>(sorted, L, obin, oofs, over[0], ((uint64_t)1 << L.cbits) - 1, add, out, d_err);
    }
    ABC_CU(cudaGetLastError());
    return ABCORE_OK;
}

// Both layers' adjacency from the edge list, offsets and numbering done. ka, kb: room for m keys each.
static int edges_into_rows(abcore_ctx *ctx, Graph &g, int32_t nU, int32_t nV, int64_t m, const int32_t *d_eu, const int32_t *d_ev,
                           uint64_t *ka, uint64_t *kb, int *d_err) {
    const int64_t n = (int64_t)nU + nV;
    const int rowbits[2] = {bits_for(std::max<int32_t>(nU, 1)), bits_for(std::max<int32_t>(nV, 1))};
    const int maxdeg[2] = {g.maxdegU, g.maxdegV};
    Bins B{};
    LayerBins *const lay[2] = {&B.u, &B.v};
    int32_t nb = 0, shift = 0;
    int64_t *words = nullptr, *oofs = nullptr;
    int32_t *rows = nullptr, *obin = nullptr;
    uint64_t *la = nullptr, *lb = nullptr;
    int rc = ABCORE_OK;
    nb = (int32_t)((m + BIN_EDGES - 1) / BIN_EDGES);
    const bool two = nb > SPLIT_BINS;
    if (two)
        while ((nb >> shift) >= (shift < 10 ? GROUPS : SPLIT_BINS)) ++shift;
    // a bin's number in its group takes 10 bits of an edge's place in its tile, and `shift` of its key beside two ids;
    // past 4.3e9 edges, or with ids of 55 bits together and a billion edges, both layers are sorted whole
    const bool fits = shift <= 10 && rowbits[0] + rowbits[1] + shift <= 64;
    const int ngroups = (nb + (1 << shift) - 1) >> shift;
    const int64_t nb1 = (int64_t)nb + 1;
#define STEP(x)            \
    do {                   \
        rc = (x);          \
        if (rc) goto done; \
    } while (0)
    STEP(ctx->alloc(&B.rec, (size_t)n, "vertex records"));
    STEP(ctx->alloc(&words, (size_t)(6 * nb1 + 8), "row bins"));
    STEP(ctx->alloc(&rows, (size_t)(2 * nb1), "row bins"));
    for (int l = 0; l < 2; ++l) {
        *lay[l] = {words + l * nb1, rows + l * nb1, (unsigned long long *)(words + (2 + l) * nb1),
                   (unsigned long long *)(words + (4 + l) * nb1), nb, shift, rowbits[l], rowbits[1 - l]};
    }
    {
        k_bins<<<grid_for(ctx, n), 256, 0, ctx->stream>>>(g.off, g.new2old, nU, n, m, B);
        k_cursors<<<dim3(grid_for(ctx, nb), 2), 256, 0, ctx->stream>>>(B);
        // rows too long for k_rows: how many edges lie in their bins
        int64_t over[2][3] = {};
        if (fits && std::max(maxdeg[0], maxdeg[1]) > ROWS_CAP_BIG - BIN_EDGES) {
            STEP(ctx->alloc(&oofs, (size_t)(2 * nb1), "long rows"));
            STEP(ctx->alloc(&obin, (size_t)(2 * nb1), "long rows"));
            int64_t *res = words + 6 * nb1;
            rc = cudaMemsetAsync(res, 0, 6 * sizeof(int64_t), ctx->stream) == cudaSuccess ? rc : ctx->fail(ABCORE_ECUDA, "long rows");
            for (int l = 0; l < 2; ++l) k_over_list<<<1, 1024, 0, ctx->stream>>>(*lay[l], obin + l * nb1, oofs + l * nb1, res + 3 * l);
            cudaMemcpyAsync(over, res, sizeof(over), cudaMemcpyDeviceToHost, ctx->stream);
            const cudaError_t e = cudaStreamSynchronize(ctx->stream);
            if (e != cudaSuccess) STEP(ctx->cuda_fail(e, "long rows"));
        }
        // a layer with more than an eighth of its edges there is sorted whole, by (row, column)
        bool whole[2];
        for (int l = 0; l < 2; ++l) {
            whole[l] = !fits || over[l][1] > m / 8;
            if (!whole[l]) continue;
            const int cbits = rowbits[1 - l];
            k_edge_keys<<<grid_for(ctx, m), 256, 0, ctx->stream>>>(d_eu, d_ev, m, g.old2new, nU, l == 0, cbits, ka);
            uint64_t *sorted;
            STEP(radix_sort_u64(ctx, ka, kb, m, 0, cbits + rowbits[l], &sorted));
            k_extract<<<grid_for(ctx, m), 256, 0, ctx->stream>>>(sorted, m, ((uint64_t)1 << cbits) - 1, l == 0 ? nU : 0,
                                                                 g.adj + l * m, d_err);
        }
        if (!(whole[0] && whole[1])) {
            const size_t split_smem = (size_t)SPLIT_TILE * 10 + (size_t)ngroups * 16;
            const size_t group_smem = (size_t)SPLIT_TILE * 10 + ((size_t)12 << shift);
            const unsigned tiles = (unsigned)((m + SPLIT_TILE - 1) / SPLIT_TILE);
            uint64_t *a2 = ka, *b2 = kb, *t2 = (uint64_t *)g.adj;
            // (the largest either uses: the limit belongs to the function, which other contexts launch too)
            cudaFuncSetAttribute(k_split, cudaFuncAttributeMaxDynamicSharedMemorySize, SPLIT_TILE * 10 + SPLIT_BINS * 16);
            cudaFuncSetAttribute(k_regroup, cudaFuncAttributeMaxDynamicSharedMemorySize, SPLIT_TILE * 10 + SPLIT_BINS * 12);
            // (one layer alone goes to ka, so that kb is free for its second move)
            k_split<<<tiles, SPLIT_THREADS, split_smem, ctx->stream>>>(d_eu, d_ev, m, nU, B, ngroups, whole[0] ? nullptr : a2,
                                                                       whole[1] ? nullptr : whole[0] ? a2 : b2);
            auto regroup = [&](int l, const uint64_t *in, uint64_t *out) {
                k_regroup<<<tiles + (unsigned)ngroups, SPLIT_THREADS, group_smem, ctx->stream>>>(in, out, *lay[l], ngroups);
            };
            auto rows_of = [&](int l, const uint64_t *keys, int32_t *out, uint64_t *p, uint64_t *q) {
                return layer_rows(ctx, g, *lay[l], l, nU, m, maxdeg[l], keys, out, over[l], obin + l * nb1, oofs + l * nb1, p, q,
                                  d_err);
            };
            if (!two) {
                const int64_t most = std::max(whole[0] ? 0 : over[0][1], whole[1] ? 0 : over[1][1]);
                if (most > 0) {
                    STEP(ctx->alloc(&la, (size_t)most, "long rows"));
                    STEP(ctx->alloc(&lb, (size_t)most, "long rows"));
                }
                if (!whole[0]) STEP(rows_of(0, a2, g.adj, la, lb));
                if (!whole[1]) STEP(rows_of(1, whole[0] ? a2 : b2, g.adj + m, la, lb));
            } else if (whole[0] || whole[1]) {
                const int l = whole[0] ? 1 : 0;
                regroup(l, a2, b2);
                STEP(rows_of(l, b2, g.adj + l * m, ka, ka + over[l][1]));
            } else {
                // three moves need a third room: the V keys' bins go to the adjacency's (m keys fill it exactly), so
                // the V rows are written aside and copied once those keys are used up
                regroup(1, b2, t2);
                regroup(0, a2, b2);
                uint64_t *list = ka + (m + 1) / 2;
                STEP(rows_of(1, t2, (int32_t *)ka, list, list + over[1][1]));
                const cudaError_t e = cudaMemcpyAsync(g.adj + m, ka, sizeof(int32_t) * (size_t)m, cudaMemcpyDeviceToDevice, ctx->stream);
                if (e != cudaSuccess) STEP(ctx->cuda_fail(e, "lower layer's rows"));
                STEP(rows_of(0, b2, g.adj, ka, ka + over[0][1]));
            }
        }
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = ctx->cuda_fail(e, "edges into rows");
    }
done:
    ctx->release(B.rec);
    ctx->release(words);
    ctx->release(rows);
    ctx->release(oofs);
    ctx->release(obin);
    ctx->release(la);
    ctx->release(lb);
    return rc;
#undef STEP
}

int build_graph(abcore_ctx *ctx, Graph &g, int32_t nU, int32_t nV, int64_t m, const int32_t *d_eu,
                const int32_t *d_ev, const int32_t *d_rank, int32_t maxrank) {
    const int64_t n = (int64_t)nU + nV;
    int32_t *deg = nullptr, *degnew = nullptr;
    int *d_words = nullptr;  // {error, largest degree of U, of V}
    uint64_t *ka = nullptr, *kb = nullptr, *rk = nullptr;
    int64_t *tables = nullptr, *h_tables = nullptr;
    int h_words[3] = {0, 0, 0};
    int rc = ABCORE_OK;

#define STEP(x)            \
    do {                   \
        rc = (x);          \
        if (rc) goto fail; \
    } while (0)
#define STEP_CU(x)                                            \
    do {                                                      \
        const cudaError_t e_ = (x);                           \
        if (e_ != cudaSuccess) STEP(ctx->cuda_fail(e_, #x));  \
    } while (0)

    STEP(ctx->alloc(&deg, (size_t)n, "degrees"));
    STEP(ctx->alloc(&degnew, (size_t)n, "sorted degrees"));
    STEP(ctx->alloc(&d_words, 3, "error word"));
    STEP(ctx->alloc(&g.off, (size_t)n + 1, "row offsets"));
    STEP(ctx->alloc(&g.adj, (size_t)(2 * m), "adjacency"));
    STEP(ctx->alloc(&g.new2old, (size_t)n, "new2old"));
    STEP(ctx->alloc(&g.old2new, (size_t)n, "old2new"));
    STEP_CU(cudaMemsetAsync(deg, 0, sizeof(int32_t) * (size_t)(n ? n : 1), ctx->stream));
    STEP_CU(cudaMemsetAsync(d_words, 0, 3 * sizeof(int), ctx->stream));
    if (m > 0)
        k_count_deg<<<grid_for(ctx, m), 256, 0, ctx->stream>>>(d_eu, d_ev, m, nU, nV, deg, deg + nU, d_words);
    if (n > 0) k_max<<<std::min<unsigned>(grid_for(ctx, n), (unsigned)ctx->num_sms * 4), 256, 0, ctx->stream>>>(deg, nU, n, d_words + 1);
    STEP_CU(cudaMemcpyAsync(h_words, d_words, sizeof(h_words), cudaMemcpyDeviceToHost, ctx->stream));
    STEP_CU(cudaStreamSynchronize(ctx->stream));
    if (h_words[0]) {
        rc = ctx->fail(ABCORE_EINVAL, "edge endpoint out of range (u must be < nU, v < nV)");
        goto fail;
    }
    g.maxdegU = h_words[1];
    g.maxdegV = h_words[2];

    {
        const int64_t kcap = std::max<int64_t>(std::max<int64_t>(m, n), 1);
        STEP(ctx->alloc(&ka, (size_t)kcap, "sort keys"));
        STEP(ctx->alloc(&kb, (size_t)kcap, "sort keys"));
        // renumber each layer by non-increasing degree; ties keep caller-id order (stable)
        const int dbits = bits_for((int64_t)std::max(g.maxdegU, g.maxdegV) + 1);
        if (n > 0) {
            k_relabel_keys<<<grid_for(ctx, n), 256, 0, ctx->stream>>>(deg, nU, n, g.maxdegU, g.maxdegV, dbits, ka);
            uint64_t *sorted;
            STEP(radix_sort_u64(ctx, ka, kb, n, 32, 32 + dbits + 1, &sorted));
            if (!d_rank) {
                k_relabel_finish<<<grid_for(ctx, n), 256, 0, ctx->stream>>>(sorted, nU, n, g.maxdegU, g.maxdegV, dbits, g.new2old,
                                                                            g.old2new, degnew);
            } else {
                // then by non-increasing rank, ties keeping the degree order
                STEP(ctx->alloc(&rk, (size_t)n * 2, "rank keys"));
                const int rbits = bits_for((int64_t)maxrank + 1);
                k_rank_keys<<<grid_for(ctx, n), 256, 0, ctx->stream>>>(sorted, nU, n, d_rank, maxrank, rbits, rk);
                uint64_t *sorted2;
                STEP(radix_sort_u64(ctx, rk, rk + n, n, 32, 32 + rbits + 1, &sorted2));
                k_rank_finish<<<grid_for(ctx, n), 256, 0, ctx->stream>>>(sorted2, sorted, nU, n, g.maxdegU, g.maxdegV, dbits, g.new2old,
                                                                         g.old2new, degnew);
                ctx->release(rk);
            }
        }
        STEP(exclusive_scan_i32(ctx, degnew, n, g.off));
        ctx->release(deg);
        ctx->release(degnew);
        if (m > 0) STEP(edges_into_rows(ctx, g, nU, nV, m, d_eu, d_ev, ka, kb, d_words));
    }
    // host tables: vertices and edges at or above each degree threshold, per layer (a graph
    // ordered by rank is not in degree order, and gets none)
    {
        const size_t tu = (size_t)g.maxdegU + 2, tv = (size_t)g.maxdegV + 2, all = 2 * (tu + tv);
        const int64_t *src = nullptr;
        if (!d_rank) {
            STEP(ctx->alloc(&tables, all, "degree tables"));
            DegTables T{{tables, tables + 2 * tu}, {tables + tu, tables + 2 * tu + tv}, {g.maxdegU, g.maxdegV}};
            k_cnt_ge<<<dim3(grid_for(ctx, std::max<int64_t>(std::max(nU, nV), 1)), 2), 256, 0, ctx->stream>>>(g.off, nU, nV, T);
            k_edges_ge<<<dim3(grid_for(ctx, (int64_t)std::max(g.maxdegU, g.maxdegV) + 2), 2), 256, 0, ctx->stream>>>(g.off, nU, T);
            g.cntU_ge.assign(tu, 0);
            g.edgesU_ge.assign(tu, 0);
            g.cntV_ge.assign(tv, 0);
            g.edgesV_ge.assign(tv, 0);
            if (all * sizeof(int64_t) <= (size_t)(8 << 20)) {  // one readback through pinned memory
                STEP(ctx->host_alloc(&h_tables, all, "degree tables"));
                STEP_CU(cudaMemcpyAsync(h_tables, tables, sizeof(int64_t) * all, cudaMemcpyDeviceToHost, ctx->stream));
                src = h_tables;
            } else {
                STEP_CU(cudaMemcpyAsync(g.cntU_ge.data(), T.cnt[0], sizeof(int64_t) * tu, cudaMemcpyDeviceToHost, ctx->stream));
                STEP_CU(cudaMemcpyAsync(g.edgesU_ge.data(), T.edges[0], sizeof(int64_t) * tu, cudaMemcpyDeviceToHost, ctx->stream));
                STEP_CU(cudaMemcpyAsync(g.cntV_ge.data(), T.cnt[1], sizeof(int64_t) * tv, cudaMemcpyDeviceToHost, ctx->stream));
                STEP_CU(cudaMemcpyAsync(g.edgesV_ge.data(), T.edges[1], sizeof(int64_t) * tv, cudaMemcpyDeviceToHost, ctx->stream));
            }
        }
        STEP_CU(cudaMemcpyAsync(h_words, d_words, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        STEP_CU(cudaStreamSynchronize(ctx->stream));
        if (h_words[0]) {
            rc = ctx->fail(ABCORE_EEXIST, "an edge appears more than once in the input");
            goto fail;
        }
        if (src) {
            std::copy(src, src + tu, g.cntU_ge.begin());
            std::copy(src + tu, src + 2 * tu, g.edgesU_ge.begin());
            std::copy(src + 2 * tu, src + 2 * tu + tv, g.cntV_ge.begin());
            std::copy(src + 2 * tu + tv, src + all, g.edgesV_ge.begin());
        }
    }
    ctx->host_release(h_tables);
    ctx->release(tables);
    ctx->release(d_words);
    ctx->release(ka);
    ctx->release(kb);
    g.nU = nU;
    g.nV = nV;
    g.m = m;
    g.loaded = true;
    return ABCORE_OK;

fail:
    cudaStreamSynchronize(ctx->stream);
    ctx->host_release(h_tables);
    ctx->release(deg); ctx->release(degnew); ctx->release(d_words);
    ctx->release(ka); ctx->release(kb); ctx->release(rk); ctx->release(tables);
    free_graph_of(ctx, g);
    return rc;
#undef STEP
#undef STEP_CU
}
