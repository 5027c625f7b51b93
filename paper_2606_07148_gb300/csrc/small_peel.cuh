// A whole (alpha, beta)-core in one block, for graphs that are small enough (Algorithm 1).
//
// The general peel spreads its work over the GPU: a count init, a first round, a cascade through a
// queue in global memory and a mask emission, each a launch, each level of the cascade a round trip
// through L2 for ticket, row, count and queue. With few candidates none of that is needed: their
// counts and the removal queue fit one block's shared memory (6 bytes a candidate), so a level costs
// two loads from L2 (the fallen vertices' offsets and rows), shared-memory atomics and a block barrier, and
// the masks are written by the same launch. What bounds it is latency: the row searches of the count
// init (a thread a candidate) and the levels. One query then takes one launch, and a batch a block per pair.
#pragma once

#include "peel_core.cuh"

namespace abc {

constexpr int SMALL_THREADS = 1024;
constexpr int SMALL_MAX = 36000;  // candidates (216 KB of counts and queue)

// One query: candidate prefixes pU, pV, certain prefixes cU, cV (see PeelArgs) and thresholds.
struct SmallQuery {
    int32_t alpha, beta, pU, pV, cU, cV;
};

// What it did, in the order of the stat counters they stand for.
struct SmallStats {
    unsigned long long inits, probes, entries, decs, pushes;
};

__host__ __device__ __forceinline__ size_t small_smem(int64_t candidates) { return (size_t)candidates * 6 + 16; }

// A removed vertex with a longer row than this is walked by the whole block, up to SMALL_LISTED of them a level: eight
// lanes take a row of 16,000 entries as a chain of 500 steps. (Three hubs of 16,000 falling at once: 407 us the
// eight lanes, 58 the block; 30 of 8,000 181 and 69. A limit of 512 cost queries on graphs with rows of 600 to 1,000 a fifth.)
constexpr int SMALL_LONG = 2048;
constexpr int SMALL_LISTED = 64;
struct SmallRow {
    int64_t s;
    int32_t len, upper;
};

struct SmallGraph {
    const int64_t *off;
    const int32_t *adj;
    const int32_t *old2new;
    int32_t nU, nV;
};

// LONG: some row of the graph is longer than SMALL_LONG. (Compiled apart: the two tests cost every level of a graph without
// them 8 %.) Block-collective; smem: small_smem(candidates) bytes. `out` (shared) receives the statistics.
template <bool LONG>
__device__ __forceinline__ void small_peel(const SmallGraph &G, const SmallQuery &Q, unsigned char *smem, uint8_t *mask_u, uint8_t *mask_v,
                                           SmallStats *out) {
    __shared__ int s_tail, s_nlong;
    __shared__ SmallRow s_long[SMALL_LISTED];
    const int nu = Q.pU - Q.cU, P = nu + (Q.pV - Q.cV);
    int *cnt = reinterpret_cast<int *>(smem);                        // [P] live-neighbour counts, U candidates first
    unsigned short *q = reinterpret_cast<unsigned short *>(cnt + P); // [P] removed candidates
    const int t = threadIdx.x, lane = t & 31;
    unsigned long long probes = 0, entries = 0, decs = 0;
    if (t == 0) {
        s_tail = s_nlong = 0;
        *out = SmallStats{};
    }
    __syncthreads();
    {
        // counts: the row prefix below the other layer's candidate boundary (see init_range)
        const int64_t mU = __ldg(&G.off[G.nU]), mV = __ldg(&G.off[(int64_t)G.nU + G.nV]) - mU;
        const float fU = mU > 0 ? (float)(__ldg(&G.off[(int64_t)G.nU + Q.pV]) - mU) / (float)mU : 0.f;
        const float fV = mV > 0 ? (float)__ldg(&G.off[Q.pU]) / (float)mV : 0.f;
        for (int i = t; i < P; i += SMALL_THREADS) {
            const bool upper = i < nu;
            const int32_t x = upper ? Q.cU + i : G.nU + Q.cV + (i - nu);
            const int64_t s = __ldg(&G.off[x]), e = __ldg(&G.off[x + 1]);
            const int len = e == s ? 0 : row_prefix(G.adj, s, e, upper ? G.nU + Q.pV : Q.pU, upper ? fU : fV, probes);
            cnt[i] = len;
            if (len < (upper ? Q.alpha : Q.beta)) q[atomicAdd(&s_tail, 1)] = (unsigned short)i;
        }
    }
    __syncthreads();
    // One entry of a removed vertex's row: entries [lo, hi) are the other layer's uncertain candidates; entry y counts in
    // cnt[y - lo + at].
    auto lower = [&](int32_t y, int32_t lo, int32_t hi, int32_t at, int thr) {
        if (y < lo || y >= hi) return;
        decs++;
        const int j = y - lo + at;
        if (atomicSub(&cnt[j], 1) == thr) q[atomicAdd(&s_tail, 1)] = (unsigned short)j;  // the crossing: once a vertex
    };
    // levels: eight lanes a removed vertex, four of its row's entries a lane at a time; then the long rows
    constexpr int W = 8, R = 4;
    int head = 0;
    for (;;) {
        const int end = s_tail;
        __syncthreads();  // (everyone has read it before anyone adds to it)
        if (head == end) break;
        for (int k = head + t / W; k < end; k += SMALL_THREADS / W) {
            const int i = q[k];
            const bool upper = i < nu;
            const int32_t x = upper ? Q.cU + i : G.nU + Q.cV + (i - nu);
            const int64_t s = __ldg(&G.off[x]), e = __ldg(&G.off[x + 1]);
            // (a count of 0: every candidate neighbour has fallen, as where hubs fall first; there is nothing to lower)
            if (LONG && cnt[i] == 0) continue;
            if (LONG && e - s > SMALL_LONG) {
                int k2 = 0;
                if (t % W == 0) k2 = atomicAdd(&s_nlong, 1);
                k2 = __shfl_sync(((1u << W) - 1u) << (lane / W * W), k2, lane / W * W);
                if (k2 < SMALL_LISTED) {
                    if (t % W == 0) s_long[k2] = SmallRow{s, (int32_t)(e - s), upper ? 1 : 0};
                    continue;
                }
            }
            const int32_t lo = upper ? G.nU + Q.cV : Q.cU, hi = upper ? G.nU + Q.pV : Q.pU, at = upper ? nu : 0;
            const int thr = upper ? Q.beta : Q.alpha;
            for (int64_t p0 = s + t % W; p0 < e; p0 += W * R) {
                int32_t y[R];
#pragma unroll
                for (int r = 0; r < R; ++r) y[r] = p0 + r * W < e ? __ldg(&G.adj[p0 + r * W]) : INT32_MAX;
#pragma unroll
                for (int r = 0; r < R; ++r) lower(y[r], lo, hi, at, thr);
                entries += R;
                if (y[0] >= hi) break;  // (rows ascend: the rest is past the candidates too)
            }
        }
        head = end;
        __syncthreads();
        if (!LONG) continue;
        const int nl = min(s_nlong, SMALL_LISTED);
        if (nl == 0) continue;
        // chunks of 256 entries, dealt to the warps one after the other
        constexpr int LR = 8, CHUNK = 32 * LR;
        for (int k = 0, dealt = 0; k < nl; ++k) {
            const SmallRow row = s_long[k];
            const int nc = (row.len + CHUNK - 1) / CHUNK;
            const int32_t lo = row.upper ? G.nU + Q.cV : Q.cU, hi = row.upper ? G.nU + Q.pV : Q.pU, at = row.upper ? nu : 0;
            const int thr = row.upper ? Q.beta : Q.alpha;
            for (int c = (t / 32 + SMALL_THREADS / 32 - dealt) % (SMALL_THREADS / 32); c < nc; c += SMALL_THREADS / 32) {
                int32_t y[LR];
#pragma unroll
                for (int r = 0; r < LR; ++r) {
                    const int i = c * CHUNK + r * 32 + lane;
                    y[r] = i < row.len ? __ldg(&G.adj[row.s + i]) : INT32_MAX;
                }
#pragma unroll
                for (int r = 0; r < LR; ++r) lower(y[r], lo, hi, at, thr);
                entries += LR;
                if (y[0] >= hi) break;  // (lane 0's: all that follows in the row is past it too; the other lanes' next chunk as well)
            }
            dealt = (dealt + nc) % (SMALL_THREADS / 32);
        }
        __syncthreads();
        if (t == 0) s_nlong = 0;
    }
    // masks in the caller's order, four ids a thread where the masks' alignment allows
    auto member = [&](int32_t x) -> uint32_t {
        if (x < G.nU) return x < Q.cU || (x < Q.pU && cnt[x - Q.cU] >= Q.alpha);
        const int32_t j = x - G.nU;
        return j < Q.cV || (j < Q.pV && cnt[nu + j - Q.cV] >= Q.beta);
    };
    const int n = G.nU + G.nV;
    if (((reinterpret_cast<uintptr_t>(mask_u) | reinterpret_cast<uintptr_t>(mask_v)) & 3) == 0 && (G.nU & 3) == 0) {
        for (int k = t; k < n / 4; k += SMALL_THREADS) {
            const int4 x = __ldg(reinterpret_cast<const int4 *>(G.old2new) + k);
            const uint32_t b = member(x.x) | member(x.y) << 8 | member(x.z) << 16 | member(x.w) << 24;
            const int i = 4 * k;
            *reinterpret_cast<uint32_t *>(i < G.nU ? mask_u + i : mask_v + (i - G.nU)) = b;
        }
        for (int i = n / 4 * 4 + t; i < n; i += SMALL_THREADS) mask_v[i - G.nU] = (uint8_t)member(__ldg(&G.old2new[i]));
    } else {
        for (int i = t; i < n; i += SMALL_THREADS) {
            const uint8_t b = (uint8_t)member(__ldg(&G.old2new[i]));
            if (i < G.nU) mask_u[i] = b;
            else mask_v[i - G.nU] = b;
        }
    }
    const unsigned long long v[3] = {probes, entries, decs};
    unsigned long long *const d[3] = {&out->probes, &out->entries, &out->decs};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const unsigned long long w = (unsigned long long)warp_sum64((long long)v[k]);
        if (lane == 0 && w) atomicAdd(d[k], w);
    }
    if (t == 0) {
        out->inits = (unsigned long long)P;
        out->pushes = (unsigned long long)head;
    }
    __syncthreads();
}

}  // namespace abc
