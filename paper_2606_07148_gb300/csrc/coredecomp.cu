// Core numbers (Definition 2) and the layout that lets the single query prune with them
// (Lemma 1; Algorithm 2, GCC+).
//
// core(x) is the largest k with x in the (k, k)-core. It is found without peeling: the core numbers are the
// largest values c with c(x) = h(x) at every vertex, h(x) being the h-index of x's neighbours' values (the
// largest h such that h of them are at least h), and replacing values by h-indices from above, in
// any order, until nothing changes reaches exactly them (Lu, Zhou, Zhang and Stanley, "The H-index of a
// network node and its relation to degree and coreness", 2016; asynchronous form: Sariyuce,
// Seshadhri and Pinar, "Local algorithms for hierarchical dense subgraph discovery", 2018). A peel
// goes through every k and every cascade level inside it, one after the other: on a 20M-edge power-law graph
// 1,322 levels of a few vertices each, 15.9 ms of latency. The h-index rounds need up to 60 there and the
// work of about eight passes over the edges, most of it in the first, wide rounds: 3.1 ms. How many rounds there are
// depends on how deep the graph is, since a change moves on by one neighbour a round: a path of n vertices
// has about n / 2. A grid round takes about 10 us whatever its lists hold (barrier, lists, one row's trips to L2), so
// rounds of a few short rows are left to one block (core_narrow), and rows that would hold up a round to
// the whole grid (core_huge). Whole calls, peel of every k / rounds: path of 200,000 vertices 281 / 165 ms, 1,000 x 1,000 grid
// 9.3 / 10.0, 300 x 300 2.96 / 3.06, 20 rows of 2M entries 98 / 60, 300M edges 176 / 60.
//
// Rows ascend in degree order, which bounds what is read: a vertex's first value is the h-index of its
// neighbours' degrees, a binary search in its row; and a neighbour can count for t only if its degree is
// at least t, a prefix of the row.
//
// GCC+ then needs, for thresholds dl <= dq, the vertices with core >= dq (certain members) and
// core >= dl (possible members) as prefixes: a second copy of the graph is built with each layer
// numbered by non-increasing core number (ties in degree order), and per-layer tables of how many
// vertices have core >= t.
#include <algorithm>
#include <chrono>
#include <vector>

#include "device.cuh"
#include "internal.h"
#include "peel_core.cuh"

namespace {

constexpr int CORE_THREADS = 256;
constexpr int CORE_WARPS = CORE_THREADS / 32;
// rows by length: up to CORE_SMALL entries by eight lanes, up to CORE_MID by a warp (in registers), up to CORE_LONG by a
// block, longer by the whole grid
constexpr int CORE_SMALL = 64, CORE_MID = 512, CORE_LONG = 32768;
constexpr int CLASSES = 4;        // 0: the longest
constexpr int CORE_CACHE = 4096;  // values of a long row a block keeps in shared memory
constexpr int CORE_BUF = 128;     // vertices a warp collects before it adds them to a list
constexpr int NARROW = 64;        // lists of up to this many short rows are left to one block (core_narrow), which
constexpr int NARROW_MAX = 256;   // goes on with what those mark while it is not more than this
constexpr int EAGER = 1 << 16;    // see core_mark
constexpr int HUGE_BATCH = 256;   // rows of class 0 the grid takes together
constexpr int HUGE_CHUNK = 4096;  // entries of one a block takes at a time

struct CoreArgs {
    const int64_t *off;
    const int32_t *adj;
    int32_t nU, nV;
    int32_t hU[CLASSES], hV[CLASSES];  // vertices of each layer in the classes up to this one (prefixes; the last: all with an edge)
    const int32_t *gU, *gV;         // vertices of each layer with at least t edges, t = 0 .. maxdeg + 1
    int32_t maxdeg;
    int32_t *val;                   // [n] values, by internal id: in the end the core numbers
    int32_t *queued;                // [n] 1: in the list of this or the next round, not yet looked at
    int32_t *list[2];               // [n] vertices to look at, each class from the number of vertices in those before it
    unsigned *count;                // [3][CLASSES] list lengths: [round % 3][class]
    int32_t *hcnt, *hval, *hist;    // [HUGE_BATCH] of a batch of class 0: entries at or above the value, the new value or -1;
                                    // [HUGE_BATCH][CORE_CACHE] entries by value
    PeelCtl *ctl;
    unsigned long long *bar;        // blocks arrived at the grid's barriers so far
    unsigned long long timeout_ns;
};

// Barrier of the grid, the `passed`-th (counted here): one count that only grows, looked at without reading the clock at
// first. A deep graph goes through hundreds of rounds with little to do between them (a grid of 1,000 x 1,000: 500), and
// the general group barrier, with its two words, its fixup and a clock reading per look, was half of each. Returns
// false if the session saw an error, in which case every block leaves. Block-collective.
__device__ __forceinline__ bool core_barrier(const CoreArgs &C, unsigned long long &passed) {
    __shared__ int s_ok;
    __syncthreads();
    const unsigned long long all = ++passed * gridDim.x;
    if (threadIdx.x == 0) {
        s_ok = 1;
        __threadfence();
        if (atomicAdd(C.bar, 1ull) + 1 < all) {
            int looks = 0;
            unsigned long long t0 = 0;
            while (abc::ld_acquire(C.bar) < all) {
                if (++looks < 64) continue;
                const unsigned long long now = abc::now_ns();
                if (t0 == 0) t0 = now;
                if (now - t0 > C.timeout_ns) abc::set_error(&C.ctl->err, ABCORE_ETIMEDOUT);
                if (abc::ld_relaxed_i32(&C.ctl->err) != 0) {
                    s_ok = 0;
                    break;
                }
                __nanosleep(256);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return s_ok != 0;
}

__device__ __forceinline__ int32_t ld_val(const int32_t *p) {
    int32_t v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The row entries of x that can count for t: ids below this have at least t edges.
__device__ __forceinline__ int32_t id_bound(const CoreArgs &C, bool upper, int32_t t) {
    const int32_t k = min(t, C.maxdeg + 1);
    return upper ? C.nU + __ldg(&C.gV[k]) : __ldg(&C.gU[k]);
}

__device__ __forceinline__ int row_class(const CoreArgs &C, int32_t x) {
    const bool upper = x < C.nU;
    const int32_t i = upper ? x : x - C.nU;
    int c = 0;
#pragma unroll
    for (int k = 0; k < CLASSES - 1; ++k) c += i >= (upper ? C.hU[k] : C.hV[k]) ? 1 : 0;
    return c;
}

// Where a class's part of a list starts.
__device__ __forceinline__ int64_t list_start(const CoreArgs &C, int cls) { return cls == 0 ? 0 : (int64_t)C.hU[cls - 1] + C.hV[cls - 1]; }

// Per warp: vertices to look at next round, collected before they take places in the lists.
struct CoreBuf {
    int32_t x[CORE_BUF];
};

__device__ __forceinline__ void core_flush(const CoreArgs &C, CoreBuf &b, int &nb, int32_t *next, unsigned *count) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    for (int i0 = 0; i0 < nb; i0 += 32) {
        const int32_t x = i0 + lane < nb ? b.x[i0 + lane] : -1;
        const int cls = x >= 0 ? row_class(C, x) : CLASSES;
#pragma unroll
        for (int c = 0; c < CLASSES; ++c) {
            const unsigned m = __ballot_sync(ABC_FULL, cls == c);
            if (m == 0) continue;
            unsigned base = 0;
            if (lane == 0) base = atomicAdd(&count[c], (unsigned)__popc(m));
            base = __shfl_sync(ABC_FULL, base, 0);
            if (cls == c) next[list_start(C, c) + base + __popc(m & abc::lanemask_lt())] = x;
        }
    }
    __syncwarp();
    nb = 0;
}

// Warp-collective: lanes with `want` have neighbour y to look at again. `eager`: the word is not read before it is
// exchanged, a trip to L2 less in rounds of few rows (many rows marking the same vertices would all write it).
__device__ __forceinline__ void core_mark(const CoreArgs &C, CoreBuf &b, int &nb, bool want, int32_t y, int32_t *next, unsigned *count,
                                          bool eager = false) {
    // (a vertex still waiting to be looked at will see the new value: the word is cleared before the values are read)
    const bool add = want && (eager || ld_val(&C.queued[y]) == 0) && atomicExch(&C.queued[y], 1) == 0;
    const unsigned m = __ballot_sync(ABC_FULL, add);
    if (m == 0) return;
    if (add) b.x[nb + __popc(m & abc::lanemask_lt())] = y;
    nb += __popc(m);
    if (nb > CORE_BUF - 32) core_flush(C, b, nb, next, count);
}

// Rows of up to W * R entries, W lanes each, all values in registers: every group of W lanes lowers its vertex x
// (x < 0: none) to the h-index of its neighbours' values. Warp-collective.
template <int W, int R>
__device__ __forceinline__ void core_rows(const CoreArgs &C, int32_t x, CoreBuf &b, int &nb, int32_t *next, unsigned *count, bool eager) {
    const int lane = threadIdx.x & 31, gl = lane % W;
    const unsigned group = W == 32 ? ABC_FULL : ((1u << (W & 31)) - 1u) << (lane / W * W);
    int64_t s = 0;
    int len = 0, e = 0;
    if (x >= 0) {
        if (gl == 0) atomicExch(&C.queued[x], 0);
        __threadfence();
    }
    __syncwarp();
    if (x >= 0) {
        s = __ldg(&C.off[x]);
        len = (int)(__ldg(&C.off[x + 1]) - s);
        e = ld_val(&C.val[x]);
    }
    int most = len;
#pragma unroll
    for (int d = 16; d >= W; d >>= 1) most = max(most, __shfl_xor_sync(ABC_FULL, most, d));
    const int nr = (most + W - 1) / W;  // the same for the warp
    int32_t y[R], v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        y[r] = -1;
        if (r < nr && r * W + gl < len) y[r] = __ldg(&C.adj[s + r * W + gl]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = y[r] >= 0 ? ld_val(&C.val[y[r]]) : -1;
    auto at_least = [&](int t) {
        int c = 0;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r < nr) c += __popc(__ballot_sync(ABC_FULL, v[r] >= t) & group);
        return c;
    };
    // of the neighbours at e or more, c < e, c are also at c or more: the new value lies in [c, e)
    const int c = at_least(e);
    const bool drops = x >= 0 && c < e;
    if (__ballot_sync(ABC_FULL, drops) == 0) return;
    int lo = drops ? c : 0, hi = drops ? e - 1 : 0;
    while (__ballot_sync(ABC_FULL, lo < hi)) {
        const int mid = lo + ((hi - lo + 1) >> 1);
        const int k = at_least(mid);
        if (lo < hi) {
            if (k >= mid) lo = mid;
            else hi = mid - 1;
        }
    }
    if (drops && gl == 0) C.val[x] = lo;
    __threadfence();
    __syncwarp();
    // neighbours above the new value may have counted this one (v was read before: it can only be too high)
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (r < nr) core_mark(C, b, nb, drops && v[r] > lo, y[r], next, count, eager);
}

// How many of the ascending entries adj[s, f) are below `bound`: every thread probes a place, which cuts the row in 257.
// Block-collective.
__device__ __forceinline__ int row_end(const CoreArgs &C, int64_t s, int64_t f, int32_t bound) {
    const int t = threadIdx.x;
    int64_t a = s, b = f;  // entries before a are below, those from b on are not
    while (b - a > CORE_THREADS) {
        const int64_t len = b - a;
        const int k = __syncthreads_count(__ldg(&C.adj[a + len * (t + 1) / (CORE_THREADS + 1)]) < bound);
        if (k < CORE_THREADS) b = a + len * (k + 1) / (CORE_THREADS + 1);
        if (k > 0) a = a + len * k / (CORE_THREADS + 1) + 1;
    }
    return (int)(a - s) + __syncthreads_count(a + t < b && __ldg(&C.adj[a + t]) < bound);
}

// Entries at or above each value, from counts of them by value: bins[k] (k < n) counts values lo + k w to lo + k w + w - 1, the last
// bin all above too. Returns the last k of which at least lo + k w entries lie in bins k and up (0 if none).
// Block-collective; ends with a barrier, s_w: a word a warp.
template <class F>
__device__ __forceinline__ int last_reached(F bin, int n, int lo, int w, int *s_best, int *s_w) {
    const int t = threadIdx.x, lane = t & 31;
    if (t == 0) *s_best = 0;
    // thread t: bins [b0, b1), above them those of the threads past it
    const int per = (n + CORE_THREADS - 1) / CORE_THREADS, b0 = min(t * per, n), b1 = min(b0 + per, n);
    int sum = 0;
    for (int k = b0; k < b1; ++k) sum += bin(k);
    int run = sum;  // this lane's and those of the lanes past it
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_down_sync(ABC_FULL, run, d);
        if (lane + d < 32) run += o;
    }
    if (lane == 0) s_w[t >> 5] = run;
    __syncthreads();
    for (int k = (t >> 5) + 1; k < CORE_WARPS; ++k) run += s_w[k];
    run -= sum;
    for (int k = b1 - 1; k >= b0; --k) {
        run += bin(k);
        if (run >= lo + k * w) {
            atomicMax(s_best, k);
            break;
        }
    }
    __syncthreads();
    const int best = *s_best;
    __syncthreads();
    return best;
}

// A long row by the whole block: up to three passes over the entries that can count, none with a barrier in it. The new
// value is searched for in the values kept in shared memory, or, with more than fit, in counts of them by value
// (a search that read such rows again for every step took k_core 310 ms of 361 with 20 rows of 2M entries).
__device__ __forceinline__ void core_long(const CoreArgs &C, int32_t x, int32_t *cache, CoreBuf &b, int &nb, int32_t *next, unsigned *count) {
    __shared__ int s_n[2];
    __shared__ int s_best, s_w[CORE_WARPS];
    const int t = threadIdx.x, lane = t & 31;
    if (t == 0) {
        atomicExch(&C.queued[x], 0);
        __threadfence();
        s_n[0] = s_n[1] = 0;
    }
    __syncthreads();
    const bool upper = x < C.nU;
    const int64_t s = __ldg(&C.off[x]), f = __ldg(&C.off[x + 1]);
    const int e = ld_val(&C.val[x]);
    constexpr int LILP = 4;
    // fn(index, value) on the row's first n entries
    auto walk = [&](int n, auto fn) {
        for (int i0 = t; i0 < n; i0 += CORE_THREADS * LILP) {
            int32_t y[LILP], v[LILP];
#pragma unroll
            for (int q = 0; q < LILP; ++q) y[q] = i0 + q * CORE_THREADS < n ? __ldg(&C.adj[s + i0 + q * CORE_THREADS]) : -1;
#pragma unroll
            for (int q = 0; q < LILP; ++q) v[q] = y[q] >= 0 ? ld_val(&C.val[y[q]]) : -1;
#pragma unroll
            for (int q = 0; q < LILP; ++q)
                if (y[q] >= 0) fn(i0 + q * CORE_THREADS, v[q]);
        }
    };
    auto total = [&](int mine, int slot) {
        mine = __reduce_add_sync(ABC_FULL, mine);
        if (lane == 0 && mine) atomicAdd(&s_n[slot], mine);
        __syncthreads();
        const int r = s_n[slot];
        if (t == 0) s_n[slot ^ 1] = 0;
        __syncthreads();
        return r;
    };
    int mine = 0;
    walk(row_end(C, s, f, id_bound(C, upper, e)), [&](int, int32_t v) { mine += v >= e ? 1 : 0; });
    const int c = total(mine, 0);
    if (c >= e) return;
    // the new value lies in [c, e), and the first n entries can count for it
    const int n = row_end(C, s, f, id_bound(C, upper, max(c, 1)));
    const bool kept = n <= CORE_CACHE;
    int lo = c, hi = e - 1;
    if (kept) {
        walk(n, [&](int i, int32_t v) { cache[i] = v; });
        __syncthreads();
        int slot = 1;
        while (lo < hi) {
            const int mid = lo + ((hi - lo + 1) >> 1);
            int k = 0;
            for (int i = t; i < n; i += CORE_THREADS) k += cache[i] >= mid ? 1 : 0;
            k = total(k, slot);
            slot ^= 1;
            if (k >= mid) lo = mid;
            else hi = mid - 1;
        }
    }
    // values from lo up, counted in steps of w: the last step k of which lo + k w entries reach that value holds the new one
    while (lo < hi) {
        const int w = (hi - lo + CORE_CACHE) / CORE_CACHE, bins = (hi - lo) / w + 1;
        for (int i = t; i < bins; i += CORE_THREADS) cache[i] = 0;
        __syncthreads();
        int top = 0;
        walk(n, [&](int, int32_t v) {
            if (v >= hi) ++top;
            else if (v >= lo) atomicAdd(&cache[(v - lo) / w], 1);
        });
        top = __reduce_add_sync(ABC_FULL, top);
        if (lane == 0 && top) atomicAdd(&cache[bins - 1], top);
        __syncthreads();
        lo += last_reached([&](int k) { return cache[k]; }, bins, lo, w, &s_best, s_w) * w;
        hi = min(hi, lo + w - 1);
    }
    if (t == 0) {
        C.val[x] = lo;
        __threadfence();
    }
    __syncthreads();
    for (int i0 = 0; i0 < n; i0 += CORE_THREADS * LILP) {
        int32_t y[LILP];
        bool in[LILP];
#pragma unroll
        for (int q = 0; q < LILP; ++q) {
            const int i = i0 + q * CORE_THREADS + t;
            y[q] = i < n ? __ldg(&C.adj[s + i]) : -1;
        }
#pragma unroll
        for (int q = 0; q < LILP; ++q) in[q] = y[q] >= 0 && (kept ? cache[i0 + q * CORE_THREADS + t] : ld_val(&C.val[y[q]])) > lo;
#pragma unroll
        for (int q = 0; q < LILP; ++q) core_mark(C, b, nb, in[q], max(y[q], 0), next, count);
    }
    __syncthreads();
}

// The rows of class 0 looked at this round, up to HUGE_BATCH at a time, by the whole grid: one block would take a row of
// 2M entries as a chain of thousands of steps, and every round waits for it (20 such rows: k_core 127 ms, so about 24). A
// batch goes through four phases with a barrier of the grid after each but the last: entries at or above each row's
// value; of rows that lack some, entries by value; the new values, a block a row; marks. No other row is looked at
// before the last phase, so the values read in the first two stand still.
struct HugeRows {
    int64_t s[HUGE_BATCH];
    int32_t x[HUGE_BATCH], pre[HUGE_BATCH + 1];  // (pre: chunks of the rows before it)
};

__device__ __forceinline__ void huge_load(const CoreArgs &C, HugeRows &H, const int32_t *rows, int n) {
    __shared__ int s_w[CORE_WARPS];
    static_assert(HUGE_BATCH == CORE_THREADS, "a thread a row");
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int nc = 0;
    __syncthreads();
    if (t < n) {
        const int32_t x = __ldcg(&rows[t]);
        const int64_t s = __ldg(&C.off[x]);
        nc = (int)((__ldg(&C.off[x + 1]) - s + HUGE_CHUNK - 1) / HUGE_CHUNK);
        H.s[t] = s;
        H.x[t] = x;
    }
    int inc = abc::warp_incl_scan(nc);
    if (lane == 31) s_w[w] = inc;
    __syncthreads();
    for (int k = 0; k < w; ++k) inc += s_w[k];
    H.pre[t + 1] = inc;
    if (t == 0) H.pre[0] = 0;
    __syncthreads();
}

// fn(row of the batch, its vertex, y[], v[]) on the entries below the row's bound, four a thread at a time (y = -1: none; the
// warp is together); before(row) says up to which id its entries can count (0: nothing is asked of it), after(row) follows each
// chunk. Block-collective.
template <class B, class F, class A>
__device__ __forceinline__ void huge_walk(const CoreArgs &C, const HugeRows &H, int n, B bound_of, F fn, A after) {
    constexpr int HILP = 4;
    const int all = H.pre[n];
    for (int k = blockIdx.x; k < all; k += gridDim.x) {
        int lo = 0, hi = n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (H.pre[mid] <= k) lo = mid;
            else hi = mid - 1;
        }
        const int32_t x = H.x[lo], bound = bound_of(lo, x);
        if (bound == 0) continue;
        const int64_t f = __ldg(&C.off[x + 1]), p0 = H.s[lo] + (int64_t)(k - H.pre[lo]) * HUGE_CHUNK, p1 = min(p0 + HUGE_CHUNK, f);
        if (__ldg(&C.adj[p0]) >= bound) continue;
        for (int64_t p = p0; p < p1; p += CORE_THREADS * HILP) {
            int32_t y[HILP], v[HILP];
#pragma unroll
            for (int q = 0; q < HILP; ++q) {
                const int64_t e = p + q * CORE_THREADS + threadIdx.x;
                y[q] = e < p1 ? __ldg(&C.adj[e]) : -1;
                if (y[q] >= bound) y[q] = -1;
            }
#pragma unroll
            for (int q = 0; q < HILP; ++q) v[q] = y[q] >= 0 ? ld_val(&C.val[y[q]]) : -1;
#pragma unroll
            for (int q = 0; q < HILP; ++q) fn(lo, x, y[q], v[q]);
        }
        after(lo, x);
    }
}

// Returns false if the grid saw an error.
__device__ __forceinline__ bool core_huge(const CoreArgs &C, HugeRows &H, const int32_t *rows, int n, int32_t *cache, CoreBuf &b, int &nb,
                                          int32_t *next, unsigned *count, unsigned long long &passed) {
    __shared__ int s_best, s_w[CORE_WARPS];
    const int t = threadIdx.x, lane = t & 31, G = gridDim.x;
    huge_load(C, H, rows, n);
    if (blockIdx.x == 0 && t < n) C.queued[H.x[t]] = 0;  // (nothing is lowered, and so nothing marked, before the next barrier)
    // entries at or above the value
    int mine = 0, e = 0;
    huge_walk(C, H, n, [&](int, int32_t x) { return id_bound(C, x < C.nU, e = ld_val(&C.val[x])); },
              [&](int, int32_t, int32_t, int32_t v) { mine += v >= e ? 1 : 0; },
              [&](int r, int32_t) {
                  mine = __reduce_add_sync(ABC_FULL, mine);
                  if (lane == 0 && mine) atomicAdd(&C.hcnt[r], mine);
                  mine = 0;
              });
    if (!core_barrier(C, passed)) return false;
    // of rows that lack some: entries by value, in steps of w over [c, e)
    auto step = [&](int c, int e) { return (e - 1 - c + CORE_CACHE) / CORE_CACHE; };
    int c = 0, w = 1;
    int held = -1;  // the row whose counts the block holds
    auto write_back = [&]() {
        if (held < 0) return;
        __syncthreads();
        for (int k = t; k < CORE_CACHE; k += CORE_THREADS)
            if (cache[k]) {
                atomicAdd(&C.hist[(int64_t)held * CORE_CACHE + k], cache[k]);
                cache[k] = 0;
            }
        held = -1;
        __syncthreads();
    };
    for (int k = t; k < CORE_CACHE; k += CORE_THREADS) cache[k] = 0;
    __syncthreads();
    huge_walk(C, H, n,
              [&](int r, int32_t x) {
                  e = ld_val(&C.val[x]);
                  c = __ldcg(&C.hcnt[r]);
                  if (c >= e) return 0;
                  w = step(c, e);
                  if (held != r) write_back();
                  held = r;
                  return id_bound(C, x < C.nU, max(c, 1));
              },
              [&](int, int32_t, int32_t, int32_t v) {
                  // (most are at the top or below it all; those at the top are counted in registers)
                  if (v >= e - 1) ++mine;
                  else if (v >= c) atomicAdd(&cache[(v - c) / w], 1);
              },
              [&](int, int32_t) {
                  mine = __reduce_add_sync(ABC_FULL, mine);
                  if (lane == 0 && mine) atomicAdd(&cache[(e - 1 - c) / w], mine);
                  mine = 0;
              });
    write_back();
    if (!core_barrier(C, passed)) return false;
    // the new values, a block a row. Where a step is several values its last one is taken, which is not too low, and the row
    // is looked at again.
    for (int r = blockIdx.x; r < n; r += G) {
        const int32_t x = H.x[r];
        e = ld_val(&C.val[x]);
        c = __ldcg(&C.hcnt[r]);
        int nv = -1;
        if (c < e) {
            w = step(c, e);
            const int bins = (e - 1 - c) / w + 1;
            int32_t *h = C.hist + (int64_t)r * CORE_CACHE;
            nv = min(e - 1, c + last_reached([&](int k) { return __ldcg(&h[k]); }, bins, c, w, &s_best, s_w) * w + w - 1);
            for (int k = t; k < bins; k += CORE_THREADS) h[k] = 0;
            if (t < 32) core_mark(C, b, nb, t == 0 && w > 1, x, next, count);
        }
        __syncthreads();
        if (t == 0) {
            if (nv >= 0) C.val[x] = nv;
            C.hval[r] = nv;
            C.hcnt[r] = 0;
        }
        __syncthreads();
    }
    if (!core_barrier(C, passed)) return false;
    // neighbours above a new value may have counted the old one
    int nv = 0;
    huge_walk(C, H, n,
              [&](int r, int32_t x) {
                  nv = __ldcg(&C.hval[r]);
                  return nv < 0 ? 0 : id_bound(C, x < C.nU, nv + 1);
              },
              [&](int, int32_t, int32_t y, int32_t v) { core_mark(C, b, nb, v > nv, max(y, 0), next, count); }, [&](int, int32_t) {});
    return true;
}

// Rounds of few short rows, by one block while the grid waits once: a round of the grid takes about 10 us (20
// when this was made), mostly its barrier and the lists, whatever it has to look at, and a change moves on by one neighbour a round, so a path of n
// vertices needs about n / 2 rounds. Here the lists stay in shared memory, with the rows' places (read while the
// mark is made), and a round is three trips to L2 and two block barriers. Rounds end when nothing is left, when a
// longer row is marked or the list is full, or after `rounds`; what is left goes to the grid's list.
struct NarrowList {
    int64_t s[NARROW_MAX];
    int32_t x[NARROW_MAX], len[NARROW_MAX];
};
static_assert(2 * sizeof(NarrowList) <= CORE_CACHE * sizeof(int32_t), "the lists lie in the cache");

__device__ __forceinline__ void core_narrow(const CoreArgs &C, const int32_t *rows, int n, int32_t *cache, int32_t *next, unsigned *count, int rounds) {
    __shared__ int s_cnt[2], s_spilt;
    NarrowList *const L = reinterpret_cast<NarrowList *>(cache);
    constexpr int W = 8, R = CORE_SMALL / W;
    const int t = threadIdx.x, lane = t & 31, gl = lane % W;
    const unsigned group = ((1u << W) - 1u) << (lane - gl);
    if (t < n) {
        const int32_t x = __ldcg(&rows[t]);
        const int64_t s = __ldg(&C.off[x]);
        L[0].x[t] = x;
        L[0].s[t] = s;
        L[0].len[t] = (int32_t)(__ldg(&C.off[x + 1]) - s);
    }
    if (t == 0) {
        s_cnt[1] = 0;
        s_spilt = 0;
    }
    __syncthreads();
    int a = 0;
    for (int round = 0; n > 0; ++round) {
        NarrowList &cur = L[a], &nxt = L[a ^ 1];
        for (int i0 = 0; i0 < n; i0 += CORE_THREADS / W) {
            const int i = i0 + t / W;
            const int32_t x = i < n ? cur.x[i] : -1;
            const int64_t s = i < n ? cur.s[i] : 0;
            const int len = i < n ? cur.len[i] : 0;
            const int e = x >= 0 ? ld_val(&C.val[x]) : 0;
            int most = len;
#pragma unroll
            for (int d = 16; d >= W; d >>= 1) most = max(most, __shfl_xor_sync(ABC_FULL, most, d));
            const int nr = (most + W - 1) / W;  // the same for the warp
            int32_t y[R], v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                y[r] = -1;
                if (r < nr && r * W + gl < len) y[r] = __ldg(&C.adj[s + r * W + gl]);
            }
            if (x >= 0 && gl == 0) C.queued[x] = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = y[r] >= 0 ? ld_val(&C.val[y[r]]) : -1;
            auto at_least = [&](int k) {
                int c = 0;
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (r < nr) c += __popc(__ballot_sync(ABC_FULL, v[r] >= k) & group);
                return c;
            };
            const int c = at_least(e);
            const bool drops = x >= 0 && c < e;
            int lo = drops ? c : 0, hi = drops ? e - 1 : 0;
            while (__ballot_sync(ABC_FULL, lo < hi)) {
                const int mid = lo + ((hi - lo + 1) >> 1);
                const int k = at_least(mid);
                if (lo < hi) {
                    if (k >= mid) lo = mid;
                    else hi = mid - 1;
                }
            }
            // (all of them have read and cleared their marks: what is lowered and marked from here on is seen by whoever is next)
            __syncthreads();
            if (drops && gl == 0) C.val[x] = lo;
            if (drops) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if (v[r] <= lo) continue;
                    const int64_t f = __ldg(&C.off[y[r]]), g = __ldg(&C.off[y[r] + 1]);
                    if (atomicExch(&C.queued[y[r]], 1) != 0) continue;
                    const int at = g - f <= CORE_SMALL ? atomicAdd(&s_cnt[a ^ 1], 1) : NARROW_MAX;
                    if (at < NARROW_MAX) {
                        nxt.x[at] = y[r];
                        nxt.s[at] = f;
                        nxt.len[at] = (int32_t)(g - f);
                    } else {
                        const int k = row_class(C, y[r]);
                        next[list_start(C, k) + atomicAdd(&count[k], 1u)] = y[r];
                        s_spilt = 1;
                    }
                }
            }
            __syncthreads();
        }
        a ^= 1;
        n = min(s_cnt[a], NARROW_MAX);
        const bool leave = s_spilt != 0 || round + 1 >= rounds;
        if (t == 0) s_cnt[a ^ 1] = 0;  // (added to after the next barrier only)
        if (leave) break;
    }
    if (t < n) next[list_start(C, CLASSES - 1) + atomicAdd(&count[CLASSES - 1], 1u)] = L[a].x[t];
    __syncthreads();
}

__global__ void __launch_bounds__(CORE_THREADS, 4) k_core(CoreArgs C) {
    __shared__ CoreBuf buf[CORE_WARPS];
    __shared__ int32_t cache[CORE_CACHE];
    __shared__ HugeRows huge;
    const int G = gridDim.x, lane = threadIdx.x & 31;
    const int64_t n = (int64_t)C.nU + C.nV;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (int64_t)G * blockDim.x;
    const int gw = (int)(t0 >> 5), nw = (int)(nt >> 5);
    CoreBuf &b = buf[threadIdx.x >> 5];
    int nb = 0;
    unsigned long long passed = 0;

    // first values: the largest h whose h-th entry has at least h edges
    for (int64_t x = t0; x < n; x += nt) {
        const bool upper = x < C.nU;
        const int64_t s = __ldg(&C.off[x]);
        int lo = 0, hi = (int)(__ldg(&C.off[x + 1]) - s);
        while (lo < hi) {
            const int h = lo + ((hi - lo + 1) >> 1);
            if (__ldg(&C.adj[s + h - 1]) < id_bound(C, upper, h)) lo = h;
            else hi = h - 1;
        }
        C.val[x] = lo;
        C.queued[x] = 1;
    }
    if (!core_barrier(C, passed)) return;
    // round 0 looks at every vertex with an edge, later rounds at the lists
    for (unsigned round = 0;; ++round) {
        const unsigned *cnt = C.count + CLASSES * (round % 3);
        unsigned *ncnt = C.count + CLASSES * ((round + 1) % 3);
        int32_t *cur = C.list[round & 1];
        int32_t *next = C.list[(round + 1) & 1];
        // a first short row per eight lanes, read along with the counts that say whether there is one
        const int64_t at0 = 4 * (int64_t)gw + lane / 8, short0 = list_start(C, CLASSES - 1), shorts = (int64_t)C.hU[CLASSES - 1] + C.hV[CLASSES - 1] - short0;
        const int32_t first = round > 0 && at0 < shorts ? __ldcg(&cur[short0 + at0]) : -1;
        int64_t num[CLASSES], sum = 0;
        for (int c = 0; c < CLASSES; ++c) {
            num[c] = round > 0 ? (int64_t)__ldcg(&cnt[c])
                               : (int64_t)(C.hU[c] - (c ? C.hU[c - 1] : 0)) + (C.hV[c] - (c ? C.hV[c - 1] : 0));
            sum += num[c];
        }
        if (sum == 0) break;
        if (t0 == 0) {  // (nothing uses this third of the counts before the round's barrier)
            unsigned *z = C.count + CLASSES * ((round + 2) % 3);
            for (int c = 0; c < CLASSES; ++c) z[c] = 0;
        }
        auto pick = [&](int c, int64_t i) -> int32_t {
            if (round > 0) return __ldcg(&cur[list_start(C, c) + i]);
            const int32_t u0 = c == 0 ? 0 : C.hU[c - 1], u1 = C.hU[c], v0 = c == 0 ? 0 : C.hV[c - 1];
            return i < u1 - u0 ? (int32_t)(u0 + i) : (int32_t)(C.nU + v0 + (i - (u1 - u0)));
        };
        if (round > 0 && sum == num[CLASSES - 1] && sum <= NARROW) {
            // (a round of it takes up to 10 us; the other blocks' wait has its limit)
            if (blockIdx.x == 0)
                core_narrow(C, cur + list_start(C, CLASSES - 1), (int)sum, cache, next, ncnt, (int)max(16ull, min(4096ull, C.timeout_ns / 20000ull)));
            if (!core_barrier(C, passed)) return;
            continue;
        }
        if (num[0] > 0) {
            if (round == 0) {  // the grid's rows come from the list
                for (int64_t i = t0; i < num[0]; i += nt) cur[i] = pick(0, i);
                if (!core_barrier(C, passed)) return;
            }
            for (int64_t i = 0; i < num[0]; i += HUGE_BATCH)
                if (!core_huge(C, huge, cur + i, (int)min((int64_t)HUGE_BATCH, num[0] - i), cache, b, nb, next, ncnt, passed)) return;
        }
        for (int64_t i = blockIdx.x; i < num[1]; i += G) core_long(C, pick(1, i), cache, b, nb, next, ncnt);
        for (int64_t i = gw; i < num[2]; i += nw) core_rows<32, CORE_MID / 32>(C, pick(2, i), b, nb, next, ncnt, sum <= EAGER);
        for (int64_t i = 4 * (int64_t)gw; i < num[3]; i += 4 * (int64_t)nw) {
            const int64_t k = i + lane / 8;
            core_rows<8, CORE_SMALL / 8>(C, k >= num[3] ? -1 : round > 0 && k == at0 ? first : pick(3, k), b, nb, next, ncnt, sum <= EAGER);
        }
        core_flush(C, b, nb, next, ncnt);
        if (!core_barrier(C, passed)) return;
    }
}

// Core numbers in the caller's order, and the largest.
__global__ void __launch_bounds__(256) k_core_by_caller(const int32_t *core, const int32_t *new2old, int32_t nU, int64_t n, int32_t *out,
                                                        int *largest) {
    __shared__ int s_max;
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    int mx = 0;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = core[x];
        out[__ldg(&new2old[x]) + (x >= nU ? nU : 0)] = c;
        mx = max(mx, c);
    }
    mx = __reduce_max_sync(ABC_FULL, mx);
    if ((threadIdx.x & 31) == 0 && mx) atomicMax(&s_max, mx);
    __syncthreads();
    if (threadIdx.x == 0 && s_max) atomicMax(largest, s_max);
}

// per layer: hist[t] = vertices with core number t. Each block counts in shared memory where both layers' counters fit
// (`held`); a few hundred counters take every vertex's atomic (1.5M vertices: 0.30 ms straight to L2).
__global__ void __launch_bounds__(256) k_core_hist(const int32_t *core_caller, int32_t nU, int64_t n, int32_t maxcore, int held,
                                                   unsigned long long *hist) {
    extern __shared__ unsigned s_hist[];
    const int size = 2 * (maxcore + 1);
    if (held)
        for (int i = threadIdx.x; i < size; i += blockDim.x) s_hist[i] = 0;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = min(core_caller[i], maxcore) + (i < nU ? 0 : maxcore + 1);
        if (held) atomicAdd(&s_hist[c], 1u);
        else atomicAdd(&hist[c], 1ull);
    }
    __syncthreads();
    if (held)
        for (int i = threadIdx.x; i < size; i += blockDim.x)
            if (s_hist[i]) atomicAdd(&hist[i], (unsigned long long)s_hist[i]);
}

}  // namespace

void free_pruning(abcore_ctx *ctx) {
    Pruning &p = ctx->pr;
    free_graph_of(ctx, p.gc);
    ctx->release(p.core_caller);
    p.coreU_ge.clear();
    p.coreV_ge.clear();
    p.maxcore = 0;
    p.ready = false;
}

// Core numbers of the loaded graph into core_caller (unified caller ids).
static int core_decompose(abcore_ctx *ctx, int32_t *core_caller, int32_t *maxcore_out) {
    const Graph &g = ctx->g;
    const int64_t n = std::max<int64_t>(g.n(), 1);
    ABC_TRY(peel_finish(ctx));
    ABC_TRY(peel_prepare(ctx));  // (for the queries this is the preprocessing of)
    constexpr size_t BAR_WORD = (3 * CLASSES + 1 + 31) / 32 * 32, SMALL_WORDS = BAR_WORD + 2, HUGE_WORDS = (size_t)HUGE_BATCH * (2 + CORE_CACHE);
    int32_t *words = nullptr, *tables = nullptr, *huge = nullptr;
    unsigned *small = nullptr;
    PeelCtl *ctl = nullptr;
    int rc = ABCORE_OK;
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_core, CORE_THREADS, 0);
    const int grid = std::max(per_sm, 1) * ctx->num_sms;
    const int32_t maxdeg = std::max(g.maxdegU, g.maxdegV);
    // degree tables padded to maxdeg + 2 entries on both layers
    const size_t nt = (size_t)maxdeg + 2;
    std::vector<int32_t> h(2 * nt, 0);
    for (size_t t = 0; t < nt; ++t) {
        h[t] = (int32_t)cnt_ge(g.cntU_ge, (int32_t)t);
        h[nt + t] = (int32_t)cnt_ge(g.cntV_ge, (int32_t)t);
    }
#define STEP(x)            \
    do {                   \
        rc = (x);          \
        if (rc) goto done; \
    } while (0)
    STEP(ctx->alloc(&words, (size_t)(4 * n), "core values"));  // values, marks, two lists
    STEP(ctx->alloc(&tables, 2 * nt, "degree tables"));
    STEP(ctx->alloc(&small, SMALL_WORDS, "core counters"));    // list lengths, largest core number, barrier
    if (maxdeg > CORE_LONG) STEP(ctx->alloc(&huge, HUGE_WORDS, "core value counts"));
    STEP(ctx->alloc(&ctl, 1, "core control"));
    {
        CoreArgs C{};
        C.off = g.off;
        C.adj = g.adj;
        C.nU = g.nU;
        C.nV = g.nV;
        const int32_t cut[CLASSES] = {CORE_LONG + 1, CORE_MID + 1, CORE_SMALL + 1, 1};
        for (int k = 0; k < CLASSES; ++k) {
            C.hU[k] = (int32_t)cnt_ge(g.cntU_ge, cut[k]);
            C.hV[k] = (int32_t)cnt_ge(g.cntV_ge, cut[k]);
        }
        C.hcnt = huge;
        C.hval = huge + HUGE_BATCH;
        C.hist = huge + 2 * HUGE_BATCH;
        C.gU = tables;
        C.gV = tables + nt;
        C.maxdeg = maxdeg;
        C.val = words;
        C.queued = words + n;
        C.list[0] = words + 2 * n;
        C.list[1] = words + 3 * n;
        C.count = small;
        C.ctl = ctl;
        C.bar = reinterpret_cast<unsigned long long *>(small + BAR_WORD);
        C.timeout_ns = (unsigned long long)ctx->prm.timeout_ms * 1000000ull;
        void *args[] = {&C};
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(CORE_THREADS);
        cfg.stream = ctx->stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const unsigned gi = (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)ctx->num_sms * 8);
        int err = 0, largest = 0;
        cudaError_t e = cudaMemcpyAsync(tables, h.data(), sizeof(int32_t) * h.size(), cudaMemcpyHostToDevice, ctx->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(small, 0, SMALL_WORDS * sizeof(unsigned), ctx->stream);
        if (e == cudaSuccess && huge) e = cudaMemsetAsync(huge, 0, HUGE_WORDS * sizeof(int32_t), ctx->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(ctl, 0, sizeof(PeelCtl), ctx->stream);
        if (e == cudaSuccess) e = cudaLaunchKernelExC(&cfg, (const void *)k_core, args);
        if (e == cudaSuccess) {
            ctx->stats.launches++;
            k_core_by_caller<<<gi, 256, 0, ctx->stream>>>(C.val, g.new2old, g.nU, g.n(), core_caller, (int *)small + 3 * CLASSES);
            e = cudaMemcpyAsync(&err, &ctl->err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream);
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(&largest, small + 3 * CLASSES, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) STEP(ctx->cuda_fail(e, "core decomposition"));
        if (err) STEP(ctx->fail(err, "core decomposition: device error %d", err));
        *maxcore_out = largest;
    }
done:
    cudaStreamSynchronize(ctx->stream);
    ctx->release(words);
    ctx->release(tables);
    ctx->release(small);
    ctx->release(huge);
    ctx->release(ctl);
    return rc;
#undef STEP
}

int prepare_pruning(abcore_ctx *ctx) {
    Pruning &p = ctx->pr;
    if (p.ready) return ABCORE_OK;
    free_pruning(ctx);
    const Graph &g = ctx->g;
    const int64_t n = g.n();
    const auto t0 = std::chrono::steady_clock::now();
    ABC_TRY(ctx->alloc(&p.core_caller, (size_t)std::max<int64_t>(n, 1), "core numbers"));
    int32_t maxcore = 0;
    int rc = core_decompose(ctx, p.core_caller, &maxcore);
    if (rc) {
        free_pruning(ctx);
        return rc;
    }
    const auto t1 = std::chrono::steady_clock::now();
    // per-layer tables: vertices with core >= t
    unsigned long long *hist = nullptr;
    rc = ctx->alloc(&hist, 2 * ((size_t)maxcore + 1), "core histogram");
    if (!rc) {
        std::vector<int64_t> h(2 * ((size_t)maxcore + 1), 0);
        cudaMemsetAsync(hist, 0, sizeof(int64_t) * h.size(), ctx->stream);
        const unsigned gi = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)ctx->num_sms * 16));
        const size_t smem = 2 * ((size_t)maxcore + 1) * sizeof(unsigned);
        const int held = smem <= 48 * 1024;
        if (n > 0) k_core_hist<<<std::min(gi, (unsigned)ctx->num_sms * 4), 256, held ? smem : 0, ctx->stream>>>(p.core_caller, g.nU, n, maxcore, held, hist);
        cudaMemcpyAsync(h.data(), hist, sizeof(int64_t) * h.size(), cudaMemcpyDeviceToHost, ctx->stream);
        const cudaError_t e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) rc = ctx->cuda_fail(e, "core histogram");
        p.coreU_ge.assign((size_t)maxcore + 2, 0);
        p.coreV_ge.assign((size_t)maxcore + 2, 0);
        for (int32_t t = maxcore; t >= 0; --t) {
            p.coreU_ge[t] = p.coreU_ge[t + 1] + h[t];
            p.coreV_ge[t] = p.coreV_ge[t + 1] + h[maxcore + 1 + t];
        }
    }
    ctx->release(hist);
    // the graph again, each layer numbered by non-increasing core number
    int32_t *eu = nullptr, *ev = nullptr;
    if (!rc) rc = ctx->alloc(&eu, (size_t)std::max<int64_t>(g.m, 1), "core layout edges");
    if (!rc) rc = ctx->alloc(&ev, (size_t)std::max<int64_t>(g.m, 1), "core layout edges");
    if (!rc) rc = csr_edges(ctx, g, eu, ev);
    if (!rc) rc = build_graph(ctx, p.gc, g.nU, g.nV, g.m, eu, ev, p.core_caller, maxcore);
    ctx->release(eu);
    ctx->release(ev);
    if (rc) {
        free_pruning(ctx);
        return rc;
    }
    const auto t2 = std::chrono::steady_clock::now();
    p.maxcore = maxcore;
    p.decomp_ms = std::chrono::duration<float, std::milli>(t1 - t0).count();
    p.layout_ms = std::chrono::duration<float, std::milli>(t2 - t1).count();
    p.ready = true;
    return ABCORE_OK;
}
