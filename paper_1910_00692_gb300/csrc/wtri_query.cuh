// Shared device machinery of the top-k query, the edge sampler and the
// batched form (included by wtri_topk.cu, wtri_batch.cu, wtri_wedge.cu and
// wtri_clique.cu).
//
// Exact top-k weighted triangles: heavy-first enumeration with a running
// threshold.
//
// Method (the exactness argument of Algorithm 2 and Section 3.2, re-derived
// for a parallel schedule):
//  * Edges are visited in the edge order (weight desc, input index asc); r is
//    an edge's position.  Each triangle is owned by its first edge in that
//    order, so edge r owns triangle {x, y, c} iff both (x,c) and (y,c) come
//    after r.  Every triangle is enumerated exactly once.
//  * Every triangle owned by r has all edge weights <= w_r, and m_p is
//    monotone in each argument with m_p <= max, so its key is at most
//    K(w_r, w_r, w_r).  Once that bound is below the threshold tau, no later
//    edge can contribute: the sweep stops.  This is the paper's heavy-first
//    threshold argument with one monotone cursor in place of two pointers.
//  * Per edge, the entries of x and y after r are suffixes of their
//    weight-sorted lists; their first entries bound the other two weights
//    (edge bound), and the wedge bound K(w_r, w_xc, max_y) only decreases
//    along x's suffix, so the wedges that can reach tau are a prefix of it,
//    the live range, found by search.  The shorter of the two live ranges is
//    scanned; the closing edge (y, c) is found by search in the oriented
//    (degree-ordered) lists.
//  * tau is the key of the k-th best of k distinct triangles found so far, a
//    valid lower bound on the true k-th key; pruning is strict (< tau), so
//    triangles tied with the k-th key are still enumerated and the triple
//    tie-break decides them.
//
// Schedule: one kernel runs the whole sweep.  Its threads form a team: every
// block of a cooperative launch (one block per SM, a grid barrier between
// phases), or one block alone (the batched form, many small graphs at once).
// The edge order is processed in rounds of geometrically growing ranges, each
// in three phases with a team barrier after each:
//   A  edges: the checks and searches of every edge of the round (a warp per
//      edge in small rounds, a thread per edge in large ones); an edge with
//      a long live range leaves it as an item, with the running number of
//      wedges before it (rounds of more edges than items, once the threshold
//      hardly moves: most live ranges are scanned by their warp);
//   B  wedges: the items' wedges, numbered through, are dealt to the team 32
//      at a time, whatever the items' lengths;
//   C  select (one block): the k-th key, in-place compaction, the new tau,
//      and the next round's range, cut where the edge bound falls below tau.
// After the last round the same kernel ranks the k best and writes the
// outputs.  What bounds a query is latency (binary searches over a pruned
// set) and the launches: with a launch per phase a query on the 2e7-edge
// graph spent about 75 of its 330 us in the launches of rounds after the
// stop, 104 us on the 64 items of the first round (one block each), and 75 us
// on selects whose histogram one thread scanned.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "wtri_internal.cuh"

namespace wtri {
namespace {

constexpr int TGRID = 1024;         // threads of a block of the grid team (one block per SM)
constexpr int SORT_MAX = 2048;      // most candidates sorted in shared memory
constexpr uint32_t WAIT_LIMIT = 1u << 26;  // bounded polling of the grid barrier
constexpr int64_t ITEM_CAP = 1 << 18;      // most items
// Largest round that takes a warp per edge (512, 4,096 or 32,768: the same to 1 %
// at p = 1 and +inf on graphs of 5e6 to 6e7 edges).
constexpr int64_t WARP_EDGES = 4096;
// Largest p = -inf round that numbers its entries through (2e7 skewed edges, us at
// 1,024 / 8,192 / 65,536: 381 / 357 / 369; 6e7 edges: 784 / 731 / 732).
constexpr int64_t MIN_FLAT = 8192;
constexpr int64_t SMALL_M = 1 << 16;       // edges of a small graph (see sweep_blocks)

// State of one query (zeroed before it starts).
struct QState {
    unsigned long long tau;       // keys below tau are pruned; 0 = no bound yet
    uint32_t err;                 // DEV_ERR_* bits
    uint32_t count;               // candidates appended (may exceed capacity)
    uint32_t selected;            // count right after the last compaction
    uint32_t bar;                 // arrivals at the grid barrier
    unsigned long long items[2];  // items of a phase (high 20 bits) and their wedges, by step parity
    long long lo, hi, size;       // the next round and its uncut size (published by the selecting block)
    uint32_t kept;                // candidates left for the ranking
    uint32_t pad;
};

// The wedges of one edge left to phase B.
struct __align__(16) Item {
    int32_t r;      // owning edge (position in the edge order)
    int32_t x, y;   // scanned endpoint, probed endpoint (p = -inf: the edge's endpoints)
    uint32_t w;     // w_r
    int64_t j0;     // first wedge's position in x's list (p = -inf: in the scanned oriented row)
    int64_t lb;     // y's oriented row (p = -inf: the searched row)
    int32_t ln;     // its length
    int32_t dy;     // y's degree
    int32_t pad[2];
};

struct Query {
    QState* st;
    unsigned long long* ckey;
    int4* ctri;
    uint32_t cap;
    Item* items;                // item_cap items
    unsigned long long* ibase;  // wedges before each item
    int64_t item_cap;
    int32_t k;
    // Sweep: edges (or drawn positions: *total_dev of them, known on the
    // device only), first round, growth.
    int64_t total;
    const int64_t* total_dev;
    int64_t first;
    int32_t growth;
    // Sampled mode (edge sampling): bitmap of drawn edges by edge-order
    // position, and the drawn positions in ascending order.
    const uint32_t* smark;
    const int32_t* slist;
    // Sharding (multi-GPU split of one query): this query owns the edges
    // whose chunk (position >> SHARD_SHIFT) is congruent to shard modulo
    // nshards; nshards <= 1 means every edge.
    int32_t shard;
    int32_t nshards;
    // Wedges an edge's warp scans itself before leaving them to phase B
    // (rounded up to a multiple of 32).
    int32_t t_short;
    // Instrumented run: bytes of the adjacency loads are added here (null:
    // no counting).
    unsigned long long* qbytes;
    // The value of p for P_GEN queries.
    double gp;
    // Weights are positive fp32 bit patterns (a float-weight graph), not
    // integers: the means and reported values read them as floats.
    int32_t fw;
    // Polls of the first grid-barrier wait and of every later one (WAIT_LIMIT
    // in production; tests lower them to take the timeout paths).
    uint32_t wait_first;
    uint32_t wait_later;
};

// Where a query's results go.
struct Out {
    wtri_tri* tri;
    double* w;
    int32_t* count;
    unsigned long long* key;  // may be null
};

// Bytes of adjacency loads issued by one thread (instrumented runs only).
struct Tally {
    unsigned long long n = 0;
    bool on = false;
    __device__ __forceinline__ void add(uint32_t b) {
        if (on) n += b;
    }
};

// Adds every lane's tally to the query's counter (one atomic per warp).
__device__ __forceinline__ void flush_tally(const Query& q, const Tally& t) {
    if (!q.qbytes) return;
    unsigned long long v = t.n;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(q.qbytes, v);
}

constexpr int SHARD_SHIFT = 10;  // 1024-edge chunks of the edge order, dealt round-robin

__device__ __forceinline__ bool drawn(const Query& q, int32_t r) {
    return (__ldg(q.smark + (r >> 5)) >> (r & 31)) & 1u;
}

// Ownership.  Exact mode: a triangle belongs to its first edge in the edge
// order, so the edge at position r owns (x, y, c) iff both other edges come
// later.  Sampled mode (Algorithm 3's set T): a triangle belongs to its
// first DRAWN edge, so each triangle with a drawn edge is reported once.
template <bool SAMPLED>
__device__ __forceinline__ bool owns(const Query& q, int32_t r, int32_t rxc, int32_t ryc) {
    if (!SAMPLED) return rxc > r && ryc > r;
    return !(rxc < r && drawn(q, rxc)) && !(ryc < r && drawn(q, ryc));
}

// m_p of Eq. 1 in fp64 for a finite p outside {0, 1, 2}: the weights in
// ascending order (equal multisets give equal bits), scaled by the largest
// (p > 0) or the smallest (p < 0) so that no power overflows:
//   m_p = s * (((a/s)^p + (b/s)^p + (c/s)^p) / 3)^(1/p).
__device__ __noinline__ double general_mean(double p, uint32_t a, uint32_t b, uint32_t c, bool fw = false) {
    uint32_t t;
    if (a > b) { t = a; a = b; b = t; }
    if (b > c) { t = b; b = c; c = t; }
    if (a > b) { t = a; a = b; b = t; }
    // positive fp32 bit patterns order like their values, so the sort holds
    const double x = fw ? (double)__uint_as_float(a) : (double)a;
    const double y = fw ? (double)__uint_as_float(b) : (double)b;
    const double z = fw ? (double)__uint_as_float(c) : (double)c;
    if (p == 0.0) return cbrt(x * y * z);  // the geometric mean (real weights only)
    const double s = p > 0 ? z : x;
    const double m = (pow(x / s, p) + pow(y / s, p) + pow(z / s, p)) / 3.0;
    return s * pow(m, 1.0 / p);
}

// Ranking key of a triangle with edge weights a, b, c: exact integers for
// p in {-inf, 0, 1, 2, +inf}; the mean's fp64 bit pattern for P_GEN.
template <int P>
__device__ __forceinline__ unsigned long long keyof(uint32_t a, uint32_t b, uint32_t c,
                                                    double gp = 0.0, bool fw = false) {
    if (P == P_ONE) return (unsigned long long)a + b + c;
    if (P == P_TWO)
        return (unsigned long long)a * a + (unsigned long long)b * b + (unsigned long long)c * c;
    if (P == P_MAX) return (unsigned long long)max(a, max(b, c));
    if (P == P_GEO) return (unsigned long long)a * b * c;  // weights < 2^21: below 2^63
    if (P == P_GEN) return (unsigned long long)__double_as_longlong(general_mean(gp, a, b, c, fw));
    return (unsigned long long)min(a, min(b, c));
}

// Upper bound used for pruning: the key itself for the exact keys; for
// P_GEN the mean raised by a relative 1e-12, far above fp64 rounding, so
// that a bound computed for larger weights is never below a key computed
// for smaller ones.
template <int P>
__device__ __forceinline__ unsigned long long boundof(uint32_t a, uint32_t b, uint32_t c,
                                                      double gp = 0.0, bool fw = false) {
    if (P == P_GEN)
        return (unsigned long long)__double_as_longlong(general_mean(gp, a, b, c, fw) * (1.0 + 1e-12));
    return keyof<P>(a, b, c);
}

__device__ __forceinline__ void sort3(int32_t& a, int32_t& b, int32_t& c) {
    int32_t t;
    if (a > b) { t = a; a = b; b = t; }
    if (b > c) { t = b; b = c; c = t; }
    if (a > b) { t = a; a = b; b = t; }
}

__device__ __forceinline__ unsigned long long ld_volatile_u64(const unsigned long long* p) {
    return *(volatile const unsigned long long*)p;
}

// Closing edge (y, c) in the oriented lists: stored once, at the endpoint of
// lower (degree, id) rank, rows ascending by id (row s at
// [orowptr[s], orowptr[s+1])).  y_owns: whether y is that endpoint.
__device__ __forceinline__ bool y_owns(const DevGraph& G, int32_t y, int64_t dy, int32_t c, Tally& tb) {
    const int64_t dc = __ldg(G.rowptr + c + 1) - __ldg(G.rowptr + c);
    tb.add(16);
    return dy < dc || (dy == dc && y < c);
}

// Searches oriented row s for t.
__device__ __forceinline__ bool search_oriented(const DevGraph& G, int32_t s, int32_t t, int32_t& wst,
                                                int32_t& rst, Tally& tb) {
    int64_t lo = __ldg(G.orowptr + s), hi = __ldg(G.orowptr + s + 1);
    const int64_t end = hi;
    tb.add(16);
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        tb.add(4);
        if (__ldg(G.ocol + mid) < t) lo = mid + 1;
        else hi = mid;
    }
    if (lo < end) tb.add(4);
    if (lo < end && __ldg(G.ocol + lo) == t) {
        wst = __ldg(G.owt + lo);
        rst = __ldg(G.ork + lo);
        tb.add(8);
        return true;
    }
    return false;
}

__device__ __forceinline__ bool probe_oriented(const DevGraph& G, int32_t y, int64_t dy, int32_t c,
                                               int32_t& wyc, int32_t& ryc, Tally& tb) {
    return y_owns(G, y, dy, c, tb) ? search_oriented(G, y, c, wyc, ryc, tb)
                                   : search_oriented(G, c, y, wyc, ryc, tb);
}

// ---------------------------------------------------------------------------
// Pruning against tau along a list of non-increasing weights: fails(x) only
// if no triangle with weights w, y and x (or less) reaches tau.
//
// The exact keys compare the bound itself.  For P_GEN (other finite p, and
// real weights) the fp64 mean costs four pow per wedge on a chip whose fp64
// rate is a sixty-fourth of its fp32 rate, so the smallest weight that can
// reach tau is found once per edge in fp32 instead: with t = tau (1 - 1e-4)
// and R = 3 - (w/t)^p - (y/t)^p, the mean reaches t iff (x/t)^p >= R (p > 0)
// or <= R (p < 0), i.e. x >= t R^(1/p) (p = 0: x >= t / ((w/t) (y/t))).  The
// 1e-4 leaves R a slack of 3e-4 |p| while fp32 rounding moves it by less than
// 4e-6 (1 + |p|) wherever R > 0, so for |p| >= 0.05 a weight is only pruned
// when the exact bound prunes it too; smaller |p| keeps the fp64 bound.  All of
// it holds in fp32's normal range only, which real weights may leave (they
// reach down to 2^-149): t, both quotients and the power must lie well inside,
// else the fp64 bound decides (a power below 2^-120: no bound; x itself may be
// subnormal, as rounding to the weights' own grid passes none of them).
// Survivors are decided by their fp64 key.
// ---------------------------------------------------------------------------
template <int P>
struct Line {
    unsigned long long tau;
    uint32_t w, y;
    double gp;
    bool fw;
    bool use_cut;
    uint32_t cut;

    __device__ __forceinline__ Line(const Query& q, unsigned long long tau_, uint32_t w_, uint32_t y_)
        : tau(tau_), w(w_), y(y_), gp(q.gp), fw(q.fw != 0), use_cut(false), cut(0) {
        if constexpr (P == P_GEN) {
            const float p = (float)gp;
            if (tau == 0 || !((fabsf(p) >= 0.05f && fabsf(p) <= 1000.0f) || p == 0.0f)) return;
            const float t = (float)__longlong_as_double((long long)tau) * (1.0f - 1e-4f);
            const float a = (fw ? __uint_as_float(w) : (float)w) / t, b = (fw ? __uint_as_float(y) : (float)y) / t;
            auto inside = [](float x) { return x >= 0x1p-100f && x <= 0x1p100f; };
            if (!inside(t) || !inside(a) || !inside(b)) return;
            float e;  // log2 of the smallest x / t
            if (p == 0.0f) {
                e = -log2f(a) - log2f(b);
            } else {
                const float R = 3.0f - exp2f(p * log2f(a)) - exp2f(p * log2f(b));
                use_cut = !(R > 0.0f);  // w and y alone reach t (p > 0), or keep any x from it
                if (use_cut) {
                    cut = p > 0.0f ? 0u : 0xffffffffu;
                    return;
                }
                e = log2f(R) / p;
            }
            if (!(e <= 120.0f)) return;
            use_cut = true;
            if (e < -120.0f) return;  // cut = 0
            const float x = t * exp2f(e) * (1.0f - 1e-6f);
            if (fw) cut = __float_as_uint(x);
            else cut = x >= 4294967040.0f ? 0xffffffffu : (uint32_t)x;
        }
    }
    __device__ __forceinline__ bool fails(uint32_t x) const {
        if (P == P_GEN && tau == 0) return false;
        if (P == P_GEN && use_cut) return x < cut;
        return boundof<P>(w, x, y, gp, fw) < tau;
    }
};

// Whether every triangle of edges no heavier than w is below tau.
template <int P>
__device__ __forceinline__ bool edge_below(const Query& q, uint32_t w, unsigned long long tau) {
    if (P == P_GEN) {
        const double x = q.fw ? (double)__uint_as_float(w) : (double)w;
        return (unsigned long long)__double_as_longlong(x * (1.0 + 1e-12)) < tau;
    }
    return boundof<P>(w, w, w) < tau;
}

__device__ __forceinline__ uint32_t lanemask_below() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// First position of [lo, hi) where `below` is false (true on a prefix), found
// by groups of W lanes (16 or 32), each group with its own range and
// predicate: W probes a step, so a list of 35,000 takes four dependent loads
// instead of fifteen.  All 32 lanes call it.
template <int W, class Pred>
__device__ __forceinline__ int64_t group_search(int64_t lo, int64_t hi, const Pred& below) {
    const int lane = threadIdx.x & 31, gl = lane & (W - 1), sh = lane & ~(W - 1);
    const uint32_t gm = W == 32 ? 0xffffffffu : ((1u << W) - 1u);
    for (;;) {
        const int64_t n = hi - lo;
        if (__all_sync(0xffffffffu, n <= 0)) break;
        const int64_t step = (n + W) / (W + 1);
        const int64_t pos = lo + (int64_t)(gl + 1) * step - 1;
        const bool b = n > 0 && pos < hi && below(pos);
        const int cnt = __popc((__ballot_sync(0xffffffffu, b) >> sh) & gm);
        if (n > 0) {
            const int64_t nlo = lo + cnt * step;
            if (cnt < W) hi = min(hi, lo + (int64_t)(cnt + 1) * step - 1);
            lo = nlo;
        }
    }
    return lo;
}

// First position of the oriented ids [lo, lo + n) not below t (three probes a
// step: half the dependent loads of a binary search).
__device__ __forceinline__ int64_t search_ids(const int32_t* __restrict__ ids, int64_t lo, int32_t n, int32_t t,
                                              Tally& tb) {
    while (n > 4) {
        const int32_t s = n >> 2;
        const int32_t a = __ldg(ids + lo + s), b = __ldg(ids + lo + 2 * s), c = __ldg(ids + lo + 3 * s);
        tb.add(12);
        if (b < t) {
            if (c < t) {
                lo += 3 * s + 1;
                n -= 3 * s + 1;
            } else {
                lo += 2 * s + 1;
                n = s - 1;
            }
        } else if (a < t) {
            lo += s + 1;
            n = s - 1;
        } else {
            n = s;
        }
    }
    while (n > 0) {
        const int32_t s = n >> 1;
        tb.add(4);
        if (__ldg(ids + lo + s) < t) {
            lo += s + 1;
            n -= s + 1;
        } else {
            n = s;
        }
    }
    return lo;
}

// Appends a candidate: the active lanes take one atomic together.
__device__ __forceinline__ void append(const Query& q, unsigned long long key, int32_t a, int32_t b, int32_t c) {
    const uint32_t active = __activemask();
    const int lane = threadIdx.x & 31, leader = __ffs(active) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(&q.st->count, (uint32_t)__popc(active));
    base = __shfl_sync(active, base, leader);
    const uint32_t idx = base + __popc(active & ((1u << lane) - 1u));
    if (idx < q.cap) {
        q.ckey[idx] = key;
        q.ctri[idx] = make_int4(a, b, c, 0);
    } else {
        atomicOr(&q.st->err, DEV_ERR_OVERFLOW);
    }
}

// ---------------------------------------------------------------------------
// Teams.  sync() is a barrier of the whole team; false: give up (a grid
// barrier whose bounded wait ran out for good).
// ---------------------------------------------------------------------------
// TB threads of a block that work through the one-block phases together:
// the whole block, or one of its parts of TB threads (each with a named
// barrier of its own).
template <int TB>
struct Part {
    __device__ __forceinline__ int tid() const { return (int)(threadIdx.x % TB); }
    __device__ __forceinline__ void sync() const {
        asm volatile("barrier.cta.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x / TB)), "n"(TB) : "memory");
    }
};

template <int TB_>
struct BlockTeam {
    static constexpr int TB = TB_;
    static constexpr bool GRID = false;
    Part<TB_> part;
    __device__ __forceinline__ int64_t thread() const { return part.tid(); }
    __device__ __forceinline__ int64_t threads() const { return TB; }
    __device__ __forceinline__ int64_t warp() const { return part.tid() >> 5; }
    __device__ __forceinline__ int64_t warps() const { return TB / 32; }
    __device__ __forceinline__ int64_t block() const { return 0; }
    __device__ __forceinline__ int64_t blocks() const { return 1; }
    __device__ __forceinline__ bool leader() const { return true; }
    __device__ __forceinline__ bool sync(const Query&) {
        part.sync();
        return true;
    }
};

// nblk blocks of a cooperative launch (all resident), from block blk0 on.  A
// barrier: every block's
// first thread arrives at a counter in the query's state and polls it up to
// a limit.  The first limit is the query's wait_first; when it runs out the
// query is marked timed out and the block waits on with the full limit
// (wait_later), so that the blocks stay in step; only when that runs out too
// does it leave.  From then on no barrier of the team can complete.
template <int TB_>
struct GridTeam {
    static constexpr int TB = TB_;
    static constexpr bool GRID = true;
    Part<TB_> part;
    uint32_t target = 0;
    uint32_t limit;
    uint32_t blk0, nblk;
    int* gone;  // shared
    __device__ __forceinline__ int64_t thread() const { return (int64_t)(blockIdx.x - blk0) * TB + threadIdx.x; }
    __device__ __forceinline__ int64_t threads() const { return (int64_t)nblk * TB; }
    __device__ __forceinline__ int64_t warp() const { return thread() >> 5; }
    __device__ __forceinline__ int64_t warps() const { return threads() >> 5; }
    __device__ __forceinline__ int64_t block() const { return blockIdx.x - blk0; }
    __device__ __forceinline__ int64_t blocks() const { return nblk; }
    __device__ __forceinline__ bool leader() const { return blockIdx.x == blk0; }
    __device__ __forceinline__ uint32_t arrivals(const Query& q) const {
        uint32_t v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&q.st->bar) : "memory");
        return v;
    }
    __device__ __forceinline__ bool sync(const Query& q) {
        target += nblk;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&q.st->bar, 1u);
            bool there = false;
            for (uint32_t i = 0; i < limit && !there; i++) there = (int32_t)(arrivals(q) - target) >= 0;
            if (!there) {
                atomicOr(&q.st->err, DEV_ERR_TIMEOUT);
                for (uint32_t i = 0; i < q.wait_later && !there; i++) there = (int32_t)(arrivals(q) - target) >= 0;
            }
            limit = q.wait_later;
            if (!there) *gone = 1;
            __threadfence();
        }
        __syncthreads();
        return *gone == 0;
    }
};

// ---------------------------------------------------------------------------
// Items.
// ---------------------------------------------------------------------------
constexpr int ITEM_SHIFT = 44;  // item count above (20 bits), wedge count below
static_assert(ITEM_CAP + (1 << 18) < (1 << (64 - ITEM_SHIFT)), "the items and 32 more per warp are counted in 20 bits");
constexpr unsigned long long WEDGE_MASK = (1ull << ITEM_SHIFT) - 1;

__device__ __forceinline__ void put_item(const Query& q, uint32_t slot, unsigned long long base, const Item& it) {
    if (slot >= (uint32_t)q.item_cap) {
        atomicOr(&q.st->err, DEV_ERR_INTERNAL);
        return;
    }
    q.items[slot] = it;
    q.ibase[slot] = base;
}

// Every lane of a warp: the lanes with len > 0 leave their item.  (For rounds of
// fewer edges than there are items.)
__device__ __forceinline__ void push_items(const Query& q, int par, int64_t len, const Item& it) {
    const int lane = threadIdx.x & 31;
    const uint32_t has = __ballot_sync(0xffffffffu, len > 0);
    if (!has) return;
    unsigned long long inc = len > 0 ? (unsigned long long)len : 0ull;
    const unsigned long long mine = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    unsigned long long old = 0;
    if (lane == 31) old = atomicAdd(&q.st->items[par], ((unsigned long long)__popc(has) << ITEM_SHIFT) + inc);
    old = __shfl_sync(0xffffffffu, old, 31);
    if (len > 0)
        put_item(q, (uint32_t)(old >> ITEM_SHIFT) + __popc(has & lanemask_below()), (old & WEDGE_MASK) + inc - mine,
                 it);
}

// Rounds of more edges than items: only live ranges above FLAT_SHORT are left
// to phase B, while there is room, the others are scanned by their warp (see
// scan_here).  The last slot stays free: whoever draws it leaves the wedges
// before it there, the total of the items that were kept.  True: left.
//
// Such rounds are for sweeps that visit most of a graph.  Rounds cut to the
// items' number, 2e8 edges at random on 5e7 vertices (86 triangles, k = 1,000)
// took 764 rounds and 141 ms at p = 1, with the 46,592 items of the fixed
// scratch 289; now 100 either way.  16, 64 or 256 as the limit: the same
// there; on rows of 200 entries a shard takes 1.74, 1.62 and 2.83 ms.
constexpr int64_t FLAT_SHORT = 64;

__device__ __forceinline__ bool push_long(const Query& q, int par, int64_t len, const Item& it) {
    const int lane = threadIdx.x & 31;
    const bool lng = len > FLAT_SHORT;
    const uint32_t has = __ballot_sync(0xffffffffu, lng);
    if (!has) return false;
    const uint32_t usable = (uint32_t)q.item_cap - 1;
    unsigned long long old = 0;
    if (lane == 0) old = ld_volatile_u64(&q.st->items[par]);
    old = __shfl_sync(0xffffffffu, old, 0);
    if ((uint32_t)(old >> ITEM_SHIFT) >= usable) return false;  // (a warp adds at most 32 past it: 20 bits hold the count)
    unsigned long long inc = lng ? (unsigned long long)len : 0ull;
    const unsigned long long mine = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) old = atomicAdd(&q.st->items[par], ((unsigned long long)__popc(has) << ITEM_SHIFT) + inc);
    old = __shfl_sync(0xffffffffu, old, 31);
    const uint32_t slot = (uint32_t)(old >> ITEM_SHIFT) + __popc(has & lanemask_below());
    const unsigned long long base = (old & WEDGE_MASK) + inc - mine;
    if (!lng || slot > usable) return false;
    q.ibase[slot] = base;
    if (slot == usable) return false;
    q.items[slot] = it;
    return true;
}

// ---------------------------------------------------------------------------
// One wedge (entry j of x's weight-sorted list) of edge r = {x, y}.  The
// neighbour's degree and both its row bounds are loaded together: one step
// of latency before the search.
// ---------------------------------------------------------------------------
template <int P, bool SAMPLED>
__device__ __forceinline__ void wedge(const DevGraph& G, const Query& q, unsigned long long tau, int32_t r, uint32_t w,
                                      int32_t x, int32_t y, int64_t dy, int64_t yb, int32_t yn, int64_t j, Tally& tb) {
    const int32_t c = __ldg(G.wcol + j);
    const uint32_t wxc = (uint32_t)__ldg(G.wwt + j);
    const int32_t rxc = __ldg(G.wrk + j);
    if (SAMPLED && c == y) return;  // the edge itself (full rows in sampled mode)
    const int64_t c0 = __ldg(G.rowptr + c), c1 = __ldg(G.rowptr + c + 1);
    const int64_t o0 = __ldg(G.orowptr + c), o1 = __ldg(G.orowptr + c + 1);
    tb.add(12 + 32);
    const int64_t dc = c1 - c0;
    const bool yo = dy < dc || (dy == dc && y < c);  // the edge lies in the row of the lower-ranked endpoint
    const int64_t lb = yo ? yb : o0;
    const int32_t ln = yo ? yn : (int32_t)(o1 - o0), t = yo ? c : y;
    const int64_t at = search_ids(G.ocol, lb, ln, t, tb);
    if (at >= lb + ln) return;
    tb.add(4);
    if (__ldg(G.ocol + at) != t) return;
    const uint32_t wyc = (uint32_t)__ldg(G.owt + at);
    tb.add(8);
    if (!owns<SAMPLED>(q, r, rxc, __ldg(G.ork + at))) return;
    if (P == P_GEN && Line<P>(q, tau, w, wxc).fails(wyc)) return;  // surely below: no fp64 key
    const unsigned long long key = keyof<P>(w, wxc, wyc, q.gp, q.fw != 0);
    if (key >= tau) {
        int32_t a = x, b = y, cc = c;
        sort3(a, b, cc);
        append(q, key, a, b, cc);
    }
}

// The live ranges of a warp's 32 edges, scanned on the spot: their wedges
// numbered through, 32 at a time.
struct WarpItems {
    Item it[32];
    unsigned long long end[32];  // wedges up to and with each range
};

template <int P, bool SAMPLED>
__device__ __forceinline__ void scan_here(const DevGraph& G, const Query& q, unsigned long long tau, int64_t len,
                                          const Item& it, WarpItems& W, Tally& tb) {
    const int lane = threadIdx.x & 31;
    if (!__any_sync(0xffffffffu, len > 0)) return;
    unsigned long long inc = (unsigned long long)len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    const unsigned long long tot = __shfl_sync(0xffffffffu, inc, 31);
    W.it[lane] = it;
    W.end[lane] = inc;
    __syncwarp();
    for (unsigned long long e = lane; e < tot; e += 32) {
        int k = 0;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1)
            if (W.end[k + s - 1] <= e) k += s;
        const Item& x = W.it[k];
        const int64_t j = x.j0 + (int64_t)(e - (k > 0 ? W.end[k - 1] : 0ull));
        wedge<P, SAMPLED>(G, q, tau, x.r, x.w, x.x, x.y, x.dy, x.lb, x.ln, j, tb);
    }
    __syncwarp();
}

// Entry j of the scanned oriented row of the edge {a, b} at p = -inf; the
// third vertex is searched in the other row [lb, lb + ln).
__device__ __forceinline__ void min_entry(const DevGraph& G, const Query& q, unsigned long long tau, uint32_t w,
                                          int32_t a, int32_t b, int64_t lb, int32_t ln, int64_t j, uint32_t wsc,
                                          Tally& tb) {
    const int32_t c = __ldg(G.ocol + j);
    tb.add(4);
    const int64_t at = search_ids(G.ocol, lb, ln, c, tb);
    if (at >= lb + ln) return;
    tb.add(4);
    if (__ldg(G.ocol + at) != c) return;
    const uint32_t wlc = (uint32_t)__ldg(G.owt + at);
    tb.add(4);
    const unsigned long long key = keyof<P_MIN>(w, wsc, wlc);
    if (key >= tau) {
        int32_t x = a, y = b, z = c;
        sort3(x, y, z);
        append(q, key, x, y, z);
    }
}

// ---------------------------------------------------------------------------
// Phase A, heavy-first sweep.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool other_shard(const Query& q, int32_t r) {
    return q.nshards > 1 && (int32_t)(((uint32_t)r >> SHARD_SHIFT) % (uint32_t)q.nshards) != q.shard;
}

// A warp per edge: lanes 0-15 search u's list, lanes 16-31 v's.
template <int P, bool SAMPLED, class Team>
__device__ __forceinline__ void edges_by_warp(const DevGraph& G, const Query& q, unsigned long long tau, int64_t lo,
                                              int64_t hi, int par, const Team& T, Tally& tb) {
    const int lane = threadIdx.x & 31;
    const bool sv_ = lane >= 16;
    for (int64_t idx = lo + T.warp(); idx < hi; idx += T.warps()) {
        const int32_t r = SAMPLED ? __ldg(q.slist + idx) : (int32_t)idx;
        if (!SAMPLED && other_shard(q, r)) continue;
        const int32_t u = __ldg(G.ord_u + r), v = __ldg(G.ord_v + r);
        const uint32_t w = (uint32_t)__ldg(G.ord_w + r);
        const int32_t me = sv_ ? v : u;
        const int64_t b = __ldg(G.rowptr + me), e = __ldg(G.rowptr + me + 1);
        const int64_t ob = __ldg(G.orowptr + me), oe = __ldg(G.orowptr + me + 1);
        if ((lane & 15) == 0) tb.add(6 + 32);
        // Exact mode scans what comes after r in each list; sampled mode scans
        // whole lists (the other two edges may be heavier than a drawn edge).
        int64_t s = b;
        bool bad = false;
        if (!SAMPLED) {
            s = group_search<16>(b, e, [&](int64_t p) {
                tb.add(4);
                return __ldg(G.wrk + p) < r;
            });
            bad = s >= e || __ldg(G.wrk + s) != r;
            s++;
        }
        if (__any_sync(0xffffffffu, bad)) {
            if (bad) atomicOr(&q.st->err, DEV_ERR_INTERNAL);
            continue;
        }
        if (__any_sync(0xffffffffu, s >= e)) continue;  // no edge after r on one side: owns nothing
        const uint32_t top = (uint32_t)__ldg(G.wwt + s);
        const uint32_t oth = __shfl_xor_sync(0xffffffffu, top, 16);
        const Line<P> line(q, tau, w, oth);
        if (__any_sync(0xffffffffu, line.fails(top))) continue;  // edge bound
        int64_t end = e;
        if (tau != 0)
            end = group_search<16>(s, e, [&](int64_t p) {
                tb.add(4);
                return !line.fails((uint32_t)__ldg(G.wwt + p));
            });
        const int64_t len = end - s, olen = __shfl_xor_sync(0xffffffffu, len, 16);
        // x: the endpoint of the shorter live range (u on a tie)
        const bool x_me = sv_ ? len < olen : len <= olen;
        const int src = __ffs(__ballot_sync(0xffffffffu, x_me)) - 1, dst = src ^ 16;
        const int64_t j0 = __shfl_sync(0xffffffffu, s, src), n = __shfl_sync(0xffffffffu, len, src);
        const int32_t x = __shfl_sync(0xffffffffu, me, src), y = __shfl_sync(0xffffffffu, me, dst);
        const int64_t dy = __shfl_sync(0xffffffffu, e - b, dst);
        const int64_t yb = __shfl_sync(0xffffffffu, ob, dst);
        const int32_t yn = (int32_t)__shfl_sync(0xffffffffu, oe - ob, dst);
        const int64_t budget = q.t_short > 32 ? ((int64_t)q.t_short + 31) / 32 * 32 : 32;
        if (n <= budget) {
            for (int64_t j = j0 + lane; j < j0 + n; j += 32)
                wedge<P, SAMPLED>(G, q, tau, r, w, x, y, dy, yb, yn, j, tb);
            __syncwarp();
        } else if (lane == 0) {
            const unsigned long long old =
                atomicAdd(&q.st->items[par], (1ull << ITEM_SHIFT) + (unsigned long long)n);
            put_item(q, (uint32_t)(old >> ITEM_SHIFT), old & WEDGE_MASK,
                     Item{r, x, y, w, j0, yb, yn, (int32_t)dy, {0, 0}});
        }
        __syncwarp();
    }
}

// A thread per edge: large rounds, where most edges fail the edge bound.  flat:
// the round may have more live ranges than there are items.
template <int P, bool SAMPLED, class Team>
__device__ __forceinline__ void edges_by_thread(const DevGraph& G, const Query& q, unsigned long long tau, int64_t lo,
                                                int64_t hi, int par, bool flat, const Team& T, WarpItems& W, Tally& tb) {
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = lo + T.warp() * 32; i0 < hi; i0 += T.warps() * 32) {
        const int64_t idx = i0 + lane;
        int64_t n = 0;
        Item it{};
        if (idx < hi) {
            const int32_t r = SAMPLED ? __ldg(q.slist + idx) : (int32_t)idx;
            if (SAMPLED || !other_shard(q, r)) {
                const int32_t u = __ldg(G.ord_u + r), v = __ldg(G.ord_v + r);
                const uint32_t w = (uint32_t)__ldg(G.ord_w + r);
                const int64_t bu = __ldg(G.rowptr + u), eu = __ldg(G.rowptr + u + 1);
                const int64_t bv = __ldg(G.rowptr + v), ev = __ldg(G.rowptr + v + 1);
                tb.add(44);
                int64_t su = bu, sv = bv;
                bool bad = false;
                if (!SAMPLED) {  // both suffix searches step together
                    int64_t hu = eu, hv = ev;
                    while (su < hu || sv < hv) {
                        const int64_t mu = (su + hu) >> 1, mv = (sv + hv) >> 1;
                        const int32_t ku = su < hu ? __ldg(G.wrk + mu) : 0, kv = sv < hv ? __ldg(G.wrk + mv) : 0;
                        tb.add(8);
                        if (su < hu) {
                            if (ku < r) su = mu + 1;
                            else hu = mu;
                        }
                        if (sv < hv) {
                            if (kv < r) sv = mv + 1;
                            else hv = mv;
                        }
                    }
                    bad = su >= eu || sv >= ev || __ldg(G.wrk + su) != r || __ldg(G.wrk + sv) != r;
                    if (bad) atomicOr(&q.st->err, DEV_ERR_INTERNAL);
                    su++;
                    sv++;
                }
                if (!bad && su < eu && sv < ev) {
                    uint32_t umax = 0, vmax = 0;
                    if (tau != 0) {  // (without a threshold nothing is bounded: two loads saved)
                        umax = (uint32_t)__ldg(G.wwt + su), vmax = (uint32_t)__ldg(G.wwt + sv);
                        tb.add(8);
                    }
                    const Line<P> lu(q, tau, w, vmax);  // along u's list
                    if (tau == 0 || !lu.fails(umax)) {
                        int64_t nu = eu - su, nv = ev - sv;
                        if (tau != 0) {  // both live ranges
                            const Line<P> lv(q, tau, w, umax);
                            int64_t pu = su + 1, hu = eu, pv = sv + 1, hv = ev;
                            while (pu < hu || pv < hv) {
                                const int64_t mu = (pu + hu) >> 1, mv = (pv + hv) >> 1;
                                const uint32_t ku = pu < hu ? (uint32_t)__ldg(G.wwt + mu) : 0u;
                                const uint32_t kv = pv < hv ? (uint32_t)__ldg(G.wwt + mv) : 0u;
                                tb.add(8);
                                if (pu < hu) {
                                    if (!lu.fails(ku)) pu = mu + 1;
                                    else hu = mu;
                                }
                                if (pv < hv) {
                                    if (!lv.fails(kv)) pv = mv + 1;
                                    else hv = mv;
                                }
                            }
                            nu = pu - su;
                            nv = pv - sv;
                        }
                        const bool xu = nu <= nv;
                        n = xu ? nu : nv;
                        it.r = r;
                        it.x = xu ? u : v;
                        it.y = xu ? v : u;
                        it.w = w;
                        it.j0 = xu ? su : sv;
                        it.lb = __ldg(G.orowptr + it.y);
                        it.ln = (int32_t)(__ldg(G.orowptr + it.y + 1) - it.lb);
                        it.dy = (int32_t)(xu ? ev - bv : eu - bu);
                        tb.add(16);
                    }
                }
            }
        }
        if (!flat) {
            push_items(q, par, n, it);
        } else {
            if (push_long(q, par, n, it)) n = 0;
            scan_here<P, SAMPLED>(G, q, tau, n, it, W, tb);
        }
    }
}

// ---------------------------------------------------------------------------
// Phase A at p = -inf by NodeIterator++ over the degree order (Section 5.2):
// for each edge r = {a, b}, a the endpoint of lower (degree, id) rank, a
// triangle a < b < c in that order is found exactly once, as c in N+(a) and
// N+(b) (the oriented rows): the shorter row is scanned and each c searched
// in the other.  Its key min(w_ab, w_ac, w_bc) is at most w_r, so the
// heavy-first stop of the sweep holds, and entries lighter than tau are
// skipped before the search.  Every edge of a qualifying triangle is at
// least tau, which is why this replaces the weight-sorted scan (whose wedge
// bound prunes little at p = -inf) for the unsampled, unsharded query.
// ---------------------------------------------------------------------------
struct MinRows {
    int32_t a, b;
    int64_t sb, se, lb;  // scanned row, searched row
    int32_t ln;
};

__device__ __forceinline__ MinRows min_rows(int32_t u, int32_t v, int64_t du, int64_t dv, int64_t u0, int64_t u1,
                                            int64_t v0, int64_t v1) {
    MinRows R;
    const bool ua = du < dv || (du == dv && u < v);
    R.a = ua ? u : v;
    R.b = ua ? v : u;
    const bool us = (u1 - u0) < (v1 - v0) || ((u1 - u0) == (v1 - v0) && ua);
    R.sb = us ? u0 : v0;
    R.se = us ? u1 : v1;
    R.lb = us ? v0 : u0;
    R.ln = (int32_t)(us ? v1 - v0 : u1 - u0);
    return R;
}

// Small rounds: every edge leaves its scanned row as an item.
template <class Team>
__device__ __forceinline__ void min_edges_items(const DevGraph& G, const Query& q, int64_t lo, int64_t hi, int par,
                                                const Team& T, Tally& tb) {
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = lo + T.warp() * 32; i0 < hi; i0 += T.warps() * 32) {
        const int64_t r = i0 + lane;
        int64_t n = 0;
        Item it{};
        if (r < hi) {
            const int32_t u = __ldg(G.ord_u + r), v = __ldg(G.ord_v + r);
            const int64_t du = __ldg(G.rowptr + u + 1) - __ldg(G.rowptr + u);
            const int64_t dv = __ldg(G.rowptr + v + 1) - __ldg(G.rowptr + v);
            const MinRows R = min_rows(u, v, du, dv, __ldg(G.orowptr + u), __ldg(G.orowptr + u + 1),
                                       __ldg(G.orowptr + v), __ldg(G.orowptr + v + 1));
            tb.add(12 + 64);
            it = Item{(int32_t)r, R.a, R.b, (uint32_t)__ldg(G.ord_w + r), R.sb, R.lb, R.ln, 0, {0, 0}};
            n = R.ln > 0 ? R.se - R.sb : 0;
        }
        push_items(q, par, n, it);
    }
}

// A warp scans its edge's row itself: small graphs (rows of at most sqrt(2
// SMALL_M) entries), whose rounds then have no second phase, and dense ones
// before there is a threshold.
template <class Team>
__device__ __forceinline__ void min_edges_by_warp(const DevGraph& G, const Query& q, unsigned long long tau, int64_t lo,
                                                  int64_t hi, const Team& T, Tally& tb) {
    const int lane = threadIdx.x & 31;
    for (int64_t r = lo + T.warp(); r < hi; r += T.warps()) {
        const int32_t u = __ldg(G.ord_u + r), v = __ldg(G.ord_v + r);
        const uint32_t w = (uint32_t)__ldg(G.ord_w + r);
        const int64_t du = __ldg(G.rowptr + u + 1) - __ldg(G.rowptr + u);
        const int64_t dv = __ldg(G.rowptr + v + 1) - __ldg(G.rowptr + v);
        const MinRows R = min_rows(u, v, du, dv, __ldg(G.orowptr + u), __ldg(G.orowptr + u + 1),
                                   __ldg(G.orowptr + v), __ldg(G.orowptr + v + 1));
        if (lane == 0) tb.add(12 + 64);
        if (R.ln == 0) continue;
        for (int64_t j = R.sb + lane; j < R.se; j += 32) {
            const uint32_t wsc = (uint32_t)__ldg(G.owt + j);
            tb.add(4);
            if (wsc >= tau) min_entry(G, q, tau, w, R.a, R.b, R.lb, R.ln, j, wsc, tb);
        }
        __syncwarp();
    }
}

// Large rounds, where few entries reach tau: GL lanes per edge read its
// scanned row 4 GL weights at a time (16-byte loads, the next ones in flight
// while these are compared), 32 / GL edges to a warp, the endpoints of the
// edges two steps ahead and the row bounds of the next step's edges loaded
// while this step scans.  The entries that reach tau wait in the warp's queue
// until 32 of them are there, and are then searched one per lane.
struct MinProbe {
    int64_t j, lb;
    int32_t ln;
    uint32_t w;
    int32_t a, b;
};
// Edges per vertex from which a scanned row gets eight lanes, not four (us with
// four / eight: random graphs of 4 / 16 edges per vertex 2,370 / 3,230, 4,140 /
// 4,860; skewed ones of 8 / 20 / 30: 280 / 276, 364 / 357, 261 / 254).
constexpr int64_t MIN_WIDE = 12;
// Edges per vertex from which a round without a threshold, whose entries all count,
// takes a warp per edge and no queue (us, warp / queue: 100 edges per vertex, no
// triangles, 1,539 / 1,694; 16 per vertex 9,990 / 4,870).
constexpr int64_t MIN_DENSE = 64;
constexpr int MINQ = 64;  // a step of at most 32 entries on top of at most 31 waiting

template <int GL, class Team>
__device__ __forceinline__ void min_edges_filtered(const DevGraph& G, const Query& q, unsigned long long tau,
                                                   int64_t lo, int64_t hi, const Team& T, MinProbe* queue, Tally& tb) {
    constexpr int EPW = 32 / GL;  // edges per warp and step
    const int lane = threadIdx.x & 31, gl = lane & (GL - 1);
    const uint32_t lt = lanemask_below();
    const int64_t first = lo + T.warp() * EPW, stride = T.warps() * EPW;
    const int32_t* ord = gl == 0 ? G.ord_u : (gl == 1 ? G.ord_v : G.ord_w);
    auto triple = [&](int64_t r) { return gl < 3 && r < hi ? __ldg(ord + r) : 0; };
    struct Bounds {
        int64_t row, orow;
    };
    auto bounds = [&](int64_t r, int32_t t) {  // lane gl: bound gl & 1 of the rows of u or v (gl & 2)
        const int32_t u = __shfl_sync(0xffffffffu, t, 0, GL), v = __shfl_sync(0xffffffffu, t, 1, GL);
        Bounds x{0, 0};
        if (r < hi) {
            const int64_t i = (int64_t)(gl & 2 ? v : u) + (gl & 1);
            x.row = __ldg(G.rowptr + i);
            x.orow = __ldg(G.orowptr + i);
        }
        return x;
    };
    int qn = 0;
    auto probe = [&](int n) {  // the queue's last n entries, one per lane
        __syncwarp();
        if (lane < n) {
            const MinProbe e = queue[qn - n + lane];
            min_entry(G, q, tau, e.w, e.a, e.b, e.lb, e.ln, e.j, (uint32_t)__ldg(G.owt + e.j), tb);
        }
        __syncwarp();
        qn -= n;
    };
    int64_t r = first + lane / GL;
    if (first >= hi) return;
    int32_t t0 = triple(r), t1 = triple(r + stride);
    Bounds b0 = bounds(r, t0);
    for (int64_t base = first; base < hi; base += stride, r += stride) {
        const int32_t t2 = triple(r + 2 * stride);
        const Bounds b1 = bounds(r + stride, t1);
        const int32_t u = __shfl_sync(0xffffffffu, t0, 0, GL), v = __shfl_sync(0xffffffffu, t0, 1, GL);
        const uint32_t w = (uint32_t)__shfl_sync(0xffffffffu, t0, 2, GL);
        int64_t x[4], ox[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            x[k] = __shfl_sync(0xffffffffu, b0.row, k, GL);
            ox[k] = __shfl_sync(0xffffffffu, b0.orow, k, GL);
        }
        const MinRows R = min_rows(u, v, x[1] - x[0], x[3] - x[2], ox[0], ox[1], ox[2], ox[3]);
        const int64_t se = r < hi && R.ln > 0 ? R.se : R.sb;
        if (gl == 0) tb.add(12 + 64);
        int64_t j = (R.sb & ~int64_t(3)) + 4 * gl;
        int4 nx = j < se ? __ldg(reinterpret_cast<const int4*>(G.owt + j)) : make_int4(0, 0, 0, 0);
        while (__any_sync(0xffffffffu, j < se)) {
            const int4 cur = nx;
            const int64_t jc = j;
            j += 4 * GL;
            nx = j < se ? __ldg(reinterpret_cast<const int4*>(G.owt + j)) : make_int4(0, 0, 0, 0);
            const uint32_t cw[4] = {(uint32_t)cur.x, (uint32_t)cur.y, (uint32_t)cur.z, (uint32_t)cur.w};
            if (jc < se) tb.add(16);
            bool heavy[4], some = false;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                heavy[k] = jc + k >= R.sb && jc + k < se && cw[k] >= tau;
                some |= heavy[k];
            }
            if (!__any_sync(0xffffffffu, some)) continue;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const uint32_t m = __ballot_sync(0xffffffffu, heavy[k]);
                if (heavy[k]) queue[qn + __popc(m & lt)] = MinProbe{jc + k, R.lb, R.ln, w, R.a, R.b};
                qn += __popc(m);
                if (qn >= 32) probe(32);
            }
        }
        t0 = t1;
        t1 = t2;
        b0 = b1;
    }
    if (qn > 0) probe(qn);
}

// ---------------------------------------------------------------------------
// Phase B: the items' wedges, numbered through.  Each warp takes a contiguous
// share, 32 at a time; a lane finds its wedge's item among the next 32 items
// (each has at least one wedge).
// ---------------------------------------------------------------------------
template <int P, bool SAMPLED, bool ORIENTED, class Team>
__device__ __forceinline__ void item_wedges(const DevGraph& G, const Query& q, unsigned long long tau,
                                            unsigned long long ctr, bool flat, const Team& T, Tally& tb) {
    const int64_t drawn_ = (int64_t)(ctr >> ITEM_SHIFT), cnt = min(drawn_, flat ? q.item_cap - 1 : q.item_cap);
    const int64_t tot = cnt == drawn_ ? (int64_t)(ctr & WEDGE_MASK) : (int64_t)q.ibase[cnt];
    if (!flat && cnt != drawn_) return;
    const int lane = threadIdx.x & 31;
    const int64_t chunks = (tot + 31) >> 5, per = (chunks + T.warps() - 1) / T.warps();
    const int64_t beg = T.warp() * per * 32, end = min(tot, beg + per * 32);
    if (beg >= end) return;
    const unsigned long long* ib = q.ibase;
    int64_t it0 = group_search<32>(0, cnt, [&](int64_t p) { return (int64_t)ib[p] <= beg; }) - 1;
    for (int64_t e0 = beg; e0 < end; e0 += 32) {
        // where item it0 + lane ends, relative to e0
        const int64_t nxt = it0 + 1 + lane;
        const int64_t rel = (nxt < cnt ? (int64_t)ib[nxt] : tot) - e0;
        const int stop = rel > 64 ? 64 : (int)rel;
        int k = 0;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) {
            const int v = __shfl_sync(0xffffffffu, stop, (k + s - 1) & 31);
            if (v <= lane) k += s;
        }
        const int64_t i = it0 + k;
        if (e0 + lane < end) {
            const int4* p = reinterpret_cast<const int4*>(q.items + i);
            const int4 a = p[0], b = p[1], c = p[2];
            const int64_t j0 = ((int64_t)(uint32_t)b.y << 32) | (uint32_t)b.x;
            const int64_t lb = ((int64_t)(uint32_t)b.w << 32) | (uint32_t)b.z;
            const int64_t j = j0 + (e0 + lane - (int64_t)ib[i]);
            if constexpr (ORIENTED) {
                const uint32_t wsc = (uint32_t)__ldg(G.owt + j);
                tb.add(4);
                if (wsc >= tau) min_entry(G, q, tau, (uint32_t)a.w, a.y, a.z, lb, c.x, j, wsc, tb);
            } else {
                wedge<P, SAMPLED>(G, q, tau, a.x, (uint32_t)a.w, a.y, a.z, c.y, lb, c.x, j, tb);
            }
        }
        __syncwarp();
        const int k31 = __shfl_sync(0xffffffffu, k, 31);
        const int s31 = __shfl_sync(0xffffffffu, stop, k31);
        it0 += k31 + (s31 <= 32 ? 1 : 0);
    }
}

// ---------------------------------------------------------------------------
// Selection under the total order (key desc, a asc, b asc, c asc), one block.
// Radix selects take digits of 11 bits from the highest bit in which the
// candidates differ; the whole block scans a histogram's bins (a serial scan
// by one thread cost 4 us per digit, half of every select).
// ---------------------------------------------------------------------------
constexpr int SEL_BITS = 11;
constexpr int SEL_BINS = 1 << SEL_BITS;

struct SelectSmem {
    uint32_t hist[SEL_BINS];
    uint32_t wsum[32];
    unsigned long long mn, mx;
    uint32_t bin, above, taken;
    uint32_t err, n, old;  // the query's error bits, candidates and `selected`, as one thread read them
    int narrow;  // a round of more edges than items filled the candidate buffer
    int gone;    // a grid barrier gave up
};

// The query's state for the whole selecting block.  One thread reads it: a
// block whose first barrier wait runs out sets the timeout bit after its
// arrival has been counted, so at any moment here, and threads that branched
// around the block's barriers on readings of their own could part.
template <int TB>
__device__ __forceinline__ void read_state(const Part<TB>& B, const Query& q, SelectSmem& S) {
    if (B.tid() == 0) {
        S.err = *(volatile uint32_t*)&q.st->err;
        S.n = min(*(volatile uint32_t*)&q.st->count, q.cap);
        S.old = *(volatile uint32_t*)&q.st->selected;
    }
    B.sync();
}

// The ranking's shared arrays (aliases the p = -inf queues of phase A).
struct SortSmem {
    unsigned long long key[SORT_MAX];
    int32_t tri[3][SORT_MAX];
    uint16_t id[SORT_MAX];
};

// First bin (in bin order) at which the running count reaches need (>= 1,
// at most the histogram's sum): S.bin, and the count before it in S.above.
template <int TB>
__device__ __forceinline__ void pick_bin(const Part<TB>& B, SelectSmem& S, uint32_t need) {
    constexpr int PER = SEL_BINS / TB;
    const int tid = B.tid(), lane = tid & 31, wid = tid >> 5;
    uint32_t h[PER], sum = 0;
#pragma unroll
    for (int i = 0; i < PER; i++) {
        h[i] = S.hist[tid * PER + i];
        sum += h[i];
    }
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) S.wsum[wid] = inc;
    B.sync();
    uint32_t before = 0;
#pragma unroll
    for (int k = 0; k < TB / 32; k++) before += k < wid ? S.wsum[k] : 0u;
    uint32_t acc = before + inc - sum;
    if (acc < need && need <= acc + sum) {
#pragma unroll
        for (int i = 0; i < PER; i++) {
            if (acc < need && need <= acc + h[i]) {
                S.bin = (uint32_t)(tid * PER + i);
                S.above = acc;
            }
            acc += h[i];
        }
    }
    B.sync();
}

template <int TB>
__device__ __forceinline__ void clear_hist(const Part<TB>& B, SelectSmem& S) {
    for (int i = B.tid(); i < SEL_BINS; i += TB) S.hist[i] = 0;
    B.sync();
}

// Counts d (< SEL_BINS; larger: nothing): the lanes of one bin add together.
__device__ __forceinline__ void count_bin(SelectSmem& S, uint32_t d) {
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    if (d < SEL_BINS && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&S.hist[d], __popc(peers));
}

// The K-th largest of n keys (K <= n).
template <int TB>
__device__ unsigned long long kth_key(const Part<TB>& B, const unsigned long long* ckey, uint32_t n, uint32_t K, SelectSmem& S) {
    const int tid = B.tid(), lane = tid & 31;
    unsigned long long mx = 0, mn = ~0ull;
#pragma unroll 4
    for (uint32_t i = tid; i < n; i += TB) {
        const unsigned long long x = ckey[i];
        mx = x > mx ? x : mx;
        mn = x < mn ? x : mn;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long a = __shfl_xor_sync(0xffffffffu, mx, o), b = __shfl_xor_sync(0xffffffffu, mn, o);
        mx = a > mx ? a : mx;
        mn = b < mn ? b : mn;
    }
    if (tid == 0) {
        S.mx = 0;
        S.mn = ~0ull;
    }
    B.sync();
    if (lane == 0) {
        atomicMax(&S.mx, mx);
        atomicMin(&S.mn, mn);
    }
    B.sync();
    mx = S.mx;
    mn = S.mn;
    if (mx == mn) return mx;
    int shift = 64 - __clzll((long long)(mx ^ mn));  // the bits that differ
    unsigned long long prefix = shift >= 64 ? 0ull : (mx >> shift) << shift;
    uint32_t need = K;
    while (shift > 0) {
        const int bits = shift < SEL_BITS ? shift : SEL_BITS, hi = shift;
        shift -= bits;
        const uint32_t mask = (1u << bits) - 1u;
        clear_hist<TB>(B, S);
#pragma unroll 4
        for (uint32_t base = 0; base < n; base += TB) {
            const uint32_t i = base + tid;
            uint32_t d = SEL_BINS;
            if (i < n) {
                const unsigned long long x = ckey[i];
                if (hi >= 64 || (x >> hi) == (prefix >> hi)) d = mask - ((uint32_t)(x >> shift) & mask);  // descending
            }
            count_bin(S, d);
        }
        B.sync();
        pick_bin<TB>(B, S, need);
        prefix |= (unsigned long long)(mask - S.bin) << shift;
        need -= S.above;
        B.sync();
    }
    return prefix;
}

// Keeps the candidates for which keep(key, triple) holds at the front, in any
// order, in place: a step's entries are in registers before any is written,
// and no more are written than were read.  Returns how many.
template <int TB, class Keep>
__device__ uint32_t compact(const Part<TB>& B, unsigned long long* ckey, int4* ctri, uint32_t n, const Keep& keep, SelectSmem& S) {
    constexpr int U = 2;
    const int tid = B.tid(), lane = tid & 31;
    if (tid == 0) S.taken = 0;
    for (uint32_t base = 0; base < n; base += U * TB) {
        unsigned long long k[U];
        int4 t[U];
        bool on[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const uint32_t i = base + u * TB + tid;
            on[u] = false;
            if (i < n) {
                k[u] = ckey[i];
                t[u] = ctri[i];
                on[u] = keep(k[u], t[u]);
            }
        }
        B.sync();
#pragma unroll
        for (int u = 0; u < U; u++) {
            const uint32_t b = __ballot_sync(0xffffffffu, on[u]);
            uint32_t at = 0;
            if (lane == 0 && b) at = atomicAdd(&S.taken, (uint32_t)__popc(b));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & lanemask_below());
            if (on[u]) {
                ckey[at] = k[u];
                ctri[at] = t[u];
            }
        }
    }
    B.sync();
    const uint32_t got = S.taken;
    B.sync();
    return got;
}

__device__ __forceinline__ uint32_t tri_word(const int4& t, int i) {
    return (uint32_t)(i == 0 ? t.x : (i == 1 ? t.y : t.z));
}

// Candidates all >= T: keeps those above T and the first of those equal to T
// in triple order, K in all (n > K; fewer than K lie above T).
template <int TB>
__device__ uint32_t keep_first_ties(const Part<TB>& B, unsigned long long* ckey, int4* ctri, uint32_t n, uint32_t K,
                                    unsigned long long T, SelectSmem& S) {
    const int tid = B.tid();
    if (tid == 0) S.taken = 0;
    B.sync();
    uint32_t mine = 0;
    for (uint32_t i = tid; i < n; i += TB) mine += ckey[i] > T ? 1u : 0u;
    if (mine) atomicAdd(&S.taken, mine);
    B.sync();
    uint32_t need = K - S.taken;
    B.sync();
    // limit: the need-th smallest triple among the ties, word by word
    uint32_t lim[3] = {0u, 0u, 0u};
    for (int wi = 0; wi < 3; wi++) {
        int shift = 32;
        while (shift > 0) {
            const int bits = shift < SEL_BITS ? shift : SEL_BITS, hi = shift;
            shift -= bits;
            const uint32_t mask = (1u << bits) - 1u;
            clear_hist<TB>(B, S);
            for (uint32_t base = 0; base < n; base += TB) {
                const uint32_t i = base + tid;
                uint32_t d = SEL_BINS;
                if (i < n && ckey[i] == T) {
                    const int4 t = ctri[i];
                    bool same = true;
                    for (int k = 0; k < wi; k++) same = same && tri_word(t, k) == lim[k];
                    const uint32_t x = tri_word(t, wi);
                    if (same && (hi >= 32 || (x >> hi) == (lim[wi] >> hi))) d = (x >> shift) & mask;
                }
                count_bin(S, d);
            }
            B.sync();
            pick_bin<TB>(B, S, need);
            lim[wi] |= S.bin << shift;
            need -= S.above;
            B.sync();
        }
    }
    const uint32_t l0 = lim[0], l1 = lim[1], l2 = lim[2];
    return compact<TB>(B, ckey, ctri, n,
                       [=](unsigned long long k, const int4& t) {
                           if (k != T) return k > T;
                           if ((uint32_t)t.x != l0) return (uint32_t)t.x < l0;
                           if ((uint32_t)t.y != l1) return (uint32_t)t.y < l1;
                           return (uint32_t)t.z <= l2;
                       },
                       S);
}

// After a round: tau = the k-th largest key among the candidates (a lower
// bound on the final k-th key, since they are k distinct triangles), and
// candidates below tau are dropped.  Ties with tau stay; the final step
// resolves them by the vertex triple.  Returns how much larger the next round
// may be: `growth`, or less where rounds as productive as this one would
// fill half of the free candidate slots (small buffers: a batched query at
// p = -inf overflowed its 16,384 slots at a fixed growth of 8); and whether it
// may have more edges than there are items: where the threshold hardly moved,
// or there is none yet, a select earlier would prune little.  Such a round
// (flat) may fill the candidate buffer where rounds of as many edges as items
// would not: then its candidates are dropped and it is to be done again, and all
// that follow, in those.
struct Growth {
    int64_t times;
    bool wide;
    bool again;
};

template <int TB>
__device__ Growth select_round(const Part<TB>& B, const Query& q, bool flat, SelectSmem& S) {
    const int64_t growth = q.growth;
    read_state<TB>(B, q, S);
    const uint32_t n = S.n, old = S.old;
    if (flat && S.err == DEV_ERR_OVERFLOW) {
        if (B.tid() == 0) {
            S.narrow = 1;
            *(volatile uint32_t*)&q.st->count = old;
            atomicAnd(&q.st->err, ~DEV_ERR_OVERFLOW);
        }
        return Growth{1, false, true};
    }
    if (S.err || n == old) return Growth{growth, true, false};
    const int64_t added = n - old;
    if (n < (uint32_t)q.k) {
        if (B.tid() == 0) *(volatile uint32_t*)&q.st->selected = n;  // all of them stay
        return Growth{max(int64_t(1), min(growth, (int64_t)(q.cap - n) / (2 * added))), true, false};
    }
    const unsigned long long T = kth_key<TB>(B, q.ckey, n, (uint32_t)q.k, S);
    const uint32_t kept = compact<TB>(B, q.ckey, q.ctri, n, [=](unsigned long long k, const int4&) { return k >= T; }, S);
    if (B.tid() == 0) {
        *(volatile uint32_t*)&q.st->count = kept;
        *(volatile uint32_t*)&q.st->selected = kept;
        if (T > q.st->tau) *(volatile unsigned long long*)&q.st->tau = T;
    }
    B.sync();
    return Growth{max(int64_t(1), min(growth, (int64_t)(q.cap - kept) / (2 * added))), 8 * added <= q.k, false};
}

// The next round's range: [lo, lo + size) cut at the first edge whose bound
// is below tau (the edges' weights do not increase); empty after an error.
template <int P, bool SAMPLED>
__device__ __forceinline__ void next_range(int tid, const DevGraph& G, const Query& q, int64_t lo, int64_t size,
                                           int64_t total, bool failed) {
    if (tid >= 32) return;
    const unsigned long long tau = ld_volatile_u64(&q.st->tau);
    int64_t hi = failed ? lo : min(total, lo + size);
    if (!SAMPLED && tau != 0)
        hi = group_search<32>(lo, hi, [&](int64_t p) { return !edge_below<P>(q, (uint32_t)__ldg(G.ord_w + p), tau); });
    if (tid == 0) {
        *(volatile long long*)&q.st->lo = lo;
        *(volatile long long*)&q.st->hi = hi;
        *(volatile long long*)&q.st->size = size;
    }
}

// ---------------------------------------------------------------------------
// Ranking and outputs.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool before(unsigned long long ka, int4 a, unsigned long long kb, int4 b) {
    if (ka != kb) return ka > kb;
    if (a.x != b.x) return a.x < b.x;
    if (a.y != b.y) return a.y < b.y;
    return a.z < b.z;
}

template <int P>
__device__ __forceinline__ void write_rank(const Query& q, const Out& o, uint32_t rank, unsigned long long key,
                                           int32_t a, int32_t b, int32_t c) {
    o.tri[rank].a = a;
    o.tri[rank].b = b;
    o.tri[rank].c = c;
    double val;
    if (P == P_ONE) val = (double)key / 3.0;
    else if (P == P_TWO) val = sqrt((double)key / 3.0);
    else if (P == P_GEO) val = cbrt((double)key);
    else if (P == P_GEN) val = __longlong_as_double((long long)key);
    else val = q.fw ? (double)__uint_as_float((uint32_t)key) : (double)key;  // min, max
    o.w[rank] = val;
    if (o.key) o.key[rank] = key;
}

// Sorts n <= SORT_MAX candidates in shared memory (bitonic over positions):
// the i-th is R.id[i].
template <int TB>
__device__ __forceinline__ void sort_ids(const Part<TB>& B, const unsigned long long* ckey, const int4* ctri, uint32_t n,
                                         SortSmem& R) {
    uint32_t N = 2;
    while (N < n) N <<= 1;
    for (uint32_t i = B.tid(); i < N; i += TB) {
        R.key[i] = i < n ? ckey[i] : 0ull;  // keys are positive: padding ranks last
        const int4 t = i < n ? ctri[i] : make_int4(INT32_MAX, INT32_MAX, INT32_MAX, 0);
        R.tri[0][i] = t.x;
        R.tri[1][i] = t.y;
        R.tri[2][i] = t.z;
        R.id[i] = (uint16_t)i;
    }
    B.sync();
    auto first = [&](uint32_t a, uint32_t b) {  // candidate a ranks before b
        if (R.key[a] != R.key[b]) return R.key[a] > R.key[b];
        if (R.tri[0][a] != R.tri[0][b]) return R.tri[0][a] < R.tri[0][b];
        if (R.tri[1][a] != R.tri[1][b]) return R.tri[1][a] < R.tri[1][b];
        return R.tri[2][a] < R.tri[2][b];
    };
    for (uint32_t size = 2; size <= N; size <<= 1)
        for (uint32_t d = size >> 1; d > 0; d >>= 1) {
            for (uint32_t t = B.tid(); t < N / 2; t += TB) {
                const uint32_t i = 2 * t - (t & (d - 1)), j = i + d;
                const uint32_t a = R.id[i], b = R.id[j];
                if ((i & size) == 0 ? first(b, a) : first(a, b)) {
                    R.id[i] = (uint16_t)b;
                    R.id[j] = (uint16_t)a;
                }
            }
            B.sync();
        }
}

// Whether the team ranks n candidates of a k above SORT_MAX together: more than
// one block sorts, or few enough to count (1,333 results of k = 3,000 on 2e5 edges,
// the whole query: 175 us, sorted by one block 194).
template <class Team>
__device__ __forceinline__ bool counts_ranks(const Team& T, uint32_t n) {
    return Team::GRID && (int64_t)n <= 2 * T.warps();
}
template <class Team>
__device__ __forceinline__ bool ranks_many(const Team& T, uint32_t n) {
    return n > SORT_MAX || counts_ranks(T, n);
}

// Ranks candidates, all of them results.  False: a barrier gave up.  Up to two
// per warp: each warp counts the candidates before its own (k = 3,000 on the
// whole GPU: the query takes 208 us, 244 by runs).  More: sorted runs of
// SORT_MAX, a block each, then every candidate's place is its place in its run
// and, for each other run, the entries before it (a lane per run searches).  By
// counting, k = 16,384 / 65,536 on the whole GPU 0.59 / 4.9 ms, by runs 0.42 /
// 0.97; and 490 ms on one SM of a batch.
template <int P, class Team>
__device__ __forceinline__ bool rank_many(const Query& q, const Out& o, uint32_t n, Team& T, SortSmem& R) {
    if (counts_ranks(T, n)) {
        for (int64_t i = T.warp(); i < (int64_t)n; i += T.warps()) {
            const unsigned long long ki = q.ckey[i];
            const int4 ti = q.ctri[i];
            uint32_t rank = 0;
            for (uint32_t j = threadIdx.x & 31; j < n; j += 32) rank += before(q.ckey[j], q.ctri[j], ki, ti) ? 1u : 0u;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, s);
            if ((threadIdx.x & 31) == 0) write_rank<P>(q, o, rank, ki, ti.x, ti.y, ti.z);
        }
        return T.sync(q);
    }
    const Part<Team::TB>& B = T.part;
    const uint32_t runs = (n + SORT_MAX - 1) / SORT_MAX;
    for (uint32_t r = (uint32_t)T.block(); r < runs; r += (uint32_t)T.blocks()) {
        const uint32_t at = r * SORT_MAX, len = min((uint32_t)SORT_MAX, n - at);
        sort_ids<Team::TB>(B, q.ckey + at, q.ctri + at, len, R);
        for (uint32_t i = B.tid(); i < len; i += Team::TB) {
            const uint32_t c = R.id[i];
            q.ckey[at + i] = R.key[c];
            q.ctri[at + i] = make_int4(R.tri[0][c], R.tri[1][c], R.tri[2][c], 0);
        }
        B.sync();  // the shared arrays are read before the next run
    }
    if (!T.sync(q)) return false;
    uint32_t G = 1;  // lanes per candidate
    while (G < runs && G < 32) G <<= 1;
    const uint32_t lane = threadIdx.x & 31, gl = lane & (G - 1), per = 32 / G;
    for (int64_t i0 = T.warp() * per; i0 < (int64_t)n; i0 += T.warps() * per) {
        const uint32_t i = (uint32_t)min(i0 + lane / G, (int64_t)n - 1);
        const unsigned long long ki = q.ckey[i];
        const int4 ti = q.ctri[i];
        uint32_t rank = 0;
        for (uint32_t r = gl; r < runs; r += G) {
            uint32_t lo = r * SORT_MAX, hi = min(lo + SORT_MAX, n);
            if (r == i / SORT_MAX) lo = hi = i;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1;
                const unsigned long long km = q.ckey[mid];
                if (km != ki ? km > ki : before(km, q.ctri[mid], ki, ti)) lo = mid + 1;
                else hi = mid;
            }
            rank += lo - r * SORT_MAX;
        }
        for (uint32_t s = G >> 1; s > 0; s >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, s);
        if (gl == 0 && i0 + lane / G < (int64_t)n) write_rank<P>(q, o, rank, ki, ti.x, ti.y, ti.z);
    }
    return T.sync(q);
}

// The k best candidates in order, and the status word: one block sorts up to
// SORT_MAX of them; above, the team ranks them, and the status is written
// after one more barrier, when every result is.  False: a barrier gave up.
template <int P, class Team>
__device__ bool finish(const Query& q, const Out& o, Team& T, SelectSmem& S, SortSmem& R) {
    const uint32_t K = (uint32_t)q.k;
    const Part<Team::TB>& B = T.part;
    int32_t status = 0;
    if (T.leader()) {
        read_state<Team::TB>(B, q, S);
        const uint32_t err = S.err;
        uint32_t n = err ? 0 : S.n;
        if (n > K) {
            unsigned long long T0 = ld_volatile_u64(&q.st->tau);
            if (n != S.old) {
                T0 = kth_key<Team::TB>(B, q.ckey, n, K, S);
                n = compact<Team::TB>(B, q.ckey, q.ctri, n, [=](unsigned long long k, const int4&) { return k >= T0; }, S);
            }
            if (n > K && (n > SORT_MAX || K > SORT_MAX)) n = keep_first_ties<Team::TB>(B, q.ckey, q.ctri, n, K, T0, S);
        }
        // a timeout first: an overflow that follows it is its consequence
        status = (int32_t)min(n, K);
        if (err & DEV_ERR_TIMEOUT) status = WTRI_ETIMEOUT;
        else if (err & DEV_ERR_OVERFLOW) status = WTRI_ENOMEM;
        else if (err) status = WTRI_ECUDA;
        if (B.tid() == 0) *(volatile uint32_t*)&q.st->kept = n;
        if (K <= SORT_MAX || !ranks_many(T, n)) {
            sort_ids<Team::TB>(B, q.ckey, q.ctri, n, R);
            for (uint32_t i = B.tid(); i < min(n, K); i += Team::TB) {
                const uint32_t c = R.id[i];
                write_rank<P>(q, o, i, R.key[c], R.tri[0][c], R.tri[1][c], R.tri[2][c]);
            }
        }
    }
    if (K > SORT_MAX) {
        if (!T.sync(q)) return false;
        const uint32_t n = *(volatile uint32_t*)&q.st->kept;
        if (ranks_many(T, n) && !rank_many<P>(q, o, n, T, R)) return false;
    }
    if (T.leader() && B.tid() == 0) *o.count = status;
    return true;
}

// ---------------------------------------------------------------------------
// The whole sweep.  False: a barrier gave up, and the leading block's caller
// writes WTRI_ETIMEOUT for the status, which is written once, at the end, either
// way.  A block that gives up has done its work up to that barrier, and the
// others, the leading one among them, cannot pass the next: where there is none,
// the answer is complete.
// ---------------------------------------------------------------------------
template <int TB>
struct SweepSmem {
    SelectSmem sel;
    union {
        SortSmem sort;
        MinProbe queue[TB / 32][MINQ];
        WarpItems here[TB / 32];
    };
};

template <int P, bool SAMPLED, class Team>
__device__ bool sweep(const DevGraph& G, const Query& q, const Out& o, Team& T, SweepSmem<Team::TB>& S) {
    const bool oriented = P == P_MIN && !SAMPLED && q.nshards <= 1;
    const int64_t total = q.total_dev ? __ldg(q.total_dev) : q.total;
    int64_t size = min(q.first, q.item_cap), lo = 0, hi = min(total, size);
    unsigned long long tau = 0;
    if (T.part.tid() == 0) S.sel.narrow = 0;
    Tally tb;
    tb.on = q.qbytes != nullptr;
    for (int par = 0; lo < hi; par ^= 1) {
        bool items = true;
        const bool flat = hi - lo > q.item_cap;  // more edges than items
        if constexpr (P == P_MIN && !SAMPLED) {
            if (oriented) {
                const bool by_warp = G.m <= SMALL_M ? hi - lo <= min(WARP_EDGES, T.warps() * 4)
                                                    : tau == 0 && hi - lo > MIN_FLAT && G.m >= MIN_DENSE * G.n;
                items = !by_warp && hi - lo <= min(MIN_FLAT, q.item_cap);
                if (by_warp) min_edges_by_warp(G, q, tau, lo, hi, T, tb);
                else if (items) min_edges_items(G, q, lo, hi, par, T, tb);
                else if (G.m < MIN_WIDE * G.n) min_edges_filtered<4>(G, q, tau, lo, hi, T, S.queue[T.part.tid() >> 5], tb);
                else min_edges_filtered<8>(G, q, tau, lo, hi, T, S.queue[T.part.tid() >> 5], tb);
            }
        }
        if (!oriented) {
            if (hi - lo <= min(WARP_EDGES, T.warps() * 4)) edges_by_warp<P, SAMPLED>(G, q, tau, lo, hi, par, T, tb);
            else edges_by_thread<P, SAMPLED>(G, q, tau, lo, hi, par, flat, T, S.here[T.part.tid() >> 5], tb);
        }
        if (!T.sync(q)) return false;
        // (none: small rounds often scan every live range in the first phase)
        const unsigned long long ctr = items ? ld_volatile_u64(&q.st->items[par]) : 0ull;
        if (ctr != 0) {
            if constexpr (P == P_MIN && !SAMPLED) {
                if (oriented) item_wedges<P, false, true>(G, q, tau, ctr, false, T, tb);
            }
            if (!oriented) item_wedges<P, SAMPLED, false>(G, q, tau, ctr, flat, T, tb);
            if (!T.sync(q)) return false;
        }
        if (T.leader()) {
            if (T.part.tid() == 0) *(volatile unsigned long long*)&q.st->items[par ^ 1] = 0;
            const Growth grow = select_round<Team::TB>(T.part, q, flat && !oriented, S.sel);
            const int64_t cap = oriented || (grow.wide && !S.sel.narrow) ? INT64_MAX / 1024 : q.item_cap;
            // (the state still holds this round's start)
            next_range<P, SAMPLED>(T.part.tid(), G, q, grow.again ? *(volatile long long*)&q.st->lo : hi,
                                   min(size * grow.times, cap), total, S.sel.err != 0 && !grow.again);
        }
        if (!T.sync(q)) return false;
        size = *(volatile long long*)&q.st->size;
        tau = ld_volatile_u64(&q.st->tau);
        lo = *(volatile long long*)&q.st->lo;
        hi = *(volatile long long*)&q.st->hi;
    }
    flush_tally(q, tb);
    return finish<P>(q, o, T, S.sel, S.sort);
}

template <int P, bool SAMPLED>
__global__ void __launch_bounds__(TGRID, 1) k_sweep(DevGraph G, Query q, Out o) {
    extern __shared__ __align__(16) unsigned char sweep_smem[];
    SweepSmem<TGRID>& S = *reinterpret_cast<SweepSmem<TGRID>*>(sweep_smem);
    GridTeam<TGRID> T;
    T.limit = q.wait_first;
    T.blk0 = 0;
    T.nblk = gridDim.x;
    T.gone = &S.sel.gone;
    if (threadIdx.x == 0) S.sel.gone = 0;
    __syncthreads();
    if (!sweep<P, SAMPLED>(G, q, o, T, S) && T.leader() && threadIdx.x == 0) *o.count = WTRI_ETIMEOUT;
}

// Blocks of a query's sweep: the whole GPU, fewer on small graphs, whose rounds
// have too few edges to fill them and pay for every block at the barriers
// (random graphs of 300 / 3,000 / 20,000 edges, p = 1, k = 50: 56 / 84 / 89 us on
// all SMs, now 40 / 62 / 76; p = -inf, k = 1,000, with the rounds of
// min_edges_by_warp: 54 / 83 / 119, now 37 / 56 / 93).  The general means spend
// their time in fp64 pow and take four times as many.
template <int P>
inline unsigned sweep_blocks(int64_t m) {
    if (m > SMALL_M) return (unsigned)sm_count();
    const int64_t fit = P == P_GEN ? (m + 15) / 16 : std::min<int64_t>(48, (m + 63) / 64);
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(sm_count(), fit));
}

// Launches the sweep of one query on the whole GPU (a cooperative launch:
// its blocks wait for one another, so all must be resident).
template <int P, bool SAMPLED>
int launch_sweep(const DevGraph& G, const Query& q, const Out& o, cudaStream_t s) {
    static std::atomic<uint64_t> done{0};
    const void* fn = (const void*)k_sweep<P, SAMPLED>;
    const size_t smem = sizeof(SweepSmem<TGRID>);
    WTRI_TRY(smem_optin(fn, (int)smem, done));
    DevGraph g = G;
    Query qq = q;
    Out oo = o;
    void* args[] = {&g, &qq, &oo};
    WTRI_CUDA(cudaLaunchCooperativeKernel(fn, dim3(sweep_blocks<P>(G.m)), dim3(TGRID), args, smem, s));
    return WTRI_OK;
}

// The ranking alone, of candidates already collected (k <= SORT_MAX): one
// block, no other has to be resident.
template <int P>
__global__ void __launch_bounds__(TGRID, 1) k_finish(Query q, Out o) {
    extern __shared__ __align__(16) unsigned char sweep_smem[];
    SweepSmem<TGRID>& S = *reinterpret_cast<SweepSmem<TGRID>*>(sweep_smem);
    BlockTeam<TGRID> T;
    finish<P>(q, o, T, S.sel, S.sort);
}

template <int P>
int launch_finish(const DevGraph& G, const Query& q, const Out& o, cudaStream_t s) {
    if (q.k > SORT_MAX) return launch_sweep<P, false>(G, q, o, s);  // (no rounds: q.total = 0)
    static std::atomic<uint64_t> done{0};
    const size_t smem = sizeof(SweepSmem<TGRID>);
    WTRI_TRY(smem_optin((const void*)k_finish<P>, (int)smem, done));
    k_finish<P><<<1, TGRID, smem, s>>>(q, o);
    WTRI_CUDA(cudaGetLastError());
    return WTRI_OK;
}

// Scratch of one query: bytes, and the pieces carved from a 256-byte aligned
// block (every piece starts 256-byte aligned).
inline size_t query_scratch_bytes(uint32_t cap, int64_t item_cap) {
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    return al(sizeof(QState)) + al((size_t)cap * 8) + al((size_t)cap * 16) + al((size_t)item_cap * sizeof(Item)) +
           al((size_t)item_cap * 8);
}
inline char* query_carve(Query& q, char* p, uint32_t cap, int64_t item_cap) {
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    q = Query{};
    q.st = (QState*)p;
    p += al(sizeof(QState));
    q.ckey = (unsigned long long*)p;
    p += al((size_t)cap * 8);
    q.ctri = (int4*)p;
    p += al((size_t)cap * 16);
    q.items = (Item*)p;
    p += al((size_t)item_cap * sizeof(Item));
    q.ibase = (unsigned long long*)p;
    p += al((size_t)item_cap * 8);
    q.cap = cap;
    q.item_cap = item_cap;
    q.nshards = 1;
    q.wait_first = q.wait_later = WAIT_LIMIT;
    return p;
}
// Items of a graph's query: at most one per edge of a round.
inline int64_t query_items(int64_t m) { return std::min<int64_t>(ITEM_CAP, std::max<int64_t>(m, 256)); }

}  // namespace
}  // namespace wtri
