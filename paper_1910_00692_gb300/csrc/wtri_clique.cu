// Top weighted 4- and 5-cliques by edge sampling (Section 4.5, Appendix A).
//
// A q-clique weighs the p-mean of its q(q-1)/2 edge weights (Appendix A).
// Its key, exact and monotone in that mean, is the minimum, sum, sum of
// squares or maximum of the edge weights (p = -inf, 1, 2, +inf).  Edge
// sampling draws edges with probability proportional to w^p (Algorithm 3:
// the draws of wtri_sample_edges) and enumerates every q-clique on a drawn
// edge (Section 4.5); with every edge taken instead of draws the answer is
// the exact top-k.
//
// A clique is reported by its first drawn edge in the edge order.  Per drawn
// edge r = {u, v} (one block), the common neighbours c of u and v (the shorter
// weight-sorted row is scanned, the other endpoint looked up in the oriented
// rows) are kept unless {u, c} or {v, c} is drawn and earlier than r: a clique
// through such a c belongs to that edge.  Likewise for the edges among them,
// so every clique formed from what is left is reported, once, unchecked.  The
// edges among the kept neighbours come from their oriented rows, scanned once
// against a hash table of the kept ids in shared memory (a search per pair
// took eight dependent loads each, twice, and cost 18.3 ms for the 10,000
// draws of the 979-vertex graph at q = 5; now 0.22 ms for the
// whole enumeration).  q = 4: each such edge closes a
// clique.  q = 5: the edges go to a bit matrix and a list; for each edge
// (i, j) of the list, each l above j adjacent to both closes a clique.  Edges
// that keep more than 128 neighbours go to a second kernel with larger tables,
// those that keep more than 256 to a third that looks pairs up one by one.  On
// large graphs a filter lists the drawn edges that may close a clique at all.
// The whole GPU then selects the candidates that reach the k-th key (a
// histogram per digit of the key, one grid barrier each), one block keeps
// exactly the k best of those under (key desc, sorted vertex tuple asc) by an
// MSB-first radix select over the tuple, and a rank pass orders them.
#include "wtri_query.cuh"

#include <algorithm>

namespace wtri {
namespace {

constexpr int CB = 256;              // threads of a clique block
constexpr int CNB = 1024;            // most common neighbours of one drawn edge
constexpr int CNW = CNB / 32;        // words of a row of the q = 5 bit matrix
constexpr int QMAX = 5;
constexpr int CSB = 1024;            // threads of the select block
constexpr uint32_t CERR_CAND = 1u;   // the candidate buffer filled up
constexpr uint32_t CERR_NBR = 2u;    // a common neighbourhood above CNB
constexpr uint32_t CERR_WAIT = 4u;   // a bounded wait of the selection ran out
constexpr uint32_t CLIQUE_CAP = 1u << 23;

struct CliqueRun {
    const uint32_t* mark;  // drawn edges: bit r = the r-th edge of the edge order
    int32_t q, pcode;
    unsigned long long* ckey;
    int32_t* cids;         // QMAX ids per candidate, ascending
    uint32_t* count;
    uint32_t cap;
    uint32_t* err;
    int32_t* cursor;       // next group of bitmap bits, or of the work list
    int32_t* work;         // the drawn edges that may close a clique (null: the bitmap is walked)
    uint32_t* nwork;
    int32_t* list[2];      // edges left to k_cliques_mid, to k_cliques_big
    uint32_t* nlist;       // their numbers
};

// Shared memory of a clique block; the q = 5 bit matrix (CNB rows of CNW
// words, upper triangle) follows it.
struct CliqueSmem {
    int32_t cid[CNB], cdg[CNB], cwu[CNB], cwv[CNB], cru[CNB], crv[CNB];
    int32_t n;
};

__device__ __forceinline__ bool drawn(const uint32_t* mark, int32_t r) {
    return (__ldg(mark + (r >> 5)) >> (r & 31)) & 1u;
}

__device__ __forceinline__ unsigned long long clique_key(int pcode, const uint32_t* w, int ne) {
    unsigned long long acc = pcode == P_MIN ? ~0ull : 0ull;
    for (int e = 0; e < ne; e++) {
        const unsigned long long x = w[e];
        if (pcode == P_MIN) acc = x < acc ? x : acc;
        else if (pcode == P_ONE) acc += x;
        else if (pcode == P_TWO) acc += x * x;
        else acc = x > acc ? x : acc;
    }
    return acc;
}

// Appends the clique (ids[0..q), edge weights w[0..ne), ranks rk[0..ne),
// rk[0] = r the drawn edge) unless another edge of it is drawn and earlier.
__device__ void emit(const CliqueRun& C, int32_t r, int32_t* ids, const uint32_t* w, const int32_t* rk,
                     int ne) {
    for (int e = 1; e < ne; e++)
        if (rk[e] < r && drawn(C.mark, rk[e])) return;
    const unsigned long long key = clique_key(C.pcode, w, ne);
    for (int a = 1; a < C.q; a++)
        for (int b = a; b > 0 && ids[b - 1] > ids[b]; b--) {
            const int32_t t = ids[b];
            ids[b] = ids[b - 1];
            ids[b - 1] = t;
        }
    const uint32_t idx = atomicAdd(C.count, 1u);
    if (idx >= C.cap) {
        atomicOr(C.err, CERR_CAND);
        return;
    }
    C.ckey[idx] = key;
    for (int a = 0; a < QMAX; a++) C.cids[(size_t)idx * QMAX + a] = a < C.q ? ids[a] : 0;
}

__device__ void clique_edge(const DevGraph& G, const CliqueRun& C, CliqueSmem& S, uint32_t* bits, int32_t r,
                            Tally& tb) {
    const int32_t u = __ldg(G.ord_u + r), v = __ldg(G.ord_v + r);
    const uint32_t wuv = (uint32_t)__ldg(G.ord_w + r);
    const int64_t bu = __ldg(G.rowptr + u), eu = __ldg(G.rowptr + u + 1);
    const int64_t bv = __ldg(G.rowptr + v), ev = __ldg(G.rowptr + v + 1);
    const bool xu = (eu - bu) <= (ev - bv);  // scan the shorter row
    const int32_t y = xu ? v : u;
    const int64_t bx = xu ? bu : bv, ex = xu ? eu : ev;
    const int64_t dy = xu ? ev - bv : eu - bu;
    if (threadIdx.x == 0) S.n = 0;
    __syncthreads();
    for (int64_t j = bx + threadIdx.x; j < ex; j += CB) {
        const int32_t c = __ldg(G.wcol + j);
        if (c == y) continue;
        int32_t wyc, ryc;
        if (!probe_oriented(G, y, dy, c, wyc, ryc, tb)) continue;
        const int idx = atomicAdd(&S.n, 1);
        if (idx >= CNB) {
            atomicOr(C.err, CERR_NBR);
            continue;
        }
        const int32_t wxc = __ldg(G.wwt + j), rxc = __ldg(G.wrk + j);
        S.cid[idx] = c;
        S.cdg[idx] = (int32_t)(__ldg(G.rowptr + c + 1) - __ldg(G.rowptr + c));
        S.cwu[idx] = xu ? wxc : wyc;
        S.cwv[idx] = xu ? wyc : wxc;
        S.cru[idx] = xu ? rxc : ryc;
        S.crv[idx] = xu ? ryc : rxc;
    }
    __syncthreads();
    const int nc = S.n;
    if (nc > CNB) {  // recorded as an error; the call fails
        __syncthreads();
        return;
    }
    if (C.q == 4) {
        for (int i = 0; i < nc; i++)
            for (int j = i + 1 + threadIdx.x; j < nc; j += CB) {
                int32_t wij, rij;
                if (!probe_oriented(G, S.cid[i], S.cdg[i], S.cid[j], wij, rij, tb)) continue;
                int32_t ids[QMAX] = {u, v, S.cid[i], S.cid[j], 0};
                const uint32_t w[6] = {wuv, (uint32_t)S.cwu[i], (uint32_t)S.cwv[i],
                                       (uint32_t)S.cwu[j], (uint32_t)S.cwv[j], (uint32_t)wij};
                const int32_t rk[6] = {r, S.cru[i], S.crv[i], S.cru[j], S.crv[j], rij};
                emit(C, r, ids, w, rk, 6);
            }
    } else {
        const int nw = (nc + 31) >> 5;
        for (int t = threadIdx.x; t < nc * nw; t += CB) bits[(t / nw) * CNW + t % nw] = 0u;
        __syncthreads();
        for (int i = 0; i < nc; i++)
            for (int j = i + 1 + threadIdx.x; j < nc; j += CB) {
                int32_t wij, rij;
                if (probe_oriented(G, S.cid[i], S.cdg[i], S.cid[j], wij, rij, tb))
                    atomicOr(&bits[i * CNW + (j >> 5)], 1u << (j & 31));
            }
        __syncthreads();
        for (int i = 0; i < nc; i++)
            for (int j = i + 1 + threadIdx.x; j < nc; j += CB) {
                if (!((bits[i * CNW + (j >> 5)] >> (j & 31)) & 1u)) continue;
                int32_t wij = 0, rij = 0;
                probe_oriented(G, S.cid[i], S.cdg[i], S.cid[j], wij, rij, tb);
                for (int wd = (j + 1) >> 5; wd < nw; wd++) {
                    uint32_t both = bits[i * CNW + wd] & bits[j * CNW + wd];
                    if (wd == ((j + 1) >> 5)) both &= ~0u << ((j + 1) & 31);  // l > j
                    while (both) {
                        const int l = wd * 32 + __ffs(both) - 1;
                        both &= both - 1;
                        int32_t wil = 0, ril = 0, wjl = 0, rjl = 0;
                        probe_oriented(G, S.cid[i], S.cdg[i], S.cid[l], wil, ril, tb);
                        probe_oriented(G, S.cid[j], S.cdg[j], S.cid[l], wjl, rjl, tb);
                        int32_t ids[QMAX] = {u, v, S.cid[i], S.cid[j], S.cid[l]};
                        const uint32_t w[10] = {wuv,
                                                (uint32_t)S.cwu[i], (uint32_t)S.cwv[i],
                                                (uint32_t)S.cwu[j], (uint32_t)S.cwv[j],
                                                (uint32_t)S.cwu[l], (uint32_t)S.cwv[l],
                                                (uint32_t)wij, (uint32_t)wil, (uint32_t)wjl};
                        const int32_t rk[10] = {r, S.cru[i], S.crv[i], S.cru[j], S.crv[j],
                                                S.cru[l], S.crv[l], rij, ril, rjl};
                        emit(C, r, ids, w, rk, 10);
                    }
                }
            }
    }
    __syncthreads();  // the shared lists are reused by the next edge
}

// The edges that keep more common neighbours than the tables of k_cliques_mid.
__global__ void __launch_bounds__(CB) k_cliques_big(DevGraph G, CliqueRun C) {
    extern __shared__ __align__(16) unsigned char csm[];
    CliqueSmem& S = *reinterpret_cast<CliqueSmem*>(csm);
    uint32_t* bits = reinterpret_cast<uint32_t*>(csm + sizeof(CliqueSmem));
    Tally tb;
    const uint32_t n = C.nlist[1];
    for (uint32_t i = blockIdx.x; i < n; i += gridDim.x) clique_edge(G, C, S, bits, C.list[1][i], tb);
}

// ---- edges with at most FNB kept neighbours --------------------------------
// Two sizes: FNB = 128 (54 KB of shared memory: three 256-thread blocks per
// SM), and FNB = 256 (208 KB: one 1,024-thread block) for the few edges that
// keep more.
constexpr int FGROUP = 4;          // bitmap bits taken at a time

template <int FNB>
struct FastSmem {
    static constexpr int HASH = 4 * FNB;    // slots of the id table (at most a quarter used)
    uint32_t wm[FNB * (FNB - 1) / 2];       // q = 5: weight of the edge (i, j), i < j, at j (j - 1) / 2 + i;
                                            // q = 4: weight of each edge of the list
    uint16_t pair[FNB * (FNB - 1) / 2];     // the edges, i << 8 | j
    uint32_t bits[FNB][FNB / 32];           // row i: adjacent j > i
    int32_t hid[HASH];                      // ids (-1: free) and their places
    uint8_t hix[HASH];
    int32_t cid[FNB], cwu[FNB], cwv[FNB];
    uint32_t wsum[32];
    uint32_t base;
    int32_t all, n, np, item;
};

// The key with another edge: acc with w added (minimum, sum, squares, maximum).
template <int PC>
__device__ __forceinline__ unsigned long long more(unsigned long long acc, uint32_t w) {
    const unsigned long long x = w;
    if (PC == P_MIN) return x < acc ? x : acc;
    if (PC == P_ONE) return acc + x;
    if (PC == P_TWO) return acc + x * x;
    return x > acc ? x : acc;
}

// Candidate idx of a clique that is known to belong to the edge at hand.
__device__ __forceinline__ void put(const CliqueRun& C, uint32_t idx, int32_t a, int32_t b, int32_t c, int32_t d,
                                    int32_t e, int q, unsigned long long key) {
    if (idx >= C.cap) {
        atomicOr(C.err, CERR_CAND);
        return;
    }
    auto sw = [](int32_t& x, int32_t& y) {
        const int32_t lo = min(x, y), hi = max(x, y);
        x = lo;
        y = hi;
    };
    if (q == 5) {  // sorting networks
        sw(a, d), sw(b, e), sw(a, c), sw(b, d), sw(a, b), sw(c, e), sw(b, c), sw(d, e), sw(c, d);
    } else {
        sw(a, c), sw(b, d), sw(a, b), sw(c, d), sw(b, c);
    }
    C.ckey[idx] = key;
    int32_t* o = C.cids + (size_t)idx * QMAX;
    o[0] = a;
    o[1] = b;
    o[2] = c;
    o[3] = d;
    o[4] = q == 5 ? e : 0;
}

template <int Q, int PC, int FNB, int NTH>
__device__ __forceinline__ void fast_edge(const DevGraph& G, const CliqueRun& C, FastSmem<FNB>& S, int32_t r,
                                          int32_t* left, uint32_t* nleft) {
    constexpr int HASH = FastSmem<FNB>::HASH, HSHIFT = FNB == 128 ? 23 : 22, FNW = FNB / 32;
    static_assert(HASH == 1 << (32 - HSHIFT), "the hash fills the table");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    Tally tb;
    const int32_t u = __ldg(G.ord_u + r), v = __ldg(G.ord_v + r);
    const uint32_t wuv = (uint32_t)__ldg(G.ord_w + r);
    const int64_t bu = __ldg(G.rowptr + u), eu = __ldg(G.rowptr + u + 1);
    const int64_t bv = __ldg(G.rowptr + v), ev = __ldg(G.rowptr + v + 1);
    const bool xu = (eu - bu) <= (ev - bv);  // scan the shorter row
    const int32_t y = xu ? v : u;
    const int64_t bx = xu ? bu : bv, ex = xu ? eu : ev;
    const int64_t dy = xu ? ev - bv : eu - bu;
    if (threadIdx.x == 0) S.all = S.n = S.np = 0;
    for (int t = threadIdx.x; t < HASH; t += NTH) S.hid[t] = -1;
    if (Q == 5)
        for (int t = threadIdx.x; t < FNB * FNW; t += NTH) (&S.bits[0][0])[t] = 0u;
    __syncthreads();
    for (int64_t j = bx + threadIdx.x; j < ex; j += NTH) {
        const int32_t c = __ldg(G.wcol + j);
        if (c == y) continue;
        int32_t wyc, ryc;
        if (!probe_oriented(G, y, dy, c, wyc, ryc, tb)) continue;
        atomicAdd(&S.all, 1);
        const int32_t rxc = __ldg(G.wrk + j);
        if ((rxc < r && drawn(C.mark, rxc)) || (ryc < r && drawn(C.mark, ryc))) continue;
        const int i = atomicAdd(&S.n, 1);
        if (i >= FNB) continue;
        const int32_t wxc = __ldg(G.wwt + j);
        S.cid[i] = c;
        S.cwu[i] = xu ? wxc : wyc;
        S.cwv[i] = xu ? wyc : wxc;
        uint32_t h = ((uint32_t)c * 2654435761u) >> HSHIFT;
        while (atomicCAS(&S.hid[h], -1, c) != -1) h = (h + 1) & (HASH - 1);  // ids are distinct
        S.hix[h] = (uint8_t)i;
    }
    __syncthreads();
    const int nc = S.n;
    if (S.all > CNB) {  // recorded as an error; the call fails
        if (threadIdx.x == 0) atomicOr(C.err, CERR_NBR);
        return;
    }
    if (nc > FNB) {
        if (threadIdx.x == 0) left[atomicAdd(nleft, 1u)] = r;
        return;
    }
    if (nc < Q - 2) return;
    auto edge = [&](int i, int j, int64_t at) {  // an edge among the kept neighbours, entry `at`
        const int32_t rij = __ldg(G.ork + at);
        if (rij < r && drawn(C.mark, rij)) return;
        const uint32_t wij = (uint32_t)__ldg(G.owt + at);
        const int a = min(i, j), b = max(i, j), t = atomicAdd(&S.np, 1);
        S.pair[t] = (uint16_t)(a << 8 | b);
        if constexpr (Q == 4) {
            S.wm[t] = wij;
        } else {
            S.wm[b * (b - 1) / 2 + a] = wij;
            atomicOr(&S.bits[a][b >> 5], 1u << (b & 31));
        }
    };
    for (int i = wid; i < nc; i += NTH / 32) {  // a warp per kept neighbour
        const int32_t c = S.cid[i];
        const int64_t ob = __ldg(G.orowptr + c), oe = __ldg(G.orowptr + c + 1);
        // its row against the table, unless that is long against nc searches of it
        // (10,000 draws of the 979-vertex graph, q = 5: rows only 0.44 ms as now,
        // searches only 0.53; hubs have rows of tens of thousands)
        if (oe - ob <= 64 + 8 * (int64_t)nc) {
            for (int64_t at = ob + lane; at < oe; at += 32) {
                const int32_t x = __ldg(G.ocol + at);
                uint32_t h = ((uint32_t)x * 2654435761u) >> HSHIFT;
                int32_t id = S.hid[h];
                while (id != -1 && id != x) id = S.hid[h = (h + 1) & (HASH - 1)];
                if (id == x) edge(i, S.hix[h], at);
            }
        } else {  // a long row: each kept neighbour searched in it
            for (int j = lane; j < nc; j += 32) {
                const int64_t at = search_ids(G.ocol, ob, (int32_t)(oe - ob), S.cid[j], tb);
                if (at < oe && __ldg(G.ocol + at) == S.cid[j]) edge(i, j, at);
            }
        }
    }
    __syncthreads();
    // every thread counts its cliques, the block takes their places at once
    // (an atomic round trip per clique made the heaviest edge the tail)
    const int np = S.np;
    auto common = [&](int i, int j, int wd) { return S.bits[i][wd] & S.bits[j][wd]; };  // (row j holds l > j only)
    uint32_t mine = 0;
    for (int t = threadIdx.x; t < np; t += NTH) {
        if (Q == 4) {
            mine++;
        } else {
            const int i = S.pair[t] >> 8, j = S.pair[t] & 255;
            for (int wd = j >> 5; wd < FNW; wd++) mine += __popc(common(i, j, wd));
        }
    }
    uint32_t inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += x;
    }
    if (lane == 31) S.wsum[wid] = inc;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t acc = 0;
        for (int k = 0; k < NTH / 32; k++) {
            const uint32_t c = S.wsum[k];
            S.wsum[k] = acc;
            acc += c;
        }
        if (acc) S.base = atomicAdd(C.count, acc);
    }
    __syncthreads();
    uint32_t idx = S.base + S.wsum[wid] + inc - mine;
    const unsigned long long k0 = more<PC>(PC == P_MIN ? ~0ull : 0ull, wuv);
    for (int t = threadIdx.x; t < np; t += NTH) {
        const int i = S.pair[t] >> 8, j = S.pair[t] & 255;
        unsigned long long kij = more<PC>(more<PC>(k0, S.cwu[i]), S.cwv[i]);
        kij = more<PC>(more<PC>(kij, S.cwu[j]), S.cwv[j]);
        if constexpr (Q == 4) {
            put(C, idx++, u, v, S.cid[i], S.cid[j], 0, 4, more<PC>(kij, S.wm[t]));
        } else {
            kij = more<PC>(kij, S.wm[j * (j - 1) / 2 + i]);
            for (int wd = j >> 5; wd < FNW; wd++) {
                uint32_t both = common(i, j, wd);
                while (both) {
                    const int l = wd * 32 + __ffs(both) - 1;
                    both &= both - 1;
                    unsigned long long k = more<PC>(more<PC>(kij, S.cwu[l]), S.cwv[l]);
                    k = more<PC>(more<PC>(k, S.wm[l * (l - 1) / 2 + i]), S.wm[l * (l - 1) / 2 + j]);
                    put(C, idx++, u, v, S.cid[i], S.cid[j], S.cid[l], 5, k);
                }
            }
        }
    }
}

// Large graphs: the drawn edges with enough kept common neighbours for a clique,
// to the work list.  A warp takes a word of the bitmap; the entries of its
// edges' shorter rows are numbered through and looked up 32 at a time, as the
// blocks below do it.  Rows above FILTER_ROW go to the list as they are (64: all
// edges of the graph below take 32 ms).  Blocks that walk the bitmap a few bits
// at a time and clear their tables for every drawn edge took 8.3 ms for 100 draws
// from 2e7 edges on 2e6 vertices and 187 ms for all of them (q = 4, k = 1,000);
// with the list 0.18 and 16.  Small graphs walk: q = 5, 10,000 draws from 29,000
// edges 0.41 ms, 0.58 with the list; from 100,000 edges 0.45 and 0.57.
constexpr int64_t WALK_MAX = 1 << 17;    // most edges whose bitmap is walked
constexpr int64_t FILTER_ROW = 256;

static_assert(3 * (sizeof(FastSmem<128>) + 1024) <= 228 * 1024, "three small-table blocks per SM");

struct FilterWarp {
    int64_t j0[32];
    uint32_t end[32], cnt[32];  // entries up to and with each row; neighbours kept
    int32_t r[32], y[32], dy[32];
};

template <int Q>
__global__ void __launch_bounds__(CB) k_clique_edges(DevGraph G, CliqueRun C) {
    __shared__ FilterWarp shared[CB / 32];
    FilterWarp& W = shared[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t words = (G.m + 31) / 32, nwarps = ((int64_t)gridDim.x * CB) >> 5;
    Tally tb;
    for (int64_t w = ((int64_t)blockIdx.x * CB + threadIdx.x) >> 5; w < words; w += nwarps) {
        const uint32_t bits = __ldg(C.mark + w);
        if (!bits) continue;
        const int32_t r = (int32_t)(32 * w + lane);
        int64_t n = 0;
        W.cnt[lane] = 0;
        W.r[lane] = r;
        if ((bits >> lane) & 1u) {
            const int32_t u = __ldg(G.ord_u + r), v = __ldg(G.ord_v + r);
            const int64_t bu = __ldg(G.rowptr + u), eu = __ldg(G.rowptr + u + 1);
            const int64_t bv = __ldg(G.rowptr + v), ev = __ldg(G.rowptr + v + 1);
            const bool xu = (eu - bu) <= (ev - bv);  // scan the shorter row
            n = xu ? eu - bu : ev - bv;
            W.j0[lane] = xu ? bu : bv;
            W.y[lane] = xu ? v : u;
            W.dy[lane] = (int32_t)(xu ? ev - bv : eu - bu);
        }
        bool keep = n > FILTER_ROW;
        uint32_t inc = keep || n < Q - 1 ? 0u : (uint32_t)n;  // (a clique takes Q - 1 entries of the row)
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += x;
        }
        W.end[lane] = inc;
        const uint32_t tot = __shfl_sync(0xffffffffu, inc, 31);
        __syncwarp();
        for (uint32_t e = lane; e < tot; e += 32) {
            int k = 0;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1)
                if (W.end[k + s - 1] <= e) k += s;
            const int64_t j = W.j0[k] + (e - (k > 0 ? W.end[k - 1] : 0u));
            const int32_t c = __ldg(G.wcol + j), y = W.y[k], rk = W.r[k];
            int32_t wyc, ryc;
            if (c == y || !probe_oriented(G, y, W.dy[k], c, wyc, ryc, tb)) continue;
            const int32_t rxc = __ldg(G.wrk + j);
            if ((rxc < rk && drawn(C.mark, rxc)) || (ryc < rk && drawn(C.mark, ryc))) continue;
            atomicAdd(&W.cnt[k], 1u);
        }
        __syncwarp();
        keep |= W.cnt[lane] >= Q - 2;
        const uint32_t b = __ballot_sync(0xffffffffu, keep);
        uint32_t at = 0;
        if (lane == 0 && b) at = atomicAdd(C.nwork, (uint32_t)__popc(b));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (keep) C.work[at + __popc(b & lanemask_below())] = r;
        __syncwarp();
    }
}

// The drawn edges: the work list one by one, or a few bitmap bits at a time.
template <int Q, int PC>
__global__ void __launch_bounds__(CB, 3) k_cliques(DevGraph G, CliqueRun C) {
    extern __shared__ __align__(16) unsigned char csm[];
    FastSmem<128>& S = *reinterpret_cast<FastSmem<128>*>(csm);
    const bool list = C.work != nullptr;
    const int64_t n = list ? (int64_t)*C.nwork : G.m, group = list ? 1 : FGROUP;
    for (;;) {
        if (threadIdx.x == 0) S.item = atomicAdd(C.cursor, 1);
        __syncthreads();
        const int64_t i0 = (int64_t)S.item * group;
        __syncthreads();
        if (i0 >= n) break;
        for (int64_t i = i0; i < min(n, i0 + group); i++) {
            const int32_t r = list ? C.work[i] : (int32_t)i;
            if (!list && !drawn(C.mark, r)) continue;
            fast_edge<Q, PC, 128, CB>(G, C, S, r, C.list[0], C.nlist);
            __syncthreads();  // the shared lists are reused by the next edge
        }
    }
}

// The edges that keep more than 128.
template <int Q, int PC>
__global__ void __launch_bounds__(1024, 1) k_cliques_mid(DevGraph G, CliqueRun C) {
    extern __shared__ __align__(16) unsigned char csm[];
    FastSmem<256>& S = *reinterpret_cast<FastSmem<256>*>(csm);
    const uint32_t n = C.nlist[0];
    for (uint32_t i = blockIdx.x; i < n; i += gridDim.x) {
        fast_edge<Q, PC, 256, 1024>(G, C, S, C.list[0][i], C.list[1], C.nlist + 1);
        __syncthreads();
    }
}

// Every edge drawn: all bits of the first m positions.
__global__ void k_mark_all(int64_t m, uint32_t* mark) {
    const int64_t words = (m + 31) / 32;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t left = m - 32 * i;
        mark[i] = left >= 32 ? ~0u : ((1u << left) - 1u);
    }
}

// ---- selection of the k best candidates ------------------------------------
// The candidates whose key reaches the K-th largest (ties included), by the
// whole GPU: their indices to ix, their number to *nix.  hist: SEL_BINS
// counters per digit, and lim[2] (largest key, complement of the smallest),
// all zero at the start.
struct CliqueSelect {
    Query q;  // barrier state
    const unsigned long long* ckey;
    const uint32_t* count;
    uint32_t cap, K;
    uint32_t* err;
    uint32_t* hist;
    unsigned long long* lim;
    uint32_t* ix;
    uint32_t* nix;
};

__global__ void __launch_bounds__(TGRID, 1) k_clique_reach(CliqueSelect A) {
    __shared__ SelectSmem S;
    const int tid = threadIdx.x, lane = tid & 31;
    // one thread reads the error word: a block that gives up below sets it,
    // maybe before this one has started
    if (tid == 0) S.err = *(volatile const uint32_t*)A.err;
    __syncthreads();
    if (S.err) return;
    const uint32_t n = min(*(volatile const uint32_t*)A.count, A.cap);
    GridTeam<TGRID> T;
    T.limit = A.q.wait_first;
    T.blk0 = 0;
    T.nblk = gridDim.x;
    T.gone = &S.gone;
    if (tid == 0) S.gone = 0;
    __syncthreads();
    const uint32_t step = (uint32_t)T.threads();
    auto wait = [&]() {
        if (T.sync(A.q)) return true;
        if (tid == 0) atomicOr(A.err, CERR_WAIT);
        return false;
    };
    unsigned long long reach = 0;  // n <= K: all of them
    if (n > A.K) {
        unsigned long long mx = 0, mn = ~0ull;
        for (uint32_t i = (uint32_t)T.thread(); i < n; i += step) {
            const unsigned long long x = A.ckey[i];
            mx = x > mx ? x : mx;
            mn = x < mn ? x : mn;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long a = __shfl_xor_sync(0xffffffffu, mx, o), b = __shfl_xor_sync(0xffffffffu, mn, o);
            mx = a > mx ? a : mx;
            mn = b < mn ? b : mn;
        }
        if (lane == 0 && mx) {
            atomicMax(A.lim, mx);
            atomicMax(A.lim + 1, ~mn);
        }
        if (!wait()) return;
        mx = ld_volatile_u64(A.lim);
        mn = ~ld_volatile_u64(A.lim + 1);
        int shift = mx == mn ? 0 : 64 - __clzll((long long)(mx ^ mn));
        reach = shift >= 64 ? 0ull : (mx >> shift) << shift;
        uint32_t need = A.K;
        for (int dig = 0; shift > 0; dig++) {
            const int bits = shift < SEL_BITS ? shift : SEL_BITS, hi = shift;
            shift -= bits;
            const uint32_t mask = (1u << bits) - 1u;
            uint32_t* gh = A.hist + dig * SEL_BINS;
            clear_hist<TGRID>(T.part, S);
            for (uint32_t base = (uint32_t)(T.thread() - lane); base < n; base += step) {
                const uint32_t i = base + lane;
                uint32_t d = SEL_BINS;
                if (i < n) {
                    const unsigned long long x = A.ckey[i];
                    if (hi >= 64 || (x >> hi) == (reach >> hi)) d = mask - ((uint32_t)(x >> shift) & mask);
                }
                count_bin(S, d);
            }
            __syncthreads();
            for (int b = tid; b < SEL_BINS; b += TGRID)
                if (S.hist[b]) atomicAdd(gh + b, S.hist[b]);
            if (!wait()) return;
            for (int b = tid; b < SEL_BINS; b += TGRID) S.hist[b] = *(volatile uint32_t*)(gh + b);
            __syncthreads();
            pick_bin<TGRID>(T.part, S, need);
            reach |= (unsigned long long)(mask - S.bin) << shift;
            need -= S.above;
            __syncthreads();
        }
    }
    for (uint32_t base = (uint32_t)(T.thread() - lane); base < n; base += step) {
        const uint32_t i = base + lane;
        const bool on = i < n && A.ckey[i] >= reach;
        const uint32_t b = __ballot_sync(0xffffffffu, on);
        uint32_t at = 0;
        if (lane == 0 && b) at = atomicAdd(A.nix, (uint32_t)__popc(b));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (on) A.ix[at + __popc(b & lanemask_below())] = i;
    }
}

// Tuple of a candidate, smaller is better: (~key_hi, ~key_lo, id_0 .. id_{q-1}).
__device__ __forceinline__ uint32_t cword(const unsigned long long* ckey, const int32_t* cids, uint32_t i,
                                          int wi) {
    if (wi == 0) return ~(uint32_t)(ckey[i] >> 32);
    if (wi == 1) return ~(uint32_t)ckey[i];
    return (uint32_t)cids[(size_t)i * QMAX + (wi - 2)];
}

struct CSelSmem {
    uint32_t hist[256];
    uint32_t pw[2 + QMAX];
    uint32_t below, eq, done, kept;
    uint32_t warp_cnt[CSB / 32];
};

// <0, 0, >0: the first `depth` bytes of candidate i's tuple against pw.
__device__ __forceinline__ int cmp_cprefix(const unsigned long long* ckey, const int32_t* cids, uint32_t i,
                                           const uint32_t* pw, int depth) {
    const int full = depth >> 2, rem = depth & 3;
    for (int wi = 0; wi < full; wi++) {
        const uint32_t a = cword(ckey, cids, i, wi);
        if (a != pw[wi]) return a < pw[wi] ? -1 : 1;
    }
    if (rem) {
        const uint32_t mask = 0xffffffffu << (32 - 8 * rem);
        const uint32_t a = cword(ckey, cids, i, full) & mask, b = pw[full] & mask;
        if (a != b) return a < b ? -1 : 1;
    }
    return 0;
}

// Keeps the indices of exactly min(K, n) best candidates at the front of ix
// (tuples are unique: every clique appears once), n = *nix; *kept receives
// their number.
__global__ void __launch_bounds__(CSB) k_clique_select(const unsigned long long* ckey, const int32_t* cids,
                                                       uint32_t* ix, const uint32_t* nix, int q, uint32_t K,
                                                       const uint32_t* err, uint32_t* kept) {
    __shared__ CSelSmem S;
    if (*(volatile const uint32_t*)err) return;
    const uint32_t n = *(volatile const uint32_t*)nix;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nbytes = 4 * (2 + q);
    if (tid < 2 + QMAX) S.pw[tid] = 0;
    if (tid == 0) {
        S.below = 0;
        S.eq = n;
        S.done = n <= K ? 1u : 0u;
    }
    __syncthreads();
    int depth = 0;
    while (!S.done && depth < nbytes) {
        for (int i = tid; i < 256; i += CSB) S.hist[i] = 0;
        __syncthreads();
        const int wi = depth >> 2, sh = 24 - 8 * (depth & 3);
        for (uint32_t t = tid; t < n; t += CSB) {
            const uint32_t i = ix[t];
            if (cmp_cprefix(ckey, cids, i, S.pw, depth) == 0)
                atomicAdd(&S.hist[(cword(ckey, cids, i, wi) >> sh) & 255u], 1u);
        }
        __syncthreads();
        if (wid == 0) {  // the bin where the running count reaches what is needed: eight bins a lane
            const uint32_t need = K - S.below;
            uint32_t h[8], sum = 0;
#pragma unroll
            for (int b = 0; b < 8; b++) sum += h[b] = S.hist[8 * lane + b];
            uint32_t acc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, acc, o);
                if (lane >= o) acc += y;
            }
            acc -= sum;
            __syncwarp();
            if (acc < need && need <= acc + sum) {
                bool hit = false;
#pragma unroll
                for (int b = 0; b < 8; b++) {
                    if (!hit && need <= acc + h[b]) {
                        hit = true;
                        S.below += acc;
                        S.eq = h[b];
                        S.pw[wi] |= (uint32_t)(8 * lane + b) << sh;
                        if (S.below + S.eq == K) S.done = 1;
                    }
                    acc += h[b];
                }
            }
        }
        __syncthreads();
        depth++;
    }
    const bool keep_all = n <= K;
    uint32_t out = 0;
    for (uint32_t base = 0; base < n; base += CSB) {
        const uint32_t t = base + tid;
        bool keep = false;
        uint32_t i = 0;
        if (t < n) {
            i = ix[t];
            keep = keep_all || cmp_cprefix(ckey, cids, i, S.pw, depth) <= 0;
        }
        const uint32_t b = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) S.warp_cnt[wid] = __popc(b);
        __syncthreads();
        if (tid == 0) {
            uint32_t acc = 0;
            for (int wv = 0; wv < CSB / 32; wv++) {
                const uint32_t c = S.warp_cnt[wv];
                S.warp_cnt[wv] = acc;
                acc += c;
            }
            S.kept = acc;
        }
        __syncthreads();
        if (keep) {
            const uint32_t p = out + S.warp_cnt[wid] + __popc(b & ((1u << lane) - 1u));
            ix[p] = i;  // p <= t: this chunk was read before the barrier
        }
        out += S.kept;
        __syncthreads();
    }
    if (tid == 0) *kept = out;
}

// Whether candidate a ranks before candidate b.
__device__ __forceinline__ bool cbefore(const unsigned long long* ckey, const int32_t* cids, uint32_t a,
                                        uint32_t b, int q) {
    if (ckey[a] != ckey[b]) return ckey[a] > ckey[b];
    for (int i = 0; i < q; i++) {
        const int32_t x = cids[(size_t)a * QMAX + i], y = cids[(size_t)b * QMAX + i];
        if (x != y) return x < y;
    }
    return false;
}

// One warp per kept candidate: its rank among the kept ones, then the
// outputs at that rank (ids, fp64 mean, key).
__global__ void k_clique_rank(const unsigned long long* ckey, const int32_t* cids, const uint32_t* ix,
                              const uint32_t* kept,
                              const uint32_t* err, int q, int pcode, uint32_t kmax, int32_t* ids_out,
                              double* w_out, unsigned long long* key_out) {
    if (*(volatile const uint32_t*)err) return;
    const uint32_t K = *kept;
    const uint32_t at = (uint32_t)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (at >= K) return;
    const uint32_t i = ix[at];
    uint32_t rank = 0;
    for (uint32_t j = lane; j < K; j += 32) rank += cbefore(ckey, cids, ix[j], i, q) ? 1u : 0u;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (lane == 0 && rank < kmax) {
        const unsigned long long key = ckey[i];
        const double ne = (double)(q * (q - 1) / 2);
        for (int a = 0; a < q; a++) ids_out[(size_t)rank * q + a] = cids[(size_t)i * QMAX + a];
        w_out[rank] = pcode == P_ONE ? (double)key / ne : (pcode == P_TWO ? sqrt((double)key / ne) : (double)key);
        key_out[rank] = key;
    }
}

}  // namespace

int clique_topk_host(const wtri_graph* g, int q, int pcode, int32_t k, int64_t nsamples, uint64_t seed,
                     int32_t* h_ids, double* h_w, uint64_t* h_keys, int32_t* h_count) {
    const DevGraph& G = g->d;
    const int64_t m = G.m;
    const int64_t words = (m + 31) / 32;
    const uint32_t cap = CLIQUE_CAP;
    cudaStream_t s = g->stream;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    // cleared at the start: counters, key limits, barrier state, histograms
    // (six digits of a 64-bit key)
    const size_t small_bytes = 256 + 256 + al(sizeof(QState)) + 6 * SEL_BINS * 4;
    const int64_t big_cap = nsamples < 0 ? m : std::min(m, nsamples);  // at most the drawn edges
    const size_t bytes = al(4 * (size_t)words) + al((size_t)cap * 8) + al((size_t)cap * 4 * QMAX) +
                         al((size_t)k * (4 * q + 16)) + al((size_t)cap * 4) + 2 * al(4 * (size_t)big_cap) + small_bytes;
    void* buf = nullptr;
    if (cudaMallocAsync(&buf, bytes, s) != cudaSuccess) {
        cudaGetLastError();
        return set_error(WTRI_ENOMEM, "clique scratch allocation failed");
    }
    char* p = (char*)buf;
    uint32_t* mark = (uint32_t*)p;
    p += al(4 * (size_t)words);
    unsigned long long* ckey = (unsigned long long*)p;
    p += al((size_t)cap * 8);
    int32_t* cids = (int32_t*)p;
    p += al((size_t)cap * 4 * QMAX);
    unsigned long long* okey = (unsigned long long*)p;
    double* ow = (double*)(okey + k);
    int32_t* oids = (int32_t*)(ow + k);
    p += al((size_t)k * (4 * q + 16));
    uint32_t* ix = (uint32_t*)p;
    p += al((size_t)cap * 4);
    int32_t* big = (int32_t*)p;
    p += 2 * al(4 * (size_t)big_cap);
    uint32_t* small = (uint32_t*)p;  // count, err, cursor, kept, nix, nlist[2], nwork
    auto done = [&](int rc) {
        cudaFreeAsync(buf, s);
        cudaStreamSynchronize(s);
        return rc;
    };
    if (cudaMemsetAsync(small, 0, small_bytes, s) != cudaSuccess)
        return done(cuda_error(cudaGetLastError(), "memset", __FILE__, __LINE__));
    if (nsamples >= 0) {
        int rc = sample_edges_device(g, pcode, nsamples, seed, mark, s);
        if (rc != WTRI_OK) return done(rc);
    } else {
        k_mark_all<<<std::max<int64_t>(1, std::min<int64_t>((words + 255) / 256, sm_count() * 8)), 256, 0, s>>>(
            m, mark);
    }
    CliqueRun C;
    C.mark = mark;
    C.q = q;
    C.pcode = pcode;
    C.ckey = ckey;
    C.cids = cids;
    C.count = small;
    C.cap = cap;
    C.err = small + 1;
    C.cursor = (int32_t*)(small + 2);
    C.list[0] = big;
    C.list[1] = (int32_t*)((char*)big + al(4 * (size_t)big_cap));
    C.nlist = small + 5;
    // (the work list is read before k_cliques_mid fills list[1])
    C.work = m > WALK_MAX ? C.list[1] : nullptr;
    C.nwork = small + 7;
    const int big_smem = (int)sizeof(CliqueSmem) + (q == 5 ? CNB * CNW * 4 : 0);
    {
        static std::atomic<uint64_t> optin{0};
        int rc = smem_optin((const void*)k_cliques_big, (int)sizeof(CliqueSmem) + CNB * CNW * 4, optin);
        if (rc != WTRI_OK) return done(rc);
    }
    auto enumerate = [&](auto kern, auto mid, std::atomic<uint64_t>* optin) -> int {
        WTRI_TRY(smem_optin((const void*)kern, (int)sizeof(FastSmem<128>), optin[0]));
        WTRI_TRY(smem_optin((const void*)mid, (int)sizeof(FastSmem<256>), optin[1]));
        if (C.work) {
            const unsigned blocks = (unsigned)std::min<int64_t>(sm_count() * 8, (words + CB / 32 - 1) / (CB / 32));
            if (q == 5) k_clique_edges<5><<<blocks, CB, 0, s>>>(G, C);
            else k_clique_edges<4><<<blocks, CB, 0, s>>>(G, C);
        }
        kern<<<sm_count() * 3, CB, sizeof(FastSmem<128>), s>>>(G, C);
        mid<<<sm_count(), 1024, sizeof(FastSmem<256>), s>>>(G, C);
        k_cliques_big<<<sm_count() * (q == 5 ? 1 : 4), CB, big_smem, s>>>(G, C);
        return WTRI_OK;
    };
    {
        ProfScope ps("cliques_enumerate", s, 0.0, C.work ? 4 : 3);
        static std::atomic<uint64_t> optin[8][2];
        int rc = WTRI_OK;
        switch (pcode + (q == 5 ? 4 : 0)) {
            case P_MIN: rc = enumerate(k_cliques<4, P_MIN>, k_cliques_mid<4, P_MIN>, optin[0]); break;
            case P_ONE: rc = enumerate(k_cliques<4, P_ONE>, k_cliques_mid<4, P_ONE>, optin[1]); break;
            case P_TWO: rc = enumerate(k_cliques<4, P_TWO>, k_cliques_mid<4, P_TWO>, optin[2]); break;
            case P_MAX: rc = enumerate(k_cliques<4, P_MAX>, k_cliques_mid<4, P_MAX>, optin[3]); break;
            case 4 + P_MIN: rc = enumerate(k_cliques<5, P_MIN>, k_cliques_mid<5, P_MIN>, optin[4]); break;
            case 4 + P_ONE: rc = enumerate(k_cliques<5, P_ONE>, k_cliques_mid<5, P_ONE>, optin[5]); break;
            case 4 + P_TWO: rc = enumerate(k_cliques<5, P_TWO>, k_cliques_mid<5, P_TWO>, optin[6]); break;
            default: rc = enumerate(k_cliques<5, P_MAX>, k_cliques_mid<5, P_MAX>, optin[7]); break;
        }
        if (rc != WTRI_OK) return done(rc);
    }
    {
        ProfScope ps("cliques_select", s, 0.0, 3);
        CliqueSelect A{};
        A.lim = (unsigned long long*)((char*)small + 256);
        A.q.st = (QState*)((char*)small + 512);
        A.q.wait_first = first_wait_limit();
        A.q.wait_later = later_wait_limit();
        A.hist = (uint32_t*)((char*)small + 512 + al(sizeof(QState)));
        A.ckey = ckey;
        A.count = small;
        A.cap = cap;
        A.K = (uint32_t)k;
        A.err = small + 1;
        A.ix = ix;
        A.nix = small + 4;
        void* args[] = {&A};
        cudaError_t le = cudaLaunchCooperativeKernel((const void*)k_clique_reach, dim3((unsigned)sm_count()),
                                                     dim3(TGRID), args, 0, s);
        if (le != cudaSuccess) return done(cuda_error(le, "clique select", __FILE__, __LINE__));
        k_clique_select<<<1, CSB, 0, s>>>(ckey, cids, ix, small + 4, q, (uint32_t)k, small + 1, small + 3);
        k_clique_rank<<<ceil_div_u(k, 8), 256, 0, s>>>(ckey, cids, ix, small + 3, small + 1, q, pcode,
                                                        (uint32_t)k, oids, ow, okey);
    }
    if (cudaGetLastError() != cudaSuccess)
        return done(set_error(WTRI_ECUDA, "clique kernel launch failed"));
    uint32_t hs[4] = {0, 0, 0, 0};
    cudaError_t e = cudaMemcpyAsync(hs, small, sizeof(hs), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return done(cuda_error(e, "clique results", __FILE__, __LINE__));
    if (hs[1] & CERR_WAIT) return done(set_error(WTRI_ETIMEOUT, "a bounded wait of the clique selection ran out"));
    if (hs[1] & CERR_NBR)
        return done(set_error(WTRI_EUNSUPPORTED, "a drawn edge has more than " + std::to_string(CNB) +
                                                     " common neighbours"));
    if (hs[1] & CERR_CAND)
        return done(set_error(WTRI_ENOMEM, "more than " + std::to_string(cap) + " cliques on the drawn edges"));
    const uint32_t kept = std::min(hs[3], (uint32_t)k);
    e = cudaMemcpyAsync(h_ids, oids, 4 * (size_t)kept * q, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h_w, ow, 8 * (size_t)kept, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && h_keys) e = cudaMemcpyAsync(h_keys, okey, 8 * (size_t)kept, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return done(cuda_error(e, "clique results", __FILE__, __LINE__));
    *h_count = (int32_t)kept;
    return done(WTRI_OK);
}

}  // namespace wtri
