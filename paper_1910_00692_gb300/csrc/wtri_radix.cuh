// Stable LSD radix sort passes (reduce-then-scan) over 16-byte records.
//
// A record is (key, v0, v1, v2), four 32-bit words.  One pass orders N
// records by the digit (key >> shift) & mask, stably, with digits of up to
// MAX_BITS bits.  The first pass of a sort reads its records through a
// Loader (a view of the source arrays, possibly a virtual stream such as
// "two adjacency entries per edge"); the last writes them through a Storer
// (the final arrays).  Passes in between read and write whole 16-byte
// records (one vector access each) and, beside every record, the next
// pass's digit as a 16-bit word, so the next histogram reads 2 bytes per
// record instead of the record.
//
//   Loader: static NARR, TILE_WORDS     source arrays copied per tile, words each
//           static REC_BYTES            bytes read per record
//           const void* tile_src(int a, int64_t tbase)
//           uint32_t skey(const uint32_t* in, int li)               from a copied tile
//           uint4 srec(const uint32_t* in, int li, int64_t tbase)
//           uint4 grec(int64_t i)       from global memory
//           uint32_t key(int64_t i)     (first-pass histogram)
//           void keys8(int64_t i, uint32_t (&k)[8])   keys i .. i + 7 (i a multiple of 8, sources aligned)
//           bool tma_ok()               sources 16-byte aligned
//   Storer: void store(int64_t p, const uint4& rec); double rec_bytes();
//           void prepare()          once per CTA before the first store
//
// Gating: every kernel of a pass first reads the device status word and
// returns at once if an earlier step reported an error, so a build needs no
// host round trip between its steps.  A pass may also be conditional on the
// largest key: with g.glo > 0 it runs only if some key has a bit at or above
// g.glo (bit length of *g.gwmax), which lets a sort over keys whose width is
// only known on the device launch the widest plan and skip the passes it
// does not need.
//
// Per pass: digit histograms of the rows of a count table (upsweep), a scan
// of the table's columns, and the scatter.  A CTA of the scatter streams its
// share of the records tile by tile (or, see spread_pass, takes every
// gridDim-th tile); the next tile's sources arrive by bulk asynchronous
// copies (cp.async.bulk, one mbarrier per buffer) while the current one is
// ranked (ballots over the digit's bits give a strip's equal digits, per-warp
// counters the ones before; stable).  The ranks give each place of the
// digit order its record's place in the tile (2 bytes); the records
// themselves stay where the copy put them, are read once, in digit order,
// and go straight out, consecutive threads storing consecutive positions of
// one digit's run.
//
// What bounds the scatter: the runs (TT / bins records) begin and end inside
// lines, and the time follows the write requests that reach L2, about 59 per
// ns (9-bit digits: 37 million for 62 million records, 2/5 of them for the
// digits), while DRAM is 45 % busy.  So one CTA per SM with the largest tile
// that shared memory holds twice.  Overlapping a CTA's phases gains nothing:
// two CTAs of 5,120 records without a second buffer take 77.0 ms where this
// takes 69.9 (the 1e9-edge build's scatters), of 2,688 with one 86.9.  One
// bulk copy per run from a tile staged in digit order: 66.3 without the
// digits, plain stores 60.7 (and histograms that read the records instead
// take back 10 ms).  Keeping the records in place instead of staging them
// (and with the ballots, which left the registers they need) allowed 5,632
// records a tile instead of 5,376: 71.3 -> 68.9 ms.
//
// One table for all: rows x bins, a row's counts written once by the block
// that counts it (no clearing, no global atomics) and scanned by 128 threads
// per column.  With counts per (digit, share) that eight blocks added into and
// one block per digit scanned, a 20,000-edge build took 515 us, now 465; 1e6
// edges 780, now 705; a 2e7-edge build 2.79 ms, now 2.51 (most of it the last
// pass's spread tiles).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>

#include "wtri_internal.cuh"

namespace wtri {
namespace radix {

constexpr int MAX_BITS = 10;               // widest digit of a pass
constexpr int MAX_BINS = 1 << MAX_BITS;
#ifndef WTRI_RADIX_NT
#define WTRI_RADIX_NT 512
#endif
#ifndef WTRI_RADIX_IT
#define WTRI_RADIX_IT 11
#endif
#ifndef WTRI_RADIX_CTAS
#define WTRI_RADIX_CTAS 1
#endif
constexpr int NT = WTRI_RADIX_NT;          // threads of the histogram and scatter CTAs
constexpr int NW = NT / 32;
constexpr int IT = WTRI_RADIX_IT;          // records per thread per tile
constexpr int TT = NT * IT;                // records per tile
constexpr int CTAS_PER_SM = WTRI_RADIX_CTAS;
constexpr int NBUF = 2;                    // tile buffers of a scatter CTA
constexpr int DPT = MAX_BINS / NT;         // digits owned by a thread in the tile scan
constexpr int MIN_SHARE = 1024;            // records
constexpr int MIN_ROW = 2048;              // records, where a share has several rows
constexpr int UP_SPLIT = 12;               // most table rows of a CTA's share (two full waves of the histogram's blocks)
constexpr int64_t OPEN_BYTES = int64_t(64) << 20;  // lines that L2 keeps open for the runs (half of it)
constexpr int SPREAD_TILES = 16;           // fewest tiles per CTA of a spread pass
constexpr int SCAN_ROWS = 2048;            // most rows that one launch scans
constexpr int SCAN_X = 8, SCAN_Y = 128;    // columns and row shares of a scan block
constexpr int UNT = 256;                   // threads of a histogram block
constexpr int UNW = UNT / 32;
constexpr uint32_t WAIT_LIMIT = 1u << 24;  // bounded mbarrier polling
static_assert(TT % 16 == 0, "tiles are whole 16-byte lines of every source array");
static_assert(DPT == 2, "a thread's digits are one 4-byte word of each warp's counters");

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Exclusive scan of one value per thread over an NTH-thread block (NTH <= 1024).
template <int NTH>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t* warp_tot,
                                                         uint32_t* total) {
    constexpr int NWW = NTH / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    if (w == 0) {
        uint32_t t = lane < NWW ? warp_tot[lane] : 0;
        uint32_t ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += y;
        }
        if (lane < NWW) warp_tot[lane] = ti - t;
        if (lane == NWW - 1) *total = ti;
    }
    __syncthreads();
    uint32_t r = warp_tot[w] + inc - x;
    __syncthreads();
    return r;
}

struct PassGeom {
    int64_t n;        // records
    int64_t share;    // records that a CTA takes at a time
    int64_t row;      // records per row of the count table
    int split;        // rows per share (the last may be shorter, or empty)
    int64_t rows;
    int shift;
    int bins;         // 1 << digit bits
    int bits;
    uint32_t mask;
    const uint32_t* gerr;   // status word: nonzero -> skip (may be null)
    const int32_t* gwmax;   // largest key value (conditional passes; may be null)
    int glo;                // conditional pass: runs iff bit_length(*gwmax) > glo
};

__device__ __forceinline__ bool pass_closed(const PassGeom& g) {
    if (g.gerr && *(volatile const uint32_t*)g.gerr) return true;
    if (g.glo > 0 && g.gwmax) {
        const int32_t wm = *(volatile const int32_t*)g.gwmax;
        const int B = wm > 0 ? 32 - __clz(wm) : 0;
        if (g.glo >= B) return true;
    }
    return false;
}

// ---- histogram sources ------------------------------------------------------
template <class Loader>
struct KeyDigits {  // first pass: the loader's keys
    static constexpr bool PACKED = false;
    Loader ld;
    int shift;
    uint32_t mask;
    bool vec;  // the sources are 16-byte aligned
    __device__ __forceinline__ uint32_t digit(int64_t i) const { return (ld.key(i) >> shift) & mask; }
    __device__ __forceinline__ void digits8(int64_t i, uint32_t (&d)[8]) const {
        ld.keys8(i, d);
#pragma unroll
        for (int k = 0; k < 8; k++) d[k] = (d[k] >> shift) & mask;
    }
};
struct StoredDigits {  // later passes: 16-bit digits written by the previous scatter
    static constexpr bool PACKED = true;
    static constexpr bool vec = true;
    const uint16_t* d;
    __device__ __forceinline__ uint32_t digit(int64_t i) const { return __ldg(d + i); }
    __device__ __forceinline__ void digits8(int64_t i, uint32_t (&x)[8]) const {
        const uint4 r = __ldg(reinterpret_cast<const uint4*>(d + i));
        x[0] = r.x & 0xffffu, x[1] = r.x >> 16, x[2] = r.y & 0xffffu, x[3] = r.y >> 16;
        x[4] = r.z & 0xffffu, x[5] = r.z >> 16, x[6] = r.w & 0xffffu, x[7] = r.w >> 16;
    }
};

// Digit histograms of equal shares: row r of the table counts part r % split
// of share r / split.  Each warp of a block counts into its own shared copy.
// Eight digits per thread and step: one 16-byte load of stored digits, two of
// sources.  1e9 and 2e9 keys take 710 and 1,580 us, 2e9 stored digits 830-900
// (with counts added into one row per share: 640, 1,430 and 850-930); with
// one key per load 730 and 1,650.
template <class Dig>
__global__ void __launch_bounds__(UNT) k_upsweep(Dig dg, PassGeom g, uint32_t* table) {
    if (pass_closed(g)) return;
    __shared__ uint32_t hist[UNW][MAX_BINS];
    const int w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < UNW * MAX_BINS; i += UNT) (&hist[0][0])[i] = 0;
    __syncthreads();
    uint32_t* h = hist[w];
    const int share = blockIdx.x / g.split, part = blockIdx.x % g.split;
    const int64_t sbeg = (int64_t)share * g.share;
    const int64_t send = min(g.n, sbeg + g.share);
    const int64_t beg = min(send, sbeg + part * g.row);
    const int64_t end = min(send, beg + g.row);
    int64_t i0 = beg;
    if (dg.vec) {
        const int64_t nv = (end - beg) >> 3;  // whole groups of 8 (beg is a multiple of 8)
#pragma unroll 2
        for (int64_t q = threadIdx.x; q < nv; q += UNT) {
            uint32_t d[8];
            dg.digits8(beg + (q << 3), d);
#pragma unroll
            for (int k = 0; k < 8; k++) atomicAdd(&h[d[k]], 1u);
        }
        i0 = beg + (nv << 3);
    } else {
        constexpr int U = 4;
        for (; i0 + (int64_t)U * UNT <= end; i0 += (int64_t)U * UNT) {
            uint32_t d[U];
#pragma unroll
            for (int u = 0; u < U; u++) d[u] = dg.digit(i0 + (int64_t)u * UNT + threadIdx.x);
#pragma unroll
            for (int u = 0; u < U; u++) atomicAdd(&h[d[u]], 1u);
        }
    }
    for (int64_t i = i0 + threadIdx.x; i < end; i += UNT) atomicAdd(&h[dg.digit(i)], 1u);
    __syncthreads();
    for (int d = threadIdx.x; d < g.bins; d += UNT) {
        uint32_t s = 0;
#pragma unroll
        for (int k = 0; k < UNW; k++) s += hist[k][d];
        table[(int64_t)blockIdx.x * g.bins + d] = s;
    }
}

// The same where a share is one tile (a row each): a block takes every
// gridDim-th tile.
__global__ void __launch_bounds__(UNT) k_upsweep_tiles(const uint16_t* __restrict__ dig, PassGeom g, uint32_t* table) {
    if (pass_closed(g)) return;
    __shared__ uint32_t hist[UNW][MAX_BINS];
    for (int i = threadIdx.x; i < UNW * MAX_BINS; i += UNT) (&hist[0][0])[i] = 0;
    __syncthreads();
    uint32_t* h = hist[threadIdx.x >> 5];
    const StoredDigits dg{dig};
    for (int64_t r = blockIdx.x; r < g.rows; r += gridDim.x) {
        const int64_t beg = r * g.share, end = min(g.n, beg + g.share), nv = (end - beg) >> 3;
        for (int64_t q = threadIdx.x; q < nv; q += UNT) {
            uint32_t d[8];
            dg.digits8(beg + (q << 3), d);
#pragma unroll
            for (int k = 0; k < 8; k++) atomicAdd(&h[d[k]], 1u);
        }
        for (int64_t i = beg + (nv << 3) + threadIdx.x; i < end; i += UNT) atomicAdd(&h[__ldg(dig + i)], 1u);
        __syncthreads();
        for (int d = threadIdx.x; d < g.bins; d += UNT) {
            uint32_t s = 0;
#pragma unroll
            for (int k = 0; k < UNW; k++) {
                s += hist[k][d];
                hist[k][d] = 0;
            }
            table[r * g.bins + d] = s;
        }
        __syncthreads();
    }
}

// Exclusive scan of the table's columns (rows x bins), in place; totals[d] =
// column d's sum.  Up to SCAN_ROWS rows: k_col_scan alone.  More: in segments
// of rows, whose sums k_seg_sum writes, k_col_scan scans and k_seg_apply
// spreads over their rows.
__global__ void __launch_bounds__(SCAN_X * SCAN_Y) k_col_scan(uint32_t* table, int64_t rows, uint32_t* totals,
                                                              PassGeom g) {
    if (pass_closed(g)) return;
    __shared__ uint32_t part[SCAN_X][SCAN_Y + 1];
    const int x = threadIdx.x % SCAN_X, y = threadIdx.x / SCAN_X, d = blockIdx.x * SCAN_X + x;
    const int64_t per = (rows + SCAN_Y - 1) / SCAN_Y, beg = min(rows, y * per), end = min(rows, beg + per);
    uint32_t s = 0;
    if (d < g.bins) {
#pragma unroll 8
        for (int64_t r = beg; r < end; r++) s += table[r * g.bins + d];
    }
    part[x][y] = s;
    __syncthreads();
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    if (c < SCAN_X) {  // a warp per column
        constexpr int PER = SCAN_Y / 32;
        uint32_t v[PER], sum = 0;
#pragma unroll
        for (int i = 0; i < PER; i++) {
            v[i] = part[c][lane * PER + i];
            sum += v[i];
        }
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t z = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += z;
        }
        uint32_t run = inc - sum;
#pragma unroll
        for (int i = 0; i < PER; i++) {
            part[c][lane * PER + i] = run;
            run += v[i];
        }
        if (lane == 31 && blockIdx.x * SCAN_X + c < g.bins) totals[blockIdx.x * SCAN_X + c] = run;
    }
    __syncthreads();
    if (d >= g.bins) return;
    uint32_t run = part[x][y];
    constexpr int U = 8;
    for (int64_t r0 = beg; r0 < end; r0 += U) {
        uint32_t v[U];
#pragma unroll
        for (int u = 0; u < U; u++) v[u] = r0 + u < end ? table[(r0 + u) * g.bins + d] : 0u;
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (r0 + u < end) table[(r0 + u) * g.bins + d] = run;
            run += v[u];
        }
    }
}

__global__ void __launch_bounds__(UNT) k_seg_sum(const uint32_t* __restrict__ table, int seg,
                                                 uint32_t* __restrict__ sums, PassGeom g) {
    if (pass_closed(g)) return;
    const int d = blockIdx.y * UNT + threadIdx.x;
    if (d >= g.bins) return;
    const int64_t beg = (int64_t)blockIdx.x * seg, end = min(g.rows, beg + seg);
    uint32_t s = 0;
#pragma unroll 8
    for (int64_t r = beg; r < end; r++) s += __ldg(table + r * g.bins + d);
    sums[(int64_t)blockIdx.x * g.bins + d] = s;
}

__global__ void __launch_bounds__(UNT) k_seg_apply(uint32_t* table, int seg, const uint32_t* __restrict__ sums,
                                                   PassGeom g) {
    if (pass_closed(g)) return;
    const int d = blockIdx.y * UNT + threadIdx.x;
    if (d >= g.bins) return;
    const int64_t beg = (int64_t)blockIdx.x * seg, end = min(g.rows, beg + seg);
    uint32_t run = sums[(int64_t)blockIdx.x * g.bins + d];
    constexpr int U = 8;
    for (int64_t r0 = beg; r0 < end; r0 += U) {
        uint32_t v[U];
#pragma unroll
        for (int u = 0; u < U; u++) v[u] = r0 + u < end ? table[(r0 + u) * g.bins + d] : 0u;
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (r0 + u < end) table[(r0 + u) * g.bins + d] = run;
            run += v[u];
        }
    }
}

// ---- scatter -----------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void bar_init(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void bar_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}
#ifndef WTRI_RADIX_LOAD_HINT
#define WTRI_RADIX_LOAD_HINT 1
#endif
// Tile sources are read once: an evict-first L2 policy keeps them from
// displacing the partially written lines of the digit runs.
__device__ __forceinline__ uint64_t evict_first_policy() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                          uint64_t policy) {
#if WTRI_RADIX_LOAD_HINT
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
        : "memory");
#else
    (void)policy;
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
#endif
}
__device__ __forceinline__ bool bar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

struct ScatterSmem {
    uint4 buf[NBUF][TT];           // tiles' sources
    uint16_t src[TT];              // tile place of the record at each place of the digit order
    uint16_t cnt[NW][MAX_BINS];    // per (warp, digit): count, then offset in the digit order
    uint32_t delta[MAX_BINS];      // output position of digit-order place p = delta[digit] + p
    uint32_t warp_tot[32];
    uint32_t total;
    int timed_out;
    uint64_t bar[NBUF];
};
static_assert(TT <= 65536, "a tile place fits 16 bits");

__device__ __forceinline__ uint32_t lo16(uint32_t x) { return x & 0xffffu; }
__device__ __forceinline__ uint32_t hi16(uint32_t x) { return x >> 16; }

// Lanes of the warp holding the same digit (of BITS bits) as this lane; lanes
// without a record group among themselves.
template <int BITS>
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, bool valid) {
    const uint32_t vb = __ballot_sync(0xffffffffu, valid);
    uint32_t p = valid ? vb : ~vb;
#pragma unroll
    for (int k = 0; k < BITS; k++) {
        const uint32_t b = __ballot_sync(0xffffffffu, (d >> k) & 1u);
        p &= b ^ (((d >> k) & 1u) - 1u);  // the ballot, or its complement
    }
    return p;
}

// A thread's DPT consecutive 16-bit counters as one word.
__device__ __forceinline__ void load_counts(const uint16_t* p, uint32_t (&c)[DPT]) {
    const uint32_t r = *reinterpret_cast<const uint32_t*>(p);
    c[0] = lo16(r);
    c[1] = hi16(r);
}
__device__ __forceinline__ void store_counts(uint16_t* p, const uint32_t (&s)[DPT]) {
    *reinterpret_cast<uint32_t*>(p) = s[0] | (s[1] << 16);
}

// Ranks a tile's digits within each warp: rk[j] = digit | rank << 16, and the
// per-(warp, digit) counts.  Item j of warp w, lane l is record
// (w * strips + j) * 32 + l of the tile, strips = IT in a full tile; strips in
// order and warps in order keep equal digits stable.
template <int BITS, bool FULL>
__device__ __forceinline__ void rank_strips(uint32_t (&rk)[IT], int strips, int tcount, ScatterSmem& S) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t lt = lanemask_lt();
    uint16_t* cnt = S.cnt[w];
    auto valid = [&](int j) { return FULL || (j < strips && (w * strips + j) * 32 + lane < tcount); };
    uint32_t peers[IT];
#pragma unroll
    for (int j = 0; j < IT; j++) {  // independent across strips
        if (!FULL && j >= strips) break;
        peers[j] = digit_peers<BITS>(rk[j], valid(j));
    }
#pragma unroll
    for (int j = 0; j < IT; j++) {
        if (!FULL && j >= strips) break;
        const uint32_t d = rk[j];
        const uint32_t b = valid(j) ? (uint32_t)cnt[d] : 0u;
        rk[j] = d | ((b + __popc(peers[j] & lt)) << 16);
        __syncwarp();
        if (valid(j) && (peers[j] & lt) == 0) cnt[d] = (uint16_t)(b + __popc(peers[j]));
        __syncwarp();
    }
}

// Ranks and writes one tile of tcount <= TT records.  key(li), rec(li): the
// tile's records, in shared memory.  On entry the counters are zero and the
// tile visible to every thread.  run[] holds this thread's digits' next
// output positions (digits threadIdx.x * DPT + i); FRESH: they are base[] +
// first[] (loads that may still be in flight on entry).
template <bool FULL, bool FRESH, class Key, class Rec, class Storer>
__device__ __forceinline__ void scatter_tile(const Key& key, const Rec& rec, int tcount, const Storer& st,
                                             const PassGeom& g, uint32_t (&run)[DPT], const uint32_t (&base)[DPT],
                                             const uint32_t (&first)[DPT], ScatterSmem& S) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int strips = FULL ? IT : (tcount + NT - 1) / NT;
    // 1. rank within the warp
    uint32_t rk[IT];
#pragma unroll
    for (int j = 0; j < IT; j++) {
        const int li = (w * strips + j) * 32 + lane;
        rk[j] = FULL || (j < strips && li < tcount) ? (key(li) >> g.shift) & g.mask : 0u;
    }
    if (g.bits > 9) rank_strips<10, FULL>(rk, strips, tcount, S);
    else if (g.bits == 9) rank_strips<9, FULL>(rk, strips, tcount, S);
    else rank_strips<8, FULL>(rk, strips, tcount, S);
    __syncthreads();
    // 2. per digit: offsets of each warp, tile start, output delta.  Thread t
    //    owns digits DPT t .. DPT t + DPT - 1: one word of each warp's counters.
    {
        const int d0 = threadIdx.x * DPT;
        const bool mine = d0 < g.bins;
        uint32_t tot[DPT];
#pragma unroll
        for (int i = 0; i < DPT; i++) tot[i] = 0;
        if (mine) {
#pragma unroll
            for (int k = 0; k < NW; k++) {
                uint32_t c[DPT];
                load_counts(&S.cnt[k][d0], c);
#pragma unroll
                for (int i = 0; i < DPT; i++) tot[i] += c[i];
            }
        }
        uint32_t sum = 0;
#pragma unroll
        for (int i = 0; i < DPT; i++) sum += tot[i];
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) S.warp_tot[w] = inc;
        __syncthreads();
        if (mine) {
            uint32_t start = inc - sum;
#pragma unroll
            for (int k = 0; k < NW; k++) start += k < w ? S.warp_tot[k] : 0u;
            uint32_t s[DPT];
            s[0] = start;
#pragma unroll
            for (int i = 1; i < DPT; i++) s[i] = s[i - 1] + tot[i - 1];
#pragma unroll
            for (int i = 0; i < DPT; i++) {
                if (FRESH) run[i] = base[i] + first[i];
                S.delta[d0 + i] = run[i] - s[i];
                run[i] += tot[i];
            }
#pragma unroll
            for (int k = 0; k < NW; k++) {
                uint32_t c[DPT];
                load_counts(&S.cnt[k][d0], c);
                store_counts(&S.cnt[k][d0], s);
#pragma unroll
                for (int i = 0; i < DPT; i++) s[i] += c[i];
            }
        }
    }
    __syncthreads();
    // 3. the digit order
#pragma unroll
    for (int j = 0; j < IT; j++) {
        const int li = (w * strips + j) * 32 + lane;
        if (FULL || (j < strips && li < tcount)) S.src[S.cnt[w][lo16(rk[j])] + hi16(rk[j])] = (uint16_t)li;
    }
    __syncthreads();
    // 4. write: consecutive threads, consecutive positions of one digit's run
#pragma unroll
    for (int i = 0; i < IT; i++) {
        const int p = i * NT + threadIdx.x;
        if (FULL || p < tcount) {
            const uint4 r = rec((int)S.src[p]);
            const uint32_t d = (r.x >> g.shift) & g.mask;
            st.store((int64_t)S.delta[d] + p, r);
        }
    }
}

// The counters of the used digits, zeroed (16-byte words, 8 digits each; at
// least one word).
__device__ __forceinline__ void zero_counts(const PassGeom& g, ScatterSmem& S) {
    const int zw = (g.bins + 7) >> 3;
    for (int q = threadIdx.x; q < zw * NW; q += NT)
        reinterpret_cast<uint4*>(&S.cnt[q / zw][0])[q % zw] = make_uint4(0, 0, 0, 0);
}

// CTA b takes share b, or, SPREAD (a share is one tile), the tiles b, b +
// gridDim.x, ...  Whole tiles arrive by bulk copies when
// USE_BULK (sources 16-byte aligned), the last partial tile of the last share
// (and every tile otherwise) by plain loads.  Waits are bounded: on timeout
// the pass sets DEV_ERR_TIMEOUT, gives copies in flight a bounded chance to
// land and the CTA returns.
template <class Loader, class Storer, bool USE_BULK, bool SPREAD>
__global__ void __launch_bounds__(NT, CTAS_PER_SM) k_scatter(Loader ld, Storer st_in, PassGeom g,
                                                           const uint32_t* __restrict__ table,
                                                           const uint32_t* __restrict__ totals, uint32_t* err) {
    if (pass_closed(g)) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    ScatterSmem& S = *reinterpret_cast<ScatterSmem*>(smem_raw);
    Storer st = st_in;
    st.prepare();
    const int d0 = threadIdx.x * DPT;
    uint32_t base[DPT], run[DPT], first[DPT];
    {   // where each digit's records start
        uint32_t t[DPT], sum = 0;
#pragma unroll
        for (int i = 0; i < DPT; i++) {
            t[i] = d0 + i < g.bins ? totals[d0 + i] : 0u;
            sum += t[i];
            run[i] = first[i] = 0;
        }
        base[0] = block_exclusive_scan<NT>(sum, S.warp_tot, &S.total);
#pragma unroll
        for (int i = 1; i < DPT; i++) base[i] = base[i - 1] + t[i - 1];
    }
    int64_t pos = (int64_t)blockIdx.x * g.share;
    int64_t end = min(g.n, pos + g.share);
    constexpr uint32_t ARR_BYTES = Loader::TILE_WORDS * 4u;
    static_assert(Loader::NARR * Loader::TILE_WORDS <= 4 * TT, "a tile's sources fit one buffer");
    if (threadIdx.x == 0) {
        for (int b = 0; b < NBUF; b++) bar_init(&S.bar[b]);
        S.timed_out = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const uint64_t policy = evict_first_policy();
    auto issue = [&](int64_t tbase, int b) {
        bar_expect(&S.bar[b], ARR_BYTES * Loader::NARR);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&S.buf[b][0]);
#pragma unroll
        for (int a = 0; a < Loader::NARR; a++)
            bulk_load(dst + (size_t)a * TT, ld.tile_src(a, tbase), ARR_BYTES, &S.bar[b], policy);
    };
    auto load_first = [&](int64_t row) {
#pragma unroll
        for (int i = 0; i < DPT; i++)
            if (d0 + i < g.bins) first[i] = __ldg(table + row * g.bins + d0 + i);
    };
    const int64_t step = (int64_t)gridDim.x * g.share;  // SPREAD: from a tile to the CTA's next
    load_first((int64_t)blockIdx.x * g.split);
    if (!SPREAD) {
#pragma unroll
        for (int i = 0; i < DPT; i++) run[i] = base[i] + first[i];
    }
    if (USE_BULK && threadIdx.x == 0 && pos + TT <= end) issue(pos, 0);
    for (int64_t k = 0; USE_BULK && pos + TT <= end; k++) {
        const int b = (int)(k % NBUF);
        const uint32_t parity = (uint32_t)((k / NBUF) & 1);
        zero_counts(g, S);  // last read before the previous tile's write
        uint32_t spins = 0;
        while (!bar_try_wait(&S.bar[b], parity)) {
            if (++spins >= WAIT_LIMIT) {
                S.timed_out = 1;
                break;
            }
        }
        __syncthreads();
        if (S.timed_out) {
            if (threadIdx.x == 0) atomicOr(err, DEV_ERR_TIMEOUT);
            for (int bb = 0; bb < NBUF; bb++) {
                uint32_t s2 = 0;
                while (!bar_try_wait(&S.bar[bb], parity) && ++s2 < WAIT_LIMIT) {
                }
            }
            return;
        }
        const int64_t next = SPREAD ? pos + step : pos + TT, nend = SPREAD ? min(g.n, next + TT) : end;
        // the buffer of the tile before was read up to the barrier above
        if (threadIdx.x == 0 && next + TT <= nend) issue(next, (b + 1) % NBUF);
        const uint32_t* in = reinterpret_cast<const uint32_t*>(&S.buf[b][0]);
        scatter_tile<true, SPREAD>([&](int li) { return ld.skey(in, li); },
                                   [&](int li) { return ld.srec(in, li, pos); }, TT, st, g, run, base, first, S);
        if (SPREAD && next < g.n) load_first(next / TT);
        pos = next;
        end = nend;
    }
    while (pos < end) {
        const int tcount = (int)min((int64_t)TT, end - pos);
        __syncthreads();  // the tile before is written
        zero_counts(g, S);
        uint4* in = S.buf[0];
        for (int li = threadIdx.x; li < tcount; li += NT) in[li] = ld.grec(pos + li);
        __syncthreads();
        scatter_tile<false, SPREAD>([&](int li) { return in[li].x; }, [&](int li) { return in[li]; }, tcount, st, g, run,
                                    base, first, S);
        if (SPREAD) {
            pos += step;
            end = min(g.n, pos + TT);
            if (pos < g.n) load_first(pos / TT);
        } else {
            pos += TT;
        }
    }
}

// ---- intermediate records -----------------------------------------------------
struct AosLoader {
    static constexpr double REC_BYTES = 16.0;
    static constexpr int NARR = 1;
    static constexpr uint32_t TILE_WORDS = 4 * TT;
    const uint4* r;
    __device__ __forceinline__ uint32_t key(int64_t i) const { return __ldg(&r[i].x); }
    __device__ __forceinline__ const void* tile_src(int, int64_t tbase) const { return r + tbase; }
    __device__ __forceinline__ uint32_t skey(const uint32_t* in, int li) const { return in[4 * li]; }
    __device__ __forceinline__ uint4 srec(const uint32_t* in, int li, int64_t) const {
        return reinterpret_cast<const uint4*>(in)[li];
    }
    __device__ __forceinline__ uint4 grec(int64_t i) const { return __ldg(r + i); }
    bool tma_ok() const { return ((uintptr_t)r & 15) == 0; }
};

struct AosStorer {
    uint4* r;
    uint16_t* dig;  // next pass's digit of each record
    int next_shift;
    uint32_t next_mask;
    __host__ __device__ double rec_bytes() const { return 18.0; }
    __device__ __forceinline__ void prepare() {}
    __device__ __forceinline__ void store(int64_t p, const uint4& x) const {
        r[p] = x;
        dig[p] = (uint16_t)((x.x >> next_shift) & next_mask);
    }
};

// A pass whose output is either the final arrays or the next pass's records:
// final iff the following pass is skipped (see PassGeom::glo), decided once
// per CTA from the device-side key width.
template <class Final>
struct SwitchStorer {
    Final fin;
    AosStorer mid;
    const int32_t* gwmax;
    int next_lo;   // lowest key bit of the following pass
    bool is_final;
    __host__ __device__ double rec_bytes() const { return mid.rec_bytes(); }
    __device__ __forceinline__ void prepare() {
        const int32_t wm = *(volatile const int32_t*)gwmax;
        const int B = wm > 0 ? 32 - __clz(wm) : 0;
        is_final = next_lo >= B;
    }
    __device__ __forceinline__ void store(int64_t p, const uint4& x) const {
        if (is_final) fin.store(p, x);
        else mid.store(p, x);
    }
};

// ---- host side ------------------------------------------------------------------
inline int64_t scatter_ctas() { return (int64_t)sm_count() * CTAS_PER_SM; }

// Shares: one per CTA, equal (a multiple of 32 records, so that every source
// stays 16-byte aligned; not of more, or the CTAs would all stand at the same
// offset of the memory channels: 4 % slower scatters at 1e8 edges with shares
// of 1,285 x 1,024 records), counted in up to UP_SPLIT rows; or, spread, one
// tile each, dealt round-robin.
inline PassGeom make_geom(int64_t n, int shift, int bits, bool spread = false) {
    PassGeom g;
    g.n = n;
    const int64_t ctas = scatter_ctas(), per = (std::max<int64_t>(MIN_SHARE, (n + ctas - 1) / ctas) + 31) / 32 * 32;
    g.share = spread ? TT : per;
    g.split = spread ? 1 : (int)std::min<int64_t>(UP_SPLIT, std::max<int64_t>(1, per / MIN_ROW));
    g.row = ((g.share + g.split - 1) / g.split + 31) / 32 * 32;
    g.rows = std::max<int64_t>(1, (n + g.share - 1) / g.share * g.split);
    g.shift = shift;
    g.bins = 1 << bits;
    g.bits = bits;
    g.mask = (uint32_t)g.bins - 1u;
    g.gerr = nullptr;
    g.gwmax = nullptr;
    g.glo = 0;
    return g;
}

// Whether a pass into `streams` arrays deals its tiles round-robin.  With a
// share each, every CTA keeps a line open for every digit and array; beyond
// what L2 holds of them, lines are evicted half written (10-bit digits into
// the four arrays of the rows: 80 MB; the pass takes 744 us at 2e7 edges, 539
// spread).  Below, the spread tiles cost their counts and scans and gain
// nothing: 10-bit digits into records and digits, 40 MB, 475 -> 404 us but 66
// us more of counting; 9-bit ones at 1e9 edges 17.4 -> 19 ms.
inline bool spread_pass(int64_t n, int bits, int streams) {
    const int64_t ctas = scatter_ctas();
    return n >= SPREAD_TILES * ctas * TT && (ctas * streams * 128 << bits) > OPEN_BYTES;
}

inline int64_t max_segs() { return (int64_t)sm_count() * 8; }

// Scratch for the counts of any sort of at most n records, with or without a
// spread pass: the table, its totals, the segments' sums (uint32).
inline size_t scratch_words(int64_t n, bool spread) {
    int64_t rows = std::min<int64_t>(scatter_ctas() * UP_SPLIT, n / MIN_SHARE + UP_SPLIT);
    if (spread) rows = std::max(rows, n / TT + 1);
    return (size_t)MAX_BINS * (size_t)(rows + 1 + (rows > SCAN_ROWS ? max_segs() : 0));
}

// Whether whole tiles use bulk copies (WTRI_RADIX_TMA=0 turns them off).
inline bool bulk_enabled() {
    static int v = -1;
    if (v < 0) {
        const char* e = getenv("WTRI_RADIX_TMA");
        v = (e && e[0] == '0') ? 0 : 1;
    }
    return v == 1;
}

// Digit widths of a sort over 'bits' key bits: as few passes as MAX_BITS
// allows, bits spread evenly (e.g. 26 -> 9, 9, 8; 20 -> 10, 10).
inline int pass_count(int bits) { return (bits + MAX_BITS - 1) / MAX_BITS; }
inline int pass_bits(int bits, int p) {
    const int passes = pass_count(bits);
    return bits / passes + (p < bits % passes ? 1 : 0);
}
inline int pass_shift(int bits, int p) {
    int s = 0;
    for (int q = 0; q < p; q++) s += pass_bits(bits, q);
    return s;
}

// alg_bytes: this pass's share of the sort's algorithmic bytes (the
// scatter's phase timer; histograms and scans declare none).  expected:
// whether the pass is expected to run (a conditional pass that the widest
// expected keys skip declares no moved bytes either).
template <bool SPREAD = false, class Dig, class Loader, class Storer>
int run_pass(const Dig& dg, const Loader& ld, const Storer& st, const PassGeom& g, uint32_t* scratch,
             cudaStream_t s, uint32_t* err, double hist_bytes, double alg_bytes, bool expected = true) {
    const double mv = expected ? 1.0 : 0.0;
    if (g.n <= 0) return WTRI_OK;
    uint32_t* table = scratch;
    uint32_t* totals = table + (size_t)MAX_BINS * g.rows;
    {
        ProfScope ps("radix_upsweep", s, 0.0, 1, mv * (hist_bytes * (double)g.n + 4.0 * g.bins * (double)g.rows));
        if constexpr (SPREAD) {
            static_assert(Dig::PACKED, "spread passes read stored digits");
            k_upsweep_tiles<<<(unsigned)std::min<int64_t>(g.rows, sm_count() * 6), UNT, 0, s>>>(dg.d, g, table);
        } else {
            k_upsweep<Dig><<<(unsigned)g.rows, UNT, 0, s>>>(dg, g, table);
        }
    }
    {
        const bool segmented = g.rows > SCAN_ROWS;
        const unsigned cols = (unsigned)((g.bins + SCAN_X - 1) / SCAN_X);
        ProfScope ps("radix_digit_scan", s, 0.0, segmented ? 3 : 1,
                     mv * (segmented ? 12.0 : 8.0) * g.bins * (double)g.rows);
        if (!segmented) {
            k_col_scan<<<cols, SCAN_X * SCAN_Y, 0, s>>>(table, g.rows, totals, g);
        } else {
            uint32_t* sums = totals + MAX_BINS;
            const int seg = (int)((g.rows + max_segs() - 1) / max_segs());
            const unsigned segs = (unsigned)((g.rows + seg - 1) / seg);
            const dim3 grid(segs, (unsigned)((g.bins + UNT - 1) / UNT));
            k_seg_sum<<<grid, UNT, 0, s>>>(table, seg, sums, g);
            k_col_scan<<<cols, SCAN_X * SCAN_Y, 0, s>>>(sums, segs, totals, g);
            k_seg_apply<<<grid, UNT, 0, s>>>(table, seg, sums, g);
        }
    }
    const size_t smem = sizeof(ScatterSmem);
    const unsigned ctas = (unsigned)std::min<int64_t>(scatter_ctas(), (g.n + g.share - 1) / g.share);
    ProfScope ps("radix_downsweep", s, alg_bytes, 1, mv * (double)g.n * (Loader::REC_BYTES + st.rec_bytes()));
    if (bulk_enabled() && ld.tma_ok()) {
        static std::atomic<uint64_t> done{0};  // per instantiation and device
        WTRI_TRY(smem_optin((const void*)k_scatter<Loader, Storer, true, SPREAD>, (int)smem, done));
        k_scatter<Loader, Storer, true, SPREAD><<<ctas, NT, smem, s>>>(ld, st, g, table, totals, err);
    } else {
        static std::atomic<uint64_t> done{0};
        WTRI_TRY(smem_optin((const void*)k_scatter<Loader, Storer, false, SPREAD>, (int)smem, done));
        k_scatter<Loader, Storer, false, SPREAD><<<ctas, NT, smem, s>>>(ld, st, g, table, totals, err);
    }
    WTRI_CUDA(cudaGetLastError());
    return WTRI_OK;
}

// Whether lsd_sort spreads the last pass of n records over 'bits' key bits.
inline bool sort_spreads(int64_t n, int bits, int streams) {
    const int last = pass_count(bits) - 1;
    return last > 0 && spread_pass(n, pass_bits(bits, last), streams);
}

// Full stable LSD sort of n records over 'bits' key bits: first pass from
// 'first', middle passes through the 16-byte record buffers rec_a / rec_b
// (n records each) with digits in 'dig' (n 16-bit words), last pass into
// 'last'.  alg_total: the sort's algorithmic bytes (one read and one write
// of its payload), spread evenly over its passes' scatters.  Every kernel
// returns at once while *err is nonzero.
template <class First, class Last>
int lsd_sort(const First& first, const Last& last, int64_t n, int bits, uint4* rec_a, uint4* rec_b,
             uint16_t* dig, uint32_t* scratch, cudaStream_t s, uint32_t* err, double alg_total) {
    const int passes = pass_count(bits);
    if (passes == 0) return set_error(WTRI_EINVAL, "internal: zero-pass sort");
    const double alg = alg_total / passes;
    uint4* cur = rec_a;
    uint4* nxt = rec_b;
    for (int p = 0; p < passes; p++) {
        const bool spread = p == passes - 1 && sort_spreads(n, bits, Last::STREAMS);
        PassGeom g = make_geom(n, pass_shift(bits, p), pass_bits(bits, p), spread);
        g.gerr = err;
        AosStorer as{nxt, dig, 0, 0u};
        if (p + 1 < passes) {
            as.next_shift = pass_shift(bits, p + 1);
            as.next_mask = (1u << pass_bits(bits, p + 1)) - 1u;
        }
        AosLoader al{cur};
        StoredDigits sd{dig};
        if (p == 0) {
            KeyDigits<First> kd{first, g.shift, g.mask, first.tma_ok()};
            if (passes == 1) {
                WTRI_TRY(run_pass(kd, first, last, g, scratch, s, err, 4.0, alg));
            } else {
                WTRI_TRY(run_pass(kd, first, as, g, scratch, s, err, 4.0, alg));
            }
        } else if (p == passes - 1) {
            if (spread) WTRI_TRY(run_pass<true>(sd, al, last, g, scratch, s, err, 2.0, alg));
            else WTRI_TRY(run_pass(sd, al, last, g, scratch, s, err, 2.0, alg));
        } else {
            WTRI_TRY(run_pass(sd, al, as, g, scratch, s, err, 2.0, alg));
        }
        if (p + 1 < passes) std::swap(cur, nxt);
    }
    return WTRI_OK;
}

// The same sort for keys whose width is known only on the device: the key's
// largest value is *wmax (written by an earlier kernel on the stream).  The
// plan covers max_bits in digits of MAX_BITS (pass p: bits [10p, 10p+10));
// pass p > 0 runs only if a key has a bit at or above 10p, and each pass
// writes the final arrays when the next one will not run.  alg_total is
// spread over the passes the widest keys need (the phase timers see what
// runs).
template <class First, class Last>
int lsd_sort_device_width(const First& first, const Last& last, int64_t n, int max_bits,
                          const int32_t* wmax, uint4* rec_a, uint4* rec_b, uint16_t* dig,
                          uint32_t* scratch, cudaStream_t s, uint32_t* err, double alg_total,
                          int expected_passes) {
    const int passes = (max_bits + MAX_BITS - 1) / MAX_BITS;
    const double alg = alg_total / std::max(1, expected_passes);
    uint4* cur = rec_a;
    uint4* nxt = rec_b;
    for (int p = 0; p < passes; p++) {
        const int shift = p * MAX_BITS;
        const int bits = std::min(MAX_BITS, max_bits - shift);
        PassGeom g = make_geom(n, shift, bits);
        g.gerr = err;
        g.gwmax = wmax;
        g.glo = shift;  // pass 0 always runs (glo = 0)
        AosStorer as{nxt, dig, 0, 0u};
        if (p + 1 < passes) {
            as.next_shift = shift + MAX_BITS;
            as.next_mask = (1u << std::min(MAX_BITS, max_bits - shift - MAX_BITS)) - 1u;
        }
        SwitchStorer<Last> sw{last, as, wmax, shift + MAX_BITS, false};
        AosLoader al{cur};
        StoredDigits sd{dig};
        const bool ex = p < expected_passes;
        const double a = ex ? alg : 0.0;
        if (p == 0) {
            KeyDigits<First> kd{first, g.shift, g.mask, first.tma_ok()};
            if (passes == 1) {
                WTRI_TRY(run_pass(kd, first, last, g, scratch, s, err, 4.0, a, ex));
            } else {
                WTRI_TRY(run_pass(kd, first, sw, g, scratch, s, err, 4.0, a, ex));
            }
        } else if (p == passes - 1) {
            WTRI_TRY(run_pass(sd, al, last, g, scratch, s, err, 2.0, a, ex));
        } else {
            WTRI_TRY(run_pass(sd, al, sw, g, scratch, s, err, 2.0, a, ex));
        }
        std::swap(cur, nxt);
    }
    return WTRI_OK;
}

inline int bit_length(uint64_t x) {
    int b = 0;
    while (x) {
        b++;
        x >>= 1;
    }
    return b;
}

}  // namespace radix
}  // namespace wtri
