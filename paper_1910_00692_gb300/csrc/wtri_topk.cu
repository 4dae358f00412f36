// Exact top-k query, weighted edge sampling and the allocation-free query:
// host orchestration of the kernels in wtri_query.cuh.
#include "wtri_query.cuh"

#include <mutex>

namespace wtri {
namespace {

// Poll limits of a grid barrier's first wait and of the later ones (test hooks
// lower them; see wtri_debug_set_wait_limits).
std::atomic<uint32_t> g_wait_first{WAIT_LIMIT}, g_wait_later{WAIT_LIMIT};

uint32_t poll_limit(int64_t polls) {
    return polls < 0 ? WAIT_LIMIT : (uint32_t)std::min<int64_t>(polls, UINT32_MAX);
}

// The fields of a query's sweep that come from its graph and call.
void set_sweep(Query& q, const wtri_graph* g, int32_t k) {
    q.k = k;
    q.total = g->d.m;
    q.first = g->tune.first_round;
    q.growth = g->tune.growth;
    q.t_short = g->tune.t_short;
    q.fw = g->d.fw;
    q.wait_first = first_wait_limit();
    q.wait_later = later_wait_limit();
}

template <int P>
int run_query(const wtri_graph* g, int32_t k, wtri_tri* d_tris, double* d_weight, int32_t* d_count,
              cudaStream_t s, int scale, int shard, int nshards, unsigned long long* d_keys,
              double gp) {
    const uint32_t cap = (uint32_t)std::min<int64_t>(
        (int64_t(1) << 20) * scale + 16 * (int64_t)k, (int64_t(1) << 31) - 1);
    const int64_t item_cap = query_items(g->d.m);
    void* buf = nullptr;
    cudaError_t e = cudaMallocAsync(&buf, query_scratch_bytes(cap, item_cap), s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(WTRI_ENOMEM, "query scratch allocation failed");
    }
    Query q;
    query_carve(q, (char*)buf, cap, item_cap);
    set_sweep(q, g, k);
    q.shard = shard;
    q.nshards = nshards;
    q.qbytes = query_bytes_on() ? query_bytes_counter() : nullptr;
    q.gp = gp;
    int rc = WTRI_OK;
    e = cudaMemsetAsync(q.st, 0, sizeof(QState), s);
    if (e != cudaSuccess) rc = cuda_error(e, "query state", __FILE__, __LINE__);
    if (rc == WTRI_OK) {
        ProfScope whole(query_name(P), s, 0.0, 1);
        rc = launch_sweep<P, false>(g->d, q, Out{d_tris, d_weight, d_count, d_keys}, s);
    }
    cudaFreeAsync(buf, s);
    return rc;
}

// ---------------------------------------------------------------------------
// Weighted edge sampling (Algorithm 3, Proposition 4.1, Section 4.1).
//
// Draw: with the edges in the edge order and C[r] = sum_{j<=r} w_j^p (exact
// integers), sample s takes x = word 0 of Philox4x64-10(counter (s,0,0,0),
// key (seed,0)), t = floor(x * Z / 2^64), and the edge is the first r with
// C[r] > t.  Equal weights are contiguous in the edge order (Section 4.1's
// weight classes), so the search runs over the class table (start, weight,
// cumulative mass) and the position inside the class is (t - C_prev) /
// w^p.  Drawn edges are marked in a bitmap; the marked positions, in
// ascending order, are then swept like the exact query (heaviest first) in
// sampled-ownership mode.
// ---------------------------------------------------------------------------
typedef unsigned __int128 u128;

// Philox4x64-10 (Salmon et al., SC'11), first output word only.
__device__ __forceinline__ uint64_t philox_word0(uint64_t c0, uint64_t k0) {
    const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
    const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
    uint64_t c1 = 0, c2 = 0, c3 = 0, k1 = 0;
#pragma unroll
    for (int i = 0; i < 10; i++) {
        const uint64_t hi0 = __umul64hi(M0, c0), lo0 = M0 * c0;
        const uint64_t hi1 = __umul64hi(M1, c2), lo1 = M1 * c2;
        const uint64_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c1 = lo1;
        c3 = lo0;
        c0 = n0;
        c2 = n2;
        k0 += W0;
        k1 += W1;
    }
    return c0;
}

// Ordered compactions (the class starts of the edge order, the drawn
// positions of the bitmap) in three launches: each block counts what it will
// write of its contiguous share, one block scans the counts, each block
// reads its share again and writes.  Both are sparse, so a step without any
// costs its loads and one barrier; an exclusive scan over all positions
// first wrote and read 20 bytes each (160 us at 2e7 edges; now 27).
constexpr int CB_T = 256;

inline unsigned compact_blocks(int64_t work) {  // work: positions or words
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)sm_count() * 8, (work + 1023) / 1024));
}

// Exclusive scan over a CB_T block; *total receives the sum.
__device__ __forceinline__ uint32_t cb_scan(uint32_t x, uint32_t* wsum, uint32_t* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int k = 0; k < CB_T / 32; k++) {
        before += k < w ? wsum[k] : 0u;
        all += wsum[k];
    }
    *total = all;
    __syncthreads();
    return before + inc - x;
}

// Exclusive scan of the blocks' counts in place (one block); *total = sum.
__global__ void __launch_bounds__(1024) k_block_offsets(uint32_t* cnt, int blocks, int64_t* total, int64_t* sentinel,
                                                        int64_t sentinel_value) {
    __shared__ uint32_t wsum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (int base = 0; base < blocks; base += 1024) {
        const int i = base + threadIdx.x;
        const uint32_t x = i < blocks ? cnt[i] : 0u;
        uint32_t inc = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) wsum[w] = inc;
        __syncthreads();
        uint32_t before = carry;
        for (int k = 0; k < 32; k++) {
            before += k < w ? wsum[k] : 0u;
            carry += wsum[k];
        }
        if (i < blocks) cnt[i] = before + inc - x;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *total = carry;
        if (sentinel) sentinel[carry] = sentinel_value;
    }
}

// The class starts among four positions from r on: bit i set when position
// r + i's weight differs from the one before.
__device__ __forceinline__ uint32_t class_starts4(const int32_t* __restrict__ ow, int64_t r, int64_t m) {
    if (r >= m) return 0u;
    int32_t prev = r > 0 ? __ldg(ow + r - 1) : 0;  // weights are positive
    int4 x;
    if (r + 4 <= m) {
        x = __ldg(reinterpret_cast<const int4*>(ow + r));  // r is a multiple of 4, ow 256-byte aligned
    } else {
        x.x = __ldg(ow + r);
        x.y = r + 1 < m ? __ldg(ow + r + 1) : x.x;
        x.z = r + 2 < m ? __ldg(ow + r + 2) : x.y;
        x.w = x.z;
    }
    return (x.x != prev ? 1u : 0u) | (x.y != x.x ? 2u : 0u) | (x.z != x.y ? 4u : 0u) | (x.w != x.z ? 8u : 0u);
}

// Items of a compaction: four positions' class starts, or a bitmap word.
struct ClassBits {
    static constexpr int PER = 4;  // positions per item
    const int32_t* ow;
    int64_t m;
    __device__ __forceinline__ uint32_t get(int64_t item) const { return class_starts4(ow, 4 * item, m); }
};
struct DrawnBits {
    static constexpr int PER = 32;
    const uint32_t* mark;
    int64_t words;
    __device__ __forceinline__ uint32_t get(int64_t item) const { return item < words ? __ldg(mark + item) : 0u; }
};

template <class Bits>
__global__ void __launch_bounds__(CB_T) k_compact_count(Bits B, int64_t items, uint32_t* cnt) {
    __shared__ uint32_t wsum[CB_T / 32];
    const int64_t per = ((items + gridDim.x - 1) / gridDim.x + CB_T - 1) / CB_T * CB_T;
    const int64_t beg = (int64_t)blockIdx.x * per, end = min(items, beg + per);
    uint32_t c = 0, total;
#pragma unroll 4
    for (int64_t i = beg + threadIdx.x; i < end; i += CB_T) c += __popc(B.get(i));
    cb_scan(c, wsum, &total);
    if (threadIdx.x == 0) cnt[blockIdx.x] = total;
}

template <class Bits, class T>
__global__ void __launch_bounds__(CB_T) k_compact_write(Bits B, int64_t items, const uint32_t* cnt, T* out) {
    __shared__ uint32_t wsum[CB_T / 32];
    const int64_t per = ((items + gridDim.x - 1) / gridDim.x + CB_T - 1) / CB_T * CB_T;
    const int64_t beg = (int64_t)blockIdx.x * per, end = min(items, beg + per);
    int64_t off = cnt[blockIdx.x];
    constexpr int U = 4;
    for (int64_t i0 = beg; i0 < end; i0 += U * CB_T) {
        uint32_t b[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = i0 + u * CB_T + threadIdx.x;
            b[u] = i < end ? B.get(i) : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (!__syncthreads_or(b[u] != 0u)) continue;
            uint32_t total;
            int64_t o = off + cb_scan((uint32_t)__popc(b[u]), wsum, &total);
            const int64_t first = (i0 + u * CB_T + threadIdx.x) * Bits::PER;
            for (uint32_t x = b[u]; x; x &= x - 1) out[o++] = (T)(first + __ffs(x) - 1);
            off += total;
        }
    }
}

// The positions of the set bits, ascending, to out; their number to *total
// (and `end` after the last one when sentinel is set).  cnt: compact_blocks.
template <class Bits, class T>
int ordered_compact(const Bits& B, int64_t items, uint32_t* cnt, T* out, int64_t* total, int64_t* sentinel, int64_t end,
                    cudaStream_t s) {
    const unsigned g = compact_blocks(items);
    k_compact_count<Bits><<<g, CB_T, 0, s>>>(B, items, cnt);
    k_block_offsets<<<1, 1024, 0, s>>>(cnt, (int)g, total, sentinel, end);
    k_compact_write<Bits, T><<<g, CB_T, 0, s>>>(B, items, cnt, out);
    WTRI_CUDA(cudaGetLastError());
    return WTRI_OK;
}

// Inclusive prefix of class masses count * w^p, one block (classes are few:
// one per distinct weight).
template <int P>
__global__ void __launch_bounds__(1024) k_class_mass(const int64_t* __restrict__ cls_total,
                                                     const int64_t* __restrict__ cstart,
                                                     const int32_t* __restrict__ ow,
                                                     u128* __restrict__ cmass) {
    __shared__ u128 warp_sum[32];
    __shared__ u128 carry;
    const int64_t nc = *cls_total;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int64_t base = 0; base < nc; base += 1024) {
        const int64_t c = base + threadIdx.x;
        u128 x = 0;
        if (c < nc) {
            const u128 wv = (u128)(uint64_t)__ldg(ow + cstart[c]);
            // w^p: p = 2 squares, p = 1 keeps, p = 0 gives 1 (uniform draws)
            x = (u128)(uint64_t)(cstart[c + 1] - cstart[c]) *
                (P == P_TWO ? wv * wv : (P == P_GEO ? (u128)1 : wv));
        }
        u128 inc = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t lo = __shfl_up_sync(0xffffffffu, (uint64_t)inc, o);
            const uint64_t hi = __shfl_up_sync(0xffffffffu, (uint64_t)(inc >> 64), o);
            if (lane >= o) inc += ((u128)hi << 64) | lo;
        }
        if (lane == 31) warp_sum[wid] = inc;
        __syncthreads();
        if (threadIdx.x == 0) {
            u128 acc = carry;
            for (int k = 0; k < 32; k++) {
                const u128 t = warp_sum[k];
                warp_sum[k] = acc;
                acc += t;
            }
            carry = acc;
        }
        __syncthreads();
        if (c < nc) cmass[c] = warp_sum[wid] + inc;
        __syncthreads();
    }
}

// (class masses below 2^64 in all, the usual case: 64-bit products and
// divisions; the 128-bit division is a subroutine of hundreds of
// instructions)
template <int P>
__global__ void k_draw(int64_t nsamples, uint64_t seed, const int64_t* __restrict__ cls_total,
                       const int64_t* __restrict__ cstart, const int32_t* __restrict__ ow,
                       const u128* __restrict__ cmass, uint32_t* __restrict__ mark) {
    const int64_t nc = *cls_total;
    const u128 Z = cmass[nc - 1];
    const uint64_t zl = (uint64_t)Z, zh = (uint64_t)(Z >> 64);
    const uint64_t* low = reinterpret_cast<const uint64_t*>(cmass);  // low words at even places
    for (int64_t sidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; sidx < nsamples;
         sidx += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t x = philox_word0((uint64_t)sidx, seed);
        int64_t lo = 0, hi = nc;  // first class with mass > t = floor(x * Z / 2^64)
        uint64_t place;
        if (zh == 0) {
            const uint64_t t = __umul64hi(x, zl);
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (__ldg(low + 2 * mid) > t) hi = mid;
                else lo = mid + 1;
            }
            const uint64_t prev = lo > 0 ? __ldg(low + 2 * lo - 2) : 0ull;
            const uint64_t wv = (uint64_t)__ldg(ow + __ldg(cstart + lo));
            place = (t - prev) / (P == P_TWO ? wv * wv : (P == P_GEO ? 1ull : wv));
        } else {
            const u128 t = (u128)x * zh + (u128)__umul64hi(x, zl);
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (cmass[mid] > t) hi = mid;
                else lo = mid + 1;
            }
            const u128 prev = lo > 0 ? cmass[lo - 1] : (u128)0;
            const u128 wv = (u128)(uint64_t)__ldg(ow + cstart[lo]);
            place = (uint64_t)((t - prev) / (P == P_TWO ? wv * wv : (P == P_GEO ? (u128)1 : wv)));
        }
        const int64_t r = __ldg(cstart + lo) + (int64_t)place;
        // heavy edges are drawn thousands of times: look before the atomic (a
        // stale reading only repeats it)
        const uint32_t bit = 1u << (r & 31);
        if (!(__ldcg(mark + (r >> 5)) & bit)) atomicOr(mark + (r >> 5), bit);
    }
}

inline unsigned grid_of(int64_t work) {
    const int64_t cap = (int64_t)sm_count() * 16;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(cap, (work + 255) / 256));
}

// Draws the samples into a bitmap over edge-order positions (words =
// ceil(m/32), zeroed here).  Scratch: cmass (m u128), cstart (m+1 int64), the
// number of classes, block counts.
template <int P>
int draw_samples(const wtri_graph* g, int64_t nsamples, uint64_t seed, uint32_t* mark,
                 cudaStream_t s) {
    const DevGraph& G = g->d;
    const int64_t m = G.m, words = (m + 31) / 32, items = (m + 3) / 4;
    const size_t bytes = 16 * (size_t)m + 8 * (size_t)(m + 2) + 4 * (size_t)compact_blocks(items) + 256;
    void* buf = nullptr;
    if (cudaMallocAsync(&buf, bytes, s) != cudaSuccess) {
        cudaGetLastError();
        return set_error(WTRI_ENOMEM, "sampling scratch allocation failed");
    }
    u128* cmass = (u128*)buf;
    int64_t* cstart = (int64_t*)(cmass + m);
    int64_t* nc = cstart + m + 1;
    uint32_t* cnt = (uint32_t*)(nc + 1);
    WTRI_CUDA(cudaMemsetAsync(mark, 0, 4 * (size_t)words, s));
    {
        ProfScope ps("sample_class_table", s, 12.0 * m, 4);
        WTRI_TRY(ordered_compact(ClassBits{G.ord_w, m}, items, cnt, cstart, nc, cstart, m, s));
        k_class_mass<P><<<1, 1024, 0, s>>>(nc, cstart, G.ord_w, cmass);
    }
    {
        ProfScope ps("sample_draw", s, 0.0, 1);
        k_draw<P><<<grid_of(nsamples), 256, 0, s>>>(nsamples, seed, nc, cstart, G.ord_w, cmass, mark);
    }
    WTRI_CUDA(cudaGetLastError());
    WTRI_CUDA(cudaFreeAsync(buf, s));
    return WTRI_OK;
}

template <int P>
int run_sample(const wtri_graph* g, int32_t k, int64_t nsamples, uint64_t seed, wtri_tri* d_tris,
               double* d_weight, int32_t* d_count, cudaStream_t s, int scale) {
    const DevGraph& G = g->d;
    const int64_t m = G.m, words = (m + 31) / 32;
    const uint32_t cap = (uint32_t)std::min<int64_t>(
        (int64_t(1) << 20) * scale + 16 * (int64_t)k, (int64_t(1) << 31) - 1);
    const int64_t item_cap = query_items(m);
    const size_t qbytes = query_scratch_bytes(cap, item_cap);
    const size_t sbytes = 4 * (size_t)words + 16 + 4 * (size_t)compact_blocks(words) + 4 * (size_t)m + 256;
    void* buf = nullptr;
    if (cudaMallocAsync(&buf, qbytes + sbytes, s) != cudaSuccess) {
        cudaGetLastError();
        return set_error(WTRI_ENOMEM, "sampling query scratch allocation failed");
    }
    Query q;
    char* p = query_carve(q, (char*)buf, cap, item_cap);
    set_sweep(q, g, k);
    uint32_t* mark = (uint32_t*)p;
    p += 4 * (size_t)words;
    p = (char*)(((uintptr_t)p + 7) & ~(uintptr_t)7);
    int64_t* count = (int64_t*)p;
    p += 8;
    uint32_t* cnt = (uint32_t*)p;
    p += 4 * (size_t)compact_blocks(words);
    int32_t* list = (int32_t*)p;
    q.smark = mark;
    q.slist = list;
    q.total_dev = count;  // the number of drawn edges stays on the device
    auto run = [&]() -> int {
        WTRI_CUDA(cudaMemsetAsync(q.st, 0, sizeof(QState), s));
        ProfScope whole(P == P_ONE ? "sample_p=1" : (P == P_TWO ? "sample_p=2" : "sample_p=0"), s, 0.0, 0);
        WTRI_TRY(draw_samples<P>(g, nsamples, seed, mark, s));
        {
            ProfScope ps("sample_compact", s, 8.0 * words, 3);
            WTRI_TRY(ordered_compact(DrawnBits{mark, words}, words, cnt, list, count, (int64_t*)nullptr, 0, s));
        }
        ProfScope ps("sample_sweep", s, 0.0, 1);
        return launch_sweep<P, true>(G, q, Out{d_tris, d_weight, d_count, nullptr}, s);
    };
    const int rc = run();
    cudaFreeAsync(buf, s);
    return rc;
}

}  // namespace

uint32_t first_wait_limit() { return g_wait_first.load(std::memory_order_relaxed); }
uint32_t later_wait_limit() { return g_wait_later.load(std::memory_order_relaxed); }

int topk_device(const wtri_graph* g, int pcode, int32_t k, wtri_tri* d_tris, double* d_weight,
                int32_t* d_count, cudaStream_t stream, int retry_scale, int shard, int nshards,
                unsigned long long* d_keys, double gp) {
    switch (pcode) {
        case P_MIN:
            return run_query<P_MIN>(g, k, d_tris, d_weight, d_count, stream, retry_scale, shard, nshards, d_keys, gp);
        case P_ONE:
            return run_query<P_ONE>(g, k, d_tris, d_weight, d_count, stream, retry_scale, shard, nshards, d_keys, gp);
        case P_TWO:
            return run_query<P_TWO>(g, k, d_tris, d_weight, d_count, stream, retry_scale, shard, nshards, d_keys, gp);
        case P_GEO:
            return run_query<P_GEO>(g, k, d_tris, d_weight, d_count, stream, retry_scale, shard, nshards, d_keys, gp);
        case P_GEN:
            return run_query<P_GEN>(g, k, d_tris, d_weight, d_count, stream, retry_scale, shard, nshards, d_keys, gp);
        default:
            return run_query<P_MAX>(g, k, d_tris, d_weight, d_count, stream, retry_scale, shard, nshards, d_keys, gp);
    }
}

}  // namespace wtri

// ---------------------------------------------------------------------------
// Query variant that allocates nothing.
//
// For callers that may not allocate device memory once they are running:
// for example a server whose device memory is all handed to its own caching
// allocator at start-up, or a latency-critical loop that must never wait on
// the allocator.  The query's scratch (status word, candidate buffer,
// items) lives in one fixed array compiled into the library.
// Every GPU that loads the library keeps this array (NOALLOC_BYTES, about
// 28 MB) until the process exits.  All calls share it: the state is cleared at
// the start of each call.  A call that cleared it under a running sweep would
// take the barrier's counter away from blocks that wait for it, so each call
// waits on the device for the one before it (an event; captured calls, which
// cannot wait for one outside their graph, are left to the caller).
// ---------------------------------------------------------------------------
namespace wtri {
namespace {

constexpr uint32_t NOALLOC_CAP = 1u << 20;     // candidates
constexpr int64_t NOALLOC_ITEMS = 46592;       // edges of a round (an item each)
constexpr int32_t NOALLOC_K_MAX = 16384;
// state, keys, triples, items and the wedges before each item, as query_carve lays them out
constexpr size_t NOALLOC_BYTES =
    256 + (size_t)NOALLOC_CAP * 24 + (size_t)NOALLOC_ITEMS * (sizeof(Item) + sizeof(unsigned long long));
static_assert(sizeof(QState) <= 256, "the state fits its slot");
static_assert(NOALLOC_ITEMS % 32 == 0, "every piece is a multiple of 256 bytes");

static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
struct Noalloc {
    std::mutex mu;  // held while a call is enqueued
    void* ptr = nullptr;
    cudaEvent_t last = nullptr;  // the end of the last call
};
Noalloc g_noalloc[NOALLOC_MAX_DEVICES];

// The fixed array of the current device (with that device current), its
// address looked up once, locked for a call.
int noalloc_scratch(Noalloc** out, std::unique_lock<std::mutex>* lock) {
    int dev = 0;
    WTRI_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES)
        return set_error(WTRI_EUNSUPPORTED, "device index above 63");
    Noalloc& N = g_noalloc[dev];
    *lock = std::unique_lock<std::mutex>(N.mu);
    if (!N.ptr) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            cudaGetLastError();
            return cuda_error(e == cudaSuccess ? cudaErrorInvalidSymbol : e,
                              "cudaGetSymbolAddress(static query scratch)", __FILE__, __LINE__);
        }
        if (!N.last) WTRI_CUDA(cudaEventCreateWithFlags(&N.last, cudaEventDisableTiming));
        N.ptr = p;
    }
    *out = &N;
    return WTRI_OK;
}

template <int P>
int run_query_noalloc(const wtri_graph* g, int32_t k, wtri_tri* d_tris, double* d_weight,
                      int32_t* d_count, cudaStream_t s, double gp) {
    Noalloc* N = nullptr;
    std::unique_lock<std::mutex> lock;
    WTRI_TRY(noalloc_scratch(&N, &lock));
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    WTRI_CUDA(cudaStreamIsCapturing(s, &capture));
    const bool ordered = capture == cudaStreamCaptureStatusNone;
    if (ordered) WTRI_CUDA(cudaStreamWaitEvent(s, N->last, 0));
    Query q;
    query_carve(q, (char*)N->ptr, NOALLOC_CAP, NOALLOC_ITEMS);
    set_sweep(q, g, k);
    q.gp = gp;
    // The array keeps the previous call's contents: reset the state
    // (counters, threshold, barrier, error bits).
    WTRI_CUDA(cudaMemsetAsync(q.st, 0, sizeof(QState), s));
    WTRI_TRY((launch_sweep<P, false>(g->d, q, Out{d_tris, d_weight, d_count, nullptr}, s)));
    if (ordered) WTRI_CUDA(cudaEventRecord(N->last, s));
    count_launches(1);
    return WTRI_OK;
}

}  // namespace
int sample_topk_device(const wtri_graph* g, int pcode, int32_t k, int64_t nsamples, uint64_t seed,
                       wtri_tri* d_tris, double* d_weight, int32_t* d_count, cudaStream_t stream,
                       int retry_scale) {
    if (pcode == P_ONE)
        return run_sample<P_ONE>(g, k, nsamples, seed, d_tris, d_weight, d_count, stream, retry_scale);
    if (pcode == P_GEO)
        return run_sample<P_GEO>(g, k, nsamples, seed, d_tris, d_weight, d_count, stream, retry_scale);
    return run_sample<P_TWO>(g, k, nsamples, seed, d_tris, d_weight, d_count, stream, retry_scale);
}

int sample_edges_device(const wtri_graph* g, int pcode, int64_t nsamples, uint64_t seed,
                        uint32_t* d_mark, cudaStream_t stream) {
    if (pcode == P_ONE) return draw_samples<P_ONE>(g, nsamples, seed, d_mark, stream);
    if (pcode == P_GEO) return draw_samples<P_GEO>(g, nsamples, seed, d_mark, stream);
    return draw_samples<P_TWO>(g, nsamples, seed, d_mark, stream);
}

}  // namespace wtri

extern "C" WTRI_API int wtri_topk_device_noalloc(const wtri_graph* g, double p, int32_t k,
                                                 wtri_tri* d_tris, double* d_weight,
                                                 int32_t* d_count, void* stream) {
    using namespace wtri;
    if (!g) return set_error(WTRI_EINVAL, "graph is NULL");
    if (k <= 0) return set_error(WTRI_EINVAL, "k must be positive");
    if (k > NOALLOC_K_MAX)
        return set_error(WTRI_EINVAL, "k above 16384, the most the fixed query scratch supports");
    int code = 0;
    WTRI_TRY(p_to_code_for(p, g, &code));
    if (!d_tris || !d_weight || !d_count) return set_error(WTRI_EINVAL, "output pointers are NULL");
    cudaStream_t s = stream ? (cudaStream_t)stream : g->stream;
    if (g->d.m == 0) {
        WTRI_CUDA(cudaMemsetAsync(d_count, 0, sizeof(int32_t), s));
        return WTRI_OK;
    }
    switch (code) {
        case P_MIN: return run_query_noalloc<P_MIN>(g, k, d_tris, d_weight, d_count, s, p);
        case P_ONE: return run_query_noalloc<P_ONE>(g, k, d_tris, d_weight, d_count, s, p);
        case P_TWO: return run_query_noalloc<P_TWO>(g, k, d_tris, d_weight, d_count, s, p);
        case P_GEO: return run_query_noalloc<P_GEO>(g, k, d_tris, d_weight, d_count, s, p);
        case P_GEN: return run_query_noalloc<P_GEN>(g, k, d_tris, d_weight, d_count, s, p);
        default: return run_query_noalloc<P_MAX>(g, k, d_tris, d_weight, d_count, s, p);
    }
}


// ---------------------------------------------------------------------------
// Instrumented query byte counter (one per device).
// ---------------------------------------------------------------------------
namespace wtri {
namespace {
__device__ unsigned long long g_query_bytes;
std::atomic<int> g_query_bytes_on{0};
std::mutex g_qb_mu;
unsigned long long* g_qb_ptr[64] = {};
}  // namespace

bool query_bytes_on() { return g_query_bytes_on.load(std::memory_order_relaxed) != 0; }

unsigned long long* query_bytes_counter() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(g_qb_mu);
    if (!g_qb_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_query_bytes) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        g_qb_ptr[dev] = (unsigned long long*)p;
    }
    return g_qb_ptr[dev];
}

}  // namespace wtri

extern "C" WTRI_API int wtri_query_bytes(int on, int reset, unsigned long long* bytes) {
    using namespace wtri;
    unsigned long long* d = query_bytes_counter();
    if (!d) return set_error(WTRI_ECUDA, "query byte counter unavailable on this device");
    WTRI_CUDA(cudaDeviceSynchronize());
    if (bytes) WTRI_CUDA(cudaMemcpy(bytes, d, sizeof(unsigned long long), cudaMemcpyDeviceToHost));
    if (reset) WTRI_CUDA(cudaMemset(d, 0, sizeof(unsigned long long)));
    g_query_bytes_on.store(on ? 1 : 0);
    return WTRI_OK;
}

extern "C" WTRI_API int wtri_debug_set_wait_limit(int64_t polls) {
    return wtri_debug_set_wait_limits(polls, -1);
}

extern "C" WTRI_API int wtri_debug_set_wait_limits(int64_t first, int64_t later) {
    wtri::g_wait_first.store(wtri::poll_limit(first));
    wtri::g_wait_later.store(wtri::poll_limit(later));
    return WTRI_OK;
}
