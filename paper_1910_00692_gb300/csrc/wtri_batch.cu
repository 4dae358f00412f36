// Batched exact top-k: many (graph, p, k) queries in one launch.
//
// Every query runs the sweep of the single query (wtri_query.cuh), with its
// own state, threshold and candidate buffer.  One kernel holds the whole GPU
// (a cooperative launch, one block per SM).  Queries whose expected work is
// above an even share get a team of SMs each, in proportion to it; every
// other block, and every team once its query is answered, works as PARTS
// parts that take the remaining queries from a list, largest first, one query
// per part: the phases of a query wait only for its own part or team, and its
// results are ranked there.  Most queries are bound by latency, so many side
// by side take little longer than one; the teams keep the few large ones
// from being the tail (64 graphs of up to 2e5 edges, one block each: 3.5 ms).
// The launch is captured in a CUDA graph.
#include "wtri_query.cuh"

#include <vector>

namespace wtri {
namespace {

constexpr int PT = 512;                   // threads of a part
constexpr int PARTS = TGRID / PT;         // parts of a block
// Items, shared evenly by the SMs: a query has those of its SMs.  A server's
// batches keep to the bytes its admission counts.
constexpr int64_t POOL_SERVED = 180000;
constexpr int64_t POOL_BATCH = 640000;
static_assert(POOL_BATCH + (1 << 18) < (1 << (64 - ITEM_SHIFT)), "a team's items, and 32 more per warp, are counted in 20 bits");
// Most teams of a launch: one per SM.  (With 64, 100 equal queries left 36 to the
// parts: 200,000 random edges each, p = 1, k = 1,000, 8.5 ms; now 5.4.)
constexpr int TEAMS = 152;
constexpr int64_t BATCH_FIRST = 64;       // first round of a batched query (edges)
constexpr int32_t BATCH_GROWTH = 8;       // growth of its rounds

struct BatchDev {
    const DevGraph* graphs;
    const Query* queries;
    const Out* outs;
    const int32_t* pcodes;
    const int32_t* order;  // the queries answered by parts, largest first
    int32_t count;
    int32_t* cursor;
    Item* items;           // per_sm for each block
    unsigned long long* ibase;
    int64_t per_sm;
};

// Teams of one launch: team t has blocks [blk[t], blk[t + 1]) and query qi[t].
struct TeamList {
    int32_t n;
    int32_t qi[TEAMS];
    int16_t blk[TEAMS + 1];
};

struct PartSmem {
    SweepSmem<PT> sweep;
    DevGraph G;
    Query q;
    Out o;
    QState st;
    int32_t at;
};

// (not inlined: the instantiations would share one frame of registers)
template <int P>
__device__ __noinline__ void sweep_part(PartSmem& S) {
    BlockTeam<PT> T;
    sweep<P, false>(S.G, S.q, S.o, T, S.sweep);
}

template <int P>
__device__ __noinline__ bool sweep_team(const DevGraph& G, const Query& q, const Out& o, SweepSmem<TGRID>& S,
                                        uint32_t blk0, uint32_t nblk) {
    GridTeam<TGRID> T;
    T.limit = q.wait_first;
    T.blk0 = blk0;
    T.nblk = nblk;
    T.gone = &S.sel.gone;
    return sweep<P, false>(G, q, o, T, S);
}

union BatchSmem {
    SweepSmem<TGRID> team;
    PartSmem part[PARTS];
};

__global__ void __launch_bounds__(TGRID, 1) k_sweep_batch(BatchDev B, TeamList L) {
    extern __shared__ __align__(16) unsigned char batch_smem[];
    BatchSmem& S = *reinterpret_cast<BatchSmem*>(batch_smem);
    __shared__ DevGraph G;
    __shared__ Query q;
    __shared__ Out o;
    int t = 0;  // this block's team: the first that ends after it
    for (int n = L.n; n > 0;) {
        const int h = n / 2;
        if ((int)blockIdx.x >= L.blk[t + h + 1]) t += h + 1, n -= h + 1;
        else n = h;
    }
    if (t < L.n) {
        const int32_t qi = L.qi[t];
        const uint32_t blk0 = (uint32_t)L.blk[t], nblk = (uint32_t)(L.blk[t + 1] - L.blk[t]);
        if (threadIdx.x == 0) {
            G = B.graphs[qi];
            q = B.queries[qi];
            o = B.outs[qi];
            q.items = B.items + B.per_sm * blk0;
            q.ibase = B.ibase + B.per_sm * blk0;
            q.item_cap = B.per_sm * nblk;
            S.team.sel.gone = 0;
        }
        __syncthreads();
        bool ok;
        switch (B.pcodes[qi]) {
            case P_MIN: ok = sweep_team<P_MIN>(G, q, o, S.team, blk0, nblk); break;
            case P_ONE: ok = sweep_team<P_ONE>(G, q, o, S.team, blk0, nblk); break;
            case P_TWO: ok = sweep_team<P_TWO>(G, q, o, S.team, blk0, nblk); break;
            case P_GEO: ok = sweep_team<P_GEO>(G, q, o, S.team, blk0, nblk); break;
            default: ok = sweep_team<P_MAX>(G, q, o, S.team, blk0, nblk); break;
        }
        // gave up: the other blocks may still be using this one's items
        if (!ok) return;
        __syncthreads();
    }
    const int p = threadIdx.x / PT;
    const Part<PT> part;
    PartSmem& M = S.part[p];
    for (;;) {
        if (part.tid() == 0) {
            M.at = atomicAdd(B.cursor, 1);
            if (M.at < B.count) {
                const int32_t qi = B.order[M.at];
                const int64_t per = B.per_sm / PARTS;
                M.G = B.graphs[qi];
                M.q = B.queries[qi];
                M.o = B.outs[qi];
                M.st = QState{};
                M.q.st = &M.st;
                M.q.items = B.items + B.per_sm * blockIdx.x + per * p;
                M.q.ibase = B.ibase + B.per_sm * blockIdx.x + per * p;
                M.q.item_cap = per;
            }
        }
        part.sync();
        const int32_t at = M.at;
        if (at >= B.count) return;
        switch (B.pcodes[B.order[at]]) {
            case P_MIN: sweep_part<P_MIN>(M); break;
            case P_ONE: sweep_part<P_ONE>(M); break;
            case P_TWO: sweep_part<P_TWO>(M); break;
            case P_GEO: sweep_part<P_GEO>(M); break;
            default: sweep_part<P_MAX>(M); break;
        }
        part.sync();
    }
}

// Expected microseconds of a query on one part (half an SM), from queries of
// k = 500 timed on graphs of 1e4 to 2e7 edges.  The arithmetic means, the
// geometric mean and the maximum are bound by latency and hardly grow with
// the graph: on one whole SM 94 us at 1e4 edges, 151 at 2e5 (the long rows of
// its heaviest edges), 117 at 2e7; on 152 SMs 64-97.  The minimum reads the
// rows of a share of all edges: 348 us on one SM at 1e4 edges, 1,151 at 5e4,
// 1,289 at 2e5, 5,881 at 5e6, 13,990 at 2e7; on 152 SMs 298 at 2e7.
// Above k = 2,048 (SORT_MAX) the selects and the ranking take about 1 us per
// result more (304 queries of k = 1,000 / 4,096 / 8,192 on a part each: 1.1 /
// 4.8 / 7.4 ms at p = 1, 4.3 / 9.1 / 13.9 at p = -inf).
double part_us(int pcode, int64_t m, int32_t k) {
    const double x = (double)m, rank = k > SORT_MAX ? (double)k : 0.0;
    if (pcode != P_MIN) return 150.0 + 100.0 * std::min(1.0, x / 2e5) + rank;
    return 300.0 + 900.0 * std::min(1.0, x / 5e4) + 1200.0 * std::min(1.0, x / 2e5) + 1.3e-3 * x + rank;
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

}  // namespace wtri

// ---------------------------------------------------------------------------
// Host side: a batch plan (schedule, buffer layout, descriptors), launching
// it on a stream into one device scratch block, and collecting results.
// Used by wtri_topk_batch and by the serving loop.
// ---------------------------------------------------------------------------
struct wtri_batch_plan {
    int32_t nq = 0;
    int64_t pool = 0;  // items
    std::vector<wtri::DevGraph> hg;
    std::vector<int32_t> pcodes;  // nq, and after them the statuses as they start: one upload
    std::vector<int32_t> ks, tshort;
    std::vector<int32_t> order;  // the queries answered by parts, largest first
    wtri::TeamList teams;
    std::vector<uint32_t> caps;
    std::vector<int64_t> koffs;
    size_t cand_total = 0;
    size_t o_st, o_key, o_tri, o_items, o_ibase, o_cur, o_g, o_q, o_o, o_pc, o_ord, o_otri, o_ow, bytes;
    std::vector<int32_t> stat;
    std::vector<wtri_tri> otri;
    std::vector<double> ow;
};

namespace wtri {

// Candidate slots of one batched query: enough for k plus ties, and for the
// first rounds of a large graph (enumerated before the threshold exists).
uint32_t batch_query_cap(int32_t k, int64_t m) {
    int64_t cap = std::max<int64_t>(16 * (int64_t)k, m / 16);
    cap = std::min<int64_t>(cap, int64_t(1) << 20);
    return (uint32_t)std::max<int64_t>(cap, 16384);
}

// Deals the SMs: a query whose expected time on one part is well above an even
// share of the whole batch gets a team of SMs in proportion to its work, the
// rest are left to the parts.
// The teams' ends are the running sum of their shares, rounded: sizes rounded
// up each gave 16 equal queries 15 teams of 10 SMs and one of two, and of 64
// equal ones 50 teams of three, 14 left to the parts (200,000 random edges
// each, p = 1, k = 1,000: 1.77 and 7.8 ms, now 0.62 and 2.6).
static void plan_teams(BatchPlan* P) {
    const int nq = P->nq, sms = sm_count();
    std::vector<double> us((size_t)nq);
    double total = 0.0;
    for (int i = 0; i < nq; i++) total += us[(size_t)i] = part_us(P->pcodes[(size_t)i], P->hg[(size_t)i].m, P->ks[(size_t)i]);
    std::vector<int32_t> by((size_t)nq);
    for (int i = 0; i < nq; i++) by[(size_t)i] = i;
    std::stable_sort(by.begin(), by.end(), [&](int32_t a, int32_t b) { return us[(size_t)a] > us[(size_t)b]; });
    P->teams.n = 0;
    P->teams.blk[0] = 0;
    P->order.clear();
    const double share = total / ((double)PARTS * sms);  // an even share of one part
    double end = 0.0;
    for (int32_t i : by) {
        const int t = P->teams.n, used = P->teams.blk[t];
        if (us[(size_t)i] > 1.5 * share && us[(size_t)i] > 150.0 && t < TEAMS && used < sms) {
            end += us[(size_t)i] / (PARTS * share);
            P->teams.qi[t] = i;
            P->teams.blk[t + 1] = (int16_t)std::min(sms, std::max(used + 1, (int)(end + 0.5)));
            P->teams.n++;
        } else {
            P->order.push_back(i);
        }
    }
}

BatchPlan* batch_plan_create(const wtri_graph* const* gs, const int32_t* pcodes, const int32_t* ks,
                             int32_t nq, bool served) {
    BatchPlan* P = new (std::nothrow) BatchPlan();
    if (!P) return nullptr;
    P->pool = served ? POOL_SERVED : POOL_BATCH;
    P->nq = nq;
    P->hg.resize((size_t)nq);
    P->pcodes.assign(pcodes, pcodes + nq);
    P->pcodes.resize(2 * (size_t)nq, WTRI_ETIMEOUT);  // until a query is answered
    P->ks.assign(ks, ks + nq);
    P->caps.resize((size_t)nq);
    P->tshort.resize((size_t)nq);
    P->koffs.assign((size_t)nq + 1, 0);
    for (int i = 0; i < nq; i++) {
        const int64_t m = gs[i]->d.m;
        P->hg[(size_t)i] = gs[i]->d;
        P->tshort[(size_t)i] = gs[i]->tune.t_short;
        P->koffs[(size_t)i + 1] = P->koffs[(size_t)i] + ks[i];
        P->caps[(size_t)i] = batch_query_cap(ks[i], m);
        P->cand_total += P->caps[(size_t)i];
    }
    plan_teams(P);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off = al256(off + bytes);
        return o;
    };
    P->o_st = take(sizeof(QState) * (size_t)(P->teams.n + 1));
    P->o_cur = take(64);  // cleared together with the states
    P->o_key = take(8 * P->cand_total);
    P->o_tri = take(16 * P->cand_total);
    P->o_items = take(sizeof(Item) * (size_t)P->pool);
    P->o_ibase = take(8 * (size_t)P->pool);
    P->o_g = take(sizeof(DevGraph) * (size_t)nq);
    P->o_q = take(sizeof(Query) * (size_t)nq);
    P->o_o = take(sizeof(Out) * (size_t)nq);
    P->o_pc = take(8 * (size_t)nq);
    P->o_ord = take(4 * (size_t)nq);
    P->o_otri = take(sizeof(wtri_tri) * (size_t)P->koffs[(size_t)nq]);
    P->o_ow = take(8 * (size_t)P->koffs[(size_t)nq]);
    P->bytes = off;
    return P;
}

size_t batch_plan_bytes(const BatchPlan* P) { return P->bytes; }

void batch_plan_destroy(BatchPlan* P) { delete P; }

// The last instantiated batch graph of this thread on each device.
struct GraphCache {
    cudaGraphExec_t exec = nullptr;
    cudaStream_t stream = nullptr;
    uint64_t instantiations = 0, updates = 0;
};

GraphCache& graph_cache() {
    static thread_local GraphCache cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    return cache[dev];
}

// Uploads the descriptors (small, from pageable memory: the call returns
// once they are staged) and enqueues every kernel of the batch on s.
int batch_plan_launch(BatchPlan* P, void* dbuf, cudaStream_t s, int use_graph) {
    const int nq = P->nq;
    char* B0 = (char*)dbuf;
    QState* st = (QState*)(B0 + P->o_st);
    unsigned long long* ckey = (unsigned long long*)(B0 + P->o_key);
    int4* ctri = (int4*)(B0 + P->o_tri);
    wtri_tri* d_otri = (wtri_tri*)(B0 + P->o_otri);
    double* d_ow = (double*)(B0 + P->o_ow);
    int32_t* d_stat = (int32_t*)(B0 + P->o_pc) + nq;
    std::vector<Query> hq((size_t)nq);
    std::vector<Out> ho((size_t)nq);
    size_t c0 = 0;
    for (int i = 0; i < nq; i++) {
        Query& q = hq[(size_t)i];
        q = Query{};
        q.ckey = ckey + c0;
        q.ctri = ctri + c0;
        q.cap = P->caps[(size_t)i];
        q.k = P->ks[(size_t)i];
        // one schedule (first round, growth) for the whole batch; each query
        // keeps its own graph's t_short
        q.total = P->hg[(size_t)i].m;
        q.first = BATCH_FIRST;
        q.growth = BATCH_GROWTH;
        q.nshards = 1;
        q.t_short = P->tshort[(size_t)i];
        q.wait_first = first_wait_limit();
        q.wait_later = later_wait_limit();
        ho[(size_t)i] = Out{d_otri + P->koffs[(size_t)i], d_ow + P->koffs[(size_t)i], d_stat + i, nullptr};
        c0 += P->caps[(size_t)i];
    }
    for (int t = 0; t < P->teams.n; t++) hq[(size_t)P->teams.qi[t]].st = st + t;
    BatchDev Bd;
    Bd.graphs = (const DevGraph*)(B0 + P->o_g);
    Bd.queries = (const Query*)(B0 + P->o_q);
    Bd.outs = (const Out*)(B0 + P->o_o);
    Bd.pcodes = (const int32_t*)(B0 + P->o_pc);
    Bd.order = (const int32_t*)(B0 + P->o_ord);
    Bd.count = (int32_t)P->order.size();
    Bd.cursor = (int32_t*)(B0 + P->o_cur);
    Bd.items = (Item*)(B0 + P->o_items);
    Bd.ibase = (unsigned long long*)(B0 + P->o_ibase);
    Bd.per_sm = P->pool / sm_count() / (32 * PARTS) * (32 * PARTS);
    WTRI_CUDA(cudaMemcpyAsync((void*)Bd.graphs, P->hg.data(), sizeof(DevGraph) * nq, cudaMemcpyHostToDevice, s));
    WTRI_CUDA(cudaMemcpyAsync((void*)Bd.queries, hq.data(), sizeof(Query) * nq, cudaMemcpyHostToDevice, s));
    WTRI_CUDA(cudaMemcpyAsync((void*)Bd.outs, ho.data(), sizeof(Out) * nq, cudaMemcpyHostToDevice, s));
    WTRI_CUDA(cudaMemcpyAsync((void*)Bd.pcodes, P->pcodes.data(), 8 * (size_t)nq, cudaMemcpyHostToDevice, s));
    if (!P->order.empty())
        WTRI_CUDA(cudaMemcpyAsync((void*)Bd.order, P->order.data(), 4 * P->order.size(), cudaMemcpyHostToDevice, s));
    static std::atomic<uint64_t> done{0};
    WTRI_TRY(smem_optin((const void*)k_sweep_batch, (int)sizeof(BatchSmem), done));
    const size_t clear = P->o_cur + 64 - P->o_st;  // states of the teams, cursor
    auto launch_all = [&]() -> int {
        WTRI_CUDA(cudaMemsetAsync(B0 + P->o_st, 0, clear, s));
        void* args[] = {&Bd, &P->teams};
        WTRI_CUDA(cudaLaunchCooperativeKernel((const void*)k_sweep_batch, dim3((unsigned)sm_count()), dim3(TGRID), args,
                                              sizeof(BatchSmem), s));
        return WTRI_OK;
    };
    int rc = WTRI_OK;
    ProfScope ps("topk_batch", s, 0.0, 1);
    if (use_graph) {
        // The descriptors must have landed before the captured work refers
        // to them only through device pointers: that holds, the copies are
        // ordered on s before the graph launch.  The instantiated graph is
        // kept (per thread and device) and refreshed with
        // cudaGraphExecUpdate for the next batch (always one memset and one
        // launch).
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            rc = launch_all();
            e = cudaStreamEndCapture(s, &graph);  // always leave capture mode
            if (rc != WTRI_OK && e == cudaSuccess) {
                cudaGraphDestroy(graph);
                return rc;
            }
        }
        cudaGraphExec_t exec = nullptr;
        if (e == cudaSuccess) {
            GraphCache& gc = graph_cache();
            if (gc.exec && gc.stream == s) {
                cudaGraphExecUpdateResultInfo info;
                if (cudaGraphExecUpdate(gc.exec, graph, &info) == cudaSuccess) {
                    exec = gc.exec;
                    gc.updates++;
                } else {
                    cudaGetLastError();
                    cudaGraphExecDestroy(gc.exec);
                    gc.exec = nullptr;
                }
            }
            if (!exec) {
                e = cudaGraphInstantiate(&exec, graph, 0);
                if (e == cudaSuccess) {
                    gc.exec = exec;
                    gc.stream = s;
                    gc.instantiations++;
                }
            }
        }
        if (e == cudaSuccess) e = cudaGraphLaunch(exec, s);
        if (graph) cudaGraphDestroy(graph);
        if (e != cudaSuccess) rc = cuda_error(e, "batch graph", __FILE__, __LINE__);
    } else {
        rc = launch_all();
        cudaError_t e = cudaGetLastError();
        if (rc == WTRI_OK && e != cudaSuccess) rc = cuda_error(e, "batch launch", __FILE__, __LINE__);
    }
    return rc;
}

// Copies statuses and results to the plan's host vectors (synchronizes s).
int batch_plan_collect(BatchPlan* P, void* dbuf, cudaStream_t s) {
    const int nq = P->nq;
    char* B0 = (char*)dbuf;
    P->stat.assign((size_t)nq, 0);
    P->otri.resize((size_t)P->koffs[(size_t)nq]);
    P->ow.resize((size_t)P->koffs[(size_t)nq]);
    WTRI_CUDA(cudaMemcpyAsync(P->stat.data(), (int32_t*)(B0 + P->o_pc) + nq, 4 * (size_t)nq, cudaMemcpyDeviceToHost,
                              s));
    WTRI_CUDA(cudaMemcpyAsync(P->otri.data(), B0 + P->o_otri, sizeof(wtri_tri) * P->otri.size(),
                              cudaMemcpyDeviceToHost, s));
    WTRI_CUDA(cudaMemcpyAsync(P->ow.data(), B0 + P->o_ow, 8 * P->ow.size(), cudaMemcpyDeviceToHost, s));
    WTRI_CUDA(cudaStreamSynchronize(s));
    for (int i = 0; i < nq; i++)
        if (P->stat[(size_t)i] > P->ks[(size_t)i]) P->stat[(size_t)i] = WTRI_ECUDA;  // no count: not to be copied by
    return WTRI_OK;
}

int32_t batch_plan_status(const BatchPlan* P, int i) { return P->stat[(size_t)i]; }
const wtri_tri* batch_plan_tris(const BatchPlan* P, int i) { return P->otri.data() + P->koffs[(size_t)i]; }
const double* batch_plan_weights(const BatchPlan* P, int i) { return P->ow.data() + P->koffs[(size_t)i]; }

// One query with larger bounded buffers (for queries that overflowed a
// batch's); results to host arrays.
int topk_retry_host(const wtri_graph* g, int pcode, int32_t k, cudaStream_t s, wtri_tri* htri,
                    double* hw, int32_t* count) {
    void* dbuf = nullptr;
    WTRI_CUDA(cudaMallocAsync(&dbuf, (sizeof(wtri_tri) + 8) * (size_t)k + 64, s));
    wtri_tri* dt = (wtri_tri*)dbuf;
    double* dw = (double*)((char*)dbuf + ((sizeof(wtri_tri) * (size_t)k + 15) & ~size_t(15)));
    int32_t* dc = (int32_t*)(dw + k);
    int32_t cnt = WTRI_ENOMEM;
    int rc = WTRI_OK;
    for (int scale = 8; scale <= 64 && cnt == WTRI_ENOMEM && rc == WTRI_OK; scale *= 8) {
        rc = topk_device(g, pcode, k, dt, dw, dc, s, scale);
        if (rc == WTRI_OK) {
            cudaError_t e = cudaMemcpyAsync(&cnt, dc, 4, cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) rc = cuda_error(e, "retry", __FILE__, __LINE__);
        }
    }
    if (rc == WTRI_OK && cnt > k) cnt = WTRI_ECUDA;
    if (rc == WTRI_OK && cnt < 0) rc = set_error(cnt, "query failed on retry with larger buffers");
    if (rc == WTRI_OK && cnt > 0) {
        cudaError_t e = cudaMemcpyAsync(htri, dt, sizeof(wtri_tri) * (size_t)cnt, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaMemcpyAsync(hw, dw, 8 * (size_t)cnt, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = cuda_error(e, "retry copy", __FILE__, __LINE__);
    }
    cudaFreeAsync(dbuf, s);
    if (rc == WTRI_OK) *count = cnt;
    return rc;
}

cudaStream_t own_stream() {
    static thread_local cudaStream_t own[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (!own[dev] && cudaStreamCreateWithFlags(&own[dev], cudaStreamNonBlocking) != cudaSuccess)
        return nullptr;
    return own[dev];
}

// Runs nq queries; results to caller host arrays.  Queries whose bounded
// buffers overflowed are re-run one by one with larger buffers.
int topk_batch(const wtri_graph* const* gs, const int32_t* pcodes, const int32_t* ks, int32_t nq,
               wtri_result* outs, cudaStream_t user_stream, int use_graph) {
    // The batch runs on a stream of its own (the legacy default stream cannot
    // be captured), ordered after the work already queued on the caller's.
    cudaStream_t s = own_stream();
    if (!s) return set_error(WTRI_ECUDA, "could not create the batch stream");
    {
        cudaEvent_t ev;
        WTRI_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        cudaError_t e = cudaEventRecord(ev, user_stream);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ev, 0);
        cudaEventDestroy(ev);
        WTRI_CUDA(e);
    }
    BatchPlan* P = batch_plan_create(gs, pcodes, ks, nq, false);
    if (!P) return set_error(WTRI_ENOMEM, "host allocation failed");
    void* buf = nullptr;
    if (cudaMallocAsync(&buf, P->bytes, s) != cudaSuccess) {
        cudaGetLastError();
        batch_plan_destroy(P);
        return set_error(WTRI_ENOMEM, "batch scratch allocation failed");
    }
    int rc = batch_plan_launch(P, buf, s, use_graph);
    if (rc == WTRI_OK) rc = batch_plan_collect(P, buf, s);
    cudaFreeAsync(buf, s);
    for (int i = 0; i < nq && rc == WTRI_OK; i++) {
        const int32_t c = P->stat[(size_t)i];
        if (c == WTRI_ENOMEM) {
            rc = topk_retry_host(gs[i], pcodes[i], ks[i], s, outs[i].tris, outs[i].weight, &outs[i].count);
            continue;
        }
        if (c < 0) {
            rc = set_error(c, "device-side error in batched query " + std::to_string(i));
            break;
        }
        std::copy(P->otri.begin() + P->koffs[(size_t)i], P->otri.begin() + P->koffs[(size_t)i] + c,
                  outs[i].tris);
        std::copy(P->ow.begin() + P->koffs[(size_t)i], P->ow.begin() + P->koffs[(size_t)i] + c,
                  outs[i].weight);
        outs[i].count = c;
    }
    batch_plan_destroy(P);
    return rc;
}

}  // namespace wtri
