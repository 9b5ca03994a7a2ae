// rcm_batch.cu -- batched ordering: G independent graphs stacked block-diagonally, ordered in one
// persistent launch. Each CTA pops graphs from a device work queue and runs the whole ordering of
// a graph with CTA barriers only (Engine<true>), so thousands of small graphs overlap on the GPU
// with no per-graph launch and no grid-wide barrier. The paper orders one matrix at a time; the
// batch only multiplies independent instances of the same method, with the same tie rules.
#include <algorithm>
#include <mutex>

#include "rcm_batch.cuh"
#include "rcm_cc.cuh"
#include "rcm_engine.cuh"
#include "rcm_host.hpp"
#include "rcm_internal.cuh"
#include "rcm_prep.cuh"

namespace rcm {

// The local sweeps' lists take levels of about a thousand vertices. The table takes the shared memory
// that is left, up to kBatchSlots: the emptier it is, the fewer probes (levels of 500 vertices on 512
// threads: claims 2,500 -> 1,650 cycles with 8,192 slots instead of 2,048), but what it takes is L1 that
// wider levels, in global memory, read their rows through (twenty graphs of up to 839,000 vertices, 3D grids
// among them: 31.8 ms with 8,192, 19.2 with 4,096, 17.1 with 2,048; a 900,000-point mesh 30.5, 30.6 and 32.1).
constexpr int kBatchEntries = 3072;
constexpr int kBatchSlots = 4096;
constexpr int kBatchMinSlots = 2048;
// What a launch takes of an SM where its largest graph is beyond the largest bitmap (1.46M vertices): that
// graph takes the longest, all in global memory, and wants L1 (graphs of 1.2M, 1.7M and 2.5M vertices: 165 ms
// with the largest bitmap, 98 so; 137 on the 256 threads that were the default before the local sweeps).
constexpr int kBatchLeanSmem = 128 * 1024;
constexpr int kBatchStaticSmem = 18 * 1024;  // EngineSmem and the rest, rounded up
constexpr int kSmemPerSm = 227 * 1024;

// The local state of a launch of G graphs, the largest of max_n vertices, that wants up to per_sm CTAs
// on an SM: the largest graph its bitmap holds and the slots of its table.
struct LocalShape {
    int cap, slots;
};
static LocalShape local_shape(int max_n, int G, int per_sm, int sms) {
    const int want = std::max(1, std::min(per_sm, (G + sms - 1) / sms));
    auto shape = [&](long long bytes) {
        const long long bitmap = bytes - (long long)local_bytes(0, kBatchMinSlots, kBatchEntries);
        return (int)std::min<long long>(std::min(max_n, kLocalMax), std::max<long long>(0, bitmap / 16 * 128));
    };
    long long bytes = kSmemPerSm / want - 1024 - kBatchStaticSmem;
    if (want == 1 && shape(bytes) < max_n) bytes = kBatchLeanSmem - 1024 - kBatchStaticSmem;
    LocalShape l{shape(bytes), kBatchMinSlots};
    while (l.slots < kBatchSlots && (long long)local_bytes(l.cap, 2 * l.slots, kBatchEntries) <= bytes) l.slots *= 2;
    return l;
}

// CTAs per SM the batched executor is compiled for: 128 registers at every width. A level's time is
// the latency of one warp's instructions; with 64 or 80 registers the local sweeps lose the overlap of
// their loads (500 graphs of up to 50,000 vertices on 256-thread CTAs: 3.2 ms with 128 registers, 4.2
// with 80; 10,000 of them on 128-thread CTAs: 13.7 ms with 4 CTAs on an SM, 15.0 with 5, 17.8 with 8).
template <int kThreads>
constexpr int batch_min_blocks() { return kThreads < 512 ? 512 / kThreads : 1; }

// CTA width when the caller names none. Wide CTAs finish a graph sooner, narrow ones order more
// vertices per SM: a batch takes about the larger of tail x (vertices of its largest graph) and
// rate x (all its vertices). Nanoseconds per vertex on GB300 (mixes of grids and meshes, log-uniform
// sizes); 10,000 graphs up to 50,000 vertices: 13.7 / 17.7 / 26.0 ms on 128 / 256 / 512 threads; 4,000:
// 10.0 / 7.1 / 10.4; 1,000: 7.9 / 4.8 / 3.4; 400 up to 200,000: 20.1 / 11.0 / 7.3.
static int batch_threads(long long n_total, int max_n) {
    static const struct { int threads; double tail, rate; } kWidths[] = {
        {128, 160.0, 0.17}, {256, 95.0, 0.22}, {512, 57.0, 0.32}};
    int best = 256;
    double least = 1e300;
    for (const auto& w : kWidths) {
        const double t = std::max(w.tail * max_n, w.rate * (double)n_total);
        if (t < least) {
            least = t;
            best = w.threads;
        }
    }
    return best;
}

template <int kThreads>
__global__ void __launch_bounds__(kThreads, batch_min_blocks<kThreads>()) k_rcm_batch(BatchArgs b) {
    // the local sweeps' state (rcm_local.cuh); component tables sort in the same bytes
    extern __shared__ __align__(16) unsigned s_local[];
    __shared__ EngineSmem smem;
    __shared__ int s_item;
    if (ld_volatile(&b.ctl->status) & kErrBadCsr) return;
    Engine<true> e;
    const int sort_cap = (int)(local_bytes(b.local_cap, b.local_slots, b.local_entries) / 12);
    if (threadIdx.x == 0) local_init(&smem.loc, b.local_cap, b.local_slots, b.local_entries, s_local);
    while (true) {
        if (threadIdx.x == 0) s_item = atomicAdd(&b.ctl->work_next, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= b.G) break;
        const int g = b.order ? b.order[item] : item;
        const int v0 = (int)b.goff[g];
        const int n = (int)(b.goff[g + 1] - b.goff[g]);
        if (n == 0) continue;
        EngineArgs a;
        a.n = n;
        a.v0 = v0;
        a.rowptr = b.rowptr;
        a.ell = b.ell;
        a.adj = b.adj;
        a.deg = b.deg;
        a.claim = b.claim;
        a.vis = b.vis;
        a.qa = b.qa + v0;
        a.qb = b.qb + v0;
        a.boff = b.boff + v0;
        a.perm = b.perm + v0;
        a.ctl = b.ctl;
        a.status = &b.ctl->status;
        a.diag = nullptr;
        a.narrow_thr = 0x7fffffff;
        a.obits = claim_order_bits(n);
        a.profile = 0;
        a.cc_parent = b.cc_parent;
        a.cc_size = b.cc_size;
        a.cc_key = b.cc_key;
        a.cc_roots = b.cc_roots + v0;
        a.cc_gkey = b.cc_gkey + 2 * (size_t)v0;
        a.cc_gidx = b.cc_gidx + 2 * (size_t)v0;
        a.cc_tab = b.cc_tab + v0;
        a.cc_cap = n;
        a.cc_big = 0;
        a.fused = 1;
        a.hubs = 0;
        a.probe = 0;
        a.hub_auto = 0;
        a.cc_first = 0;
        a.limit_ns = 0;
        a.fkey = nullptr;  // CTA engines: top-down, level by level
        a.expand_mode = 1;
        a.bu_divisor = 16;
        a.adist = nullptr;
        a.aq = nullptr;
        a.actl = nullptr;
        a.aq_cap = 0;
        a.mid_k = 0;  // CTA engines: no middle tier
        a.mid_thr = 0;
        a.local_hi = a.local_slots = a.local_entries = 0;  // (the grid executor's)
        a.gvis = nullptr;
        __syncthreads();
        e.init(a, &smem);
        e.sm_sort = (unsigned long long*)s_local;
        e.sm_sort_cap = sort_cap;
        if (!e.run()) return;
        __syncthreads();
        // the segment holds global ids while running; the result is in local ids
        for (int i = threadIdx.x; i < n; i += kThreads) a.perm[i] -= v0;
        __syncthreads();
    }
}

BatchLayout batch_layout(long long n_total, long long nnz, long long G) {
    const size_t N = (size_t)std::max<long long>(n_total, 1), E = (size_t)std::max<long long>(nnz, 1);
    BatchLayout L;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = align_up(o + bytes, 256);
        return at;
    };
    L.ctl = take(sizeof(Ctl));
    L.pool = take(sizeof(int) * 4 * N);
    L.deg = take(sizeof(int) * N);
    L.claim = take(sizeof(unsigned long long) * N);
    L.vis = take(sizeof(int) * N);
    L.big = take(sizeof(int) * N);
    L.adj = take(sizeof(int) * E);
    L.ell = take(sizeof(int4) * 2 * N);
    L.ccs = take(sizeof(int) * N);
    L.cck = take(sizeof(unsigned long long) * N);
    L.ccr = take(sizeof(int) * N);
    L.ccgk = take(sizeof(unsigned long long) * 2 * N);
    L.ccgi = take(sizeof(int) * 2 * N);
    L.cct = take(sizeof(int4) * N);
    L.order = take(sizeof(int) * (size_t)std::max<long long>(G, 1));
    L.total = o;
    return L;
}

std::vector<int> batch_order(const std::vector<long long>& goff) {
    const int G = (int)goff.size() - 1;
    std::vector<int> order(std::max(G, 0));
    for (int i = 0; i < G; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(),
                     [&](int x, int y) { return goff[x + 1] - goff[x] > goff[y + 1] - goff[y]; });
    return order;
}

// Vertices of the largest graph.
static int batch_max(const std::vector<long long>& goff) {
    long long m = 0;
    for (size_t i = 0; i + 1 < goff.size(); ++i) m = std::max(m, goff[i + 1] - goff[i]);
    return (int)std::min<long long>(std::max<long long>(m, 0), kIntMax);
}

static std::mutex g_batch_mu;
static int g_batch_per_sm[3] = {-1, -1, -1};  // CTAs per SM of the 128-, 256- and 512-thread executor

static int batch_index(int threads) { return threads == 128 ? 0 : threads == 256 ? 1 : threads == 512 ? 2 : -1; }

static const void* batch_kernel(int threads) {
    switch (threads) {
        case 128: return (const void*)k_rcm_batch<128>;
        case 512: return (const void*)k_rcm_batch<512>;
    }
    return (const void*)k_rcm_batch<256>;
}

static int batch_blocks_per_sm(int threads) {
    const int idx = batch_index(threads);
    if (idx < 0) return 0;
    std::lock_guard<std::mutex> g(g_batch_mu);
    if (g_batch_per_sm[idx] < 0) {
        int bps = 0;
        const void* k = batch_kernel(threads);
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerSm - kBatchStaticSmem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k, threads, local_bytes(0, kBatchMinSlots, kBatchEntries));
        g_batch_per_sm[idx] = bps;
        cudaFuncSetAttribute(k_sort_rows_big, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(unsigned long long) * kBigRowSmem));
    }
    return g_batch_per_sm[idx];
}

rcm_status batch_tuning(const rcm_batch_options* o, BatchTuning* out) {
    BatchTuning t;
    t.threads = 0;
    if (o) {
        if (o->block_threads) t.threads = o->block_threads;
        if (o->row_sort_split) t.small_max = o->row_sort_split;
        if (o->row_order != 0 && o->row_order != 1) return RCM_ERR_INVALID_ARG;
        t.by_degree = o->row_order ? 0 : 1;
    }
    if ((t.threads && batch_index(t.threads) < 0) || t.small_max < 4 || t.small_max > kSmallRowMax) return RCM_ERR_INVALID_ARG;
    *out = t;
    return RCM_OK;
}

bool batch_prepare(const BatchTuning& t) {
    device_info();
    return batch_blocks_per_sm(t.threads) > 0;
}

cudaError_t enqueue_batch(int G, long long n_total, int nnz, const long long* goff, const int* order,
                          const int* rowptr, const int* colidx, int* perm, char* base, const BatchLayout& L,
                          const BatchTuning& t, cudaStream_t s, int max_n) {
    const DeviceInfo& di = device_info();
    const int per_sm = batch_blocks_per_sm(t.threads);
    if (per_sm <= 0) return cudaErrorInvalidConfiguration;
    const long long N = std::max<long long>(n_total, 1);
    Ctl* ctl = (Ctl*)(base + L.ctl);
    int* pool4 = (int*)(base + L.pool);
    int* deg = (int*)(base + L.deg);
    unsigned char* deg8 = deg8_at(pool4, N);
    unsigned long long* claim = (unsigned long long*)(base + L.claim);
    int* vis = (int*)(base + L.vis);
    int* big = (int*)(base + L.big);
    int* adj = (int*)(base + L.adj);
    int4* ell = (int4*)(base + L.ell);
    cudaError_t e = cudaMemsetAsync(ctl, 0, sizeof(Ctl), s);
    if (e != cudaSuccess) return e;
    const int pb = 256;
    const int pgrid = (int)std::max<long long>(1, std::min<long long>((n_total + pb - 1) / pb, (long long)di.sms * 16));
    // rows longer than small_max entries number at most nnz / (small_max + 1)
    const int big_grid = (int)std::max<long long>(1, std::min<long long>(3LL * di.sms, nnz / (t.small_max + 1)));
    // one pass over the entries checks the structure and each graph's block (G > 1) and counts degrees
    k_degree_validate<<<pgrid, pb, 0, s>>>((int)n_total, nnz, rowptr, colidx, deg, deg8, claim, vis, big, ctl, t.small_max,
                                           nullptr, nullptr, G > 1 ? goff : nullptr, G);
    k_sort_rows_small<<<pgrid, pb, 0, s>>>((int)n_total, rowptr, colidx, deg, deg8, adj, ell, ctl, t.small_max,
                                           t.by_degree);
    k_sort_rows_big<<<big_grid, kBigRowThreads, sizeof(unsigned long long) * kBigRowSmem, s>>>(
        (int)n_total, rowptr, colidx, deg, adj, ell, big, ctl, (unsigned long long*)pool4, t.by_degree);
    BatchArgs b;
    b.G = G;
    b.goff = goff;
    b.order = order;
    b.rowptr = rowptr;
    b.ell = ell;
    b.adj = adj;
    b.deg = deg;
    b.claim = claim;
    b.vis = vis;
    b.qa = pool4;
    b.qb = pool4 + N;
    b.boff = pool4 + 2 * N;
    b.perm = perm;
    b.ctl = ctl;
    b.cc_parent = pool4 + 3 * N;
    b.cc_size = (int*)(base + L.ccs);
    b.cc_key = (unsigned long long*)(base + L.cck);
    b.cc_roots = (int*)(base + L.ccr);
    b.cc_gkey = (unsigned long long*)(base + L.ccgk);
    b.cc_gidx = (int*)(base + L.ccgi);
    b.cc_tab = (int4*)(base + L.cct);
    const LocalShape shape = local_shape(max_n, G, per_sm, di.sms);
    b.local_cap = shape.cap;
    b.local_slots = shape.slots;
    b.local_entries = kBatchEntries;
    const size_t smem = local_bytes(b.local_cap, b.local_slots, b.local_entries);
    // at most as many CTAs as the local state leaves room for (more would only wait)
    const long long fit = std::max<long long>(1, std::min<long long>(per_sm, kSmemPerSm / (long long)(smem + kBatchStaticSmem + 1024)));
    const int blocks = (int)std::min<long long>(fit * di.sms, std::max(G, 1));
    void* kargs[] = {&b};
    return cudaLaunchKernel(batch_kernel(t.threads), dim3(blocks), dim3(t.threads), kargs, smem, s);
}

rcm_status order_batch(int32_t G, int64_t n_total, const int64_t* goff, const int32_t* rowptr,
                       const int32_t* colidx, int32_t* perm, const rcm_batch_options* opts, cudaStream_t s) {
    BatchTuning t;
    rcm_status st = batch_tuning(opts, &t);
    if (st != RCM_OK) return st;
    // nnz sizes the sorted-adjacency copy and the graph sizes set the work-queue order: one
    // synchronised read of rowptr[n_total] and goff
    int nnz = 0;
    std::vector<long long> goff_h((size_t)G + 1);
    cudaError_t e = cudaMemcpyAsync(&nnz, rowptr + n_total, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(goff_h.data(), goff, sizeof(long long) * goff_h.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_status(e);
    if (nnz < 0) return RCM_ERR_BAD_CSR;
    const int max_n = batch_max(goff_h);
    if (t.threads == 0) t.threads = batch_threads(n_total, max_n);
    if (!batch_prepare(t)) return RCM_ERR_CUDA;
    const BatchLayout L = batch_layout(n_total, nnz, G);
    int* latch = stream_latch(s);
    if (!latch) return RCM_ERR_TOO_LARGE;  // every latch slot held by streams whose status is unread
    void* ws = nullptr;
    st = ws_alloc(&ws, L.total, s);
    if (st != RCM_OK) return st;
    char* base = (char*)ws;
    // pageable source: the copy returns once the data is staged, so the vector may go
    const std::vector<int> order = batch_order(goff_h);
    e = cudaMemcpyAsync(base + L.order, order.data(), sizeof(int) * (size_t)G, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = enqueue_batch(G, n_total, nnz, (const long long*)goff, (const int*)(base + L.order), rowptr, colidx,
                          perm, base, L, t, s, max_n);
    if (e == cudaSuccess) e = enqueue_latch((Ctl*)(base + L.ctl), latch, nullptr, s);
    ws_free(ws, s);
    return e == cudaSuccess ? RCM_OK : cuda_status(e);
}

// Replay plan: the batched launches for fixed buffers, captured once into a CUDA graph.
struct BatchPlan {
    void* ws = nullptr;
    Ctl* ctl = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

rcm_status batch_plan_create(int32_t G, int64_t n_total, int64_t nnz, const int64_t* goff, const int32_t* rowptr,
                             const int32_t* colidx, int32_t* perm, const rcm_batch_options* opts, BatchPlan** out) {
    BatchTuning t;
    rcm_status st = batch_tuning(opts, &t);
    if (st != RCM_OK) return st;
    BatchPlan* p = new (std::nothrow) BatchPlan();
    if (!p) return RCM_ERR_OOM;
    const BatchLayout L = batch_layout(n_total, nnz, G);
    cudaError_t e = cudaMalloc(&p->ws, L.total);
    // work-queue order (largest graph first) from the graph offsets at creation
    std::vector<long long> goff_h((size_t)G + 1);
    if (e == cudaSuccess) e = cudaMemcpy(goff_h.data(), goff, sizeof(long long) * goff_h.size(), cudaMemcpyDeviceToHost);
    const int max_n = batch_max(goff_h);
    if (t.threads == 0) t.threads = batch_threads(n_total, max_n);
    if (e == cudaSuccess && !batch_prepare(t)) e = cudaErrorInvalidConfiguration;
    if (e == cudaSuccess) {
        const std::vector<int> order = batch_order(goff_h);
        e = cudaMemcpy((char*)p->ws + L.order, order.data(), sizeof(int) * (size_t)G, cudaMemcpyHostToDevice);
    }
    cudaStream_t cs = nullptr;
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        const cudaError_t ee = enqueue_batch(G, n_total, (int)nnz, (const long long*)goff,
                                             (const int*)((char*)p->ws + L.order), rowptr, colidx, perm,
                                             (char*)p->ws, L, t, cs, max_n);
        e = cudaStreamEndCapture(cs, &p->graph);
        if (e == cudaSuccess) e = ee;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&p->exec, p->graph, 0);
    if (cs) cudaStreamDestroy(cs);
    if (e != cudaSuccess) {
        if (p->exec) cudaGraphExecDestroy(p->exec);
        if (p->graph) cudaGraphDestroy(p->graph);
        if (p->ws) cudaFree(p->ws);
        delete p;
        return cuda_status(e);
    }
    p->ctl = (Ctl*)((char*)p->ws + L.ctl);
    *out = p;
    return RCM_OK;
}

rcm_status batch_plan_launch(BatchPlan* p, cudaStream_t s) {
    const cudaError_t e = cudaGraphLaunch(p->exec, s);
    return e == cudaSuccess ? RCM_OK : cuda_status(e);
}

rcm_status batch_plan_status(BatchPlan* p, cudaStream_t s) {
    int bits = 0;
    cudaError_t e = cudaMemcpyAsync(&bits, &p->ctl->status, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_status(e);
    return status_from_bits(bits);
}

void batch_plan_destroy(BatchPlan* p) {
    cudaDeviceSynchronize();
    if (p->exec) cudaGraphExecDestroy(p->exec);
    if (p->graph) cudaGraphDestroy(p->graph);
    if (p->ws) cudaFree(p->ws);
    delete p;
}

}  // namespace rcm

struct rcm_batch_plan {
    rcm::BatchPlan* p;
};

extern "C" {

rcm_status rcm_batch_plan_create(int32_t G, int64_t n_total, int64_t nnz, const int64_t* goff,
                                 const int32_t* rowptr, const int32_t* colidx, int32_t* perm_out,
                                 const rcm_batch_options* opts, rcm_batch_plan** out) {
    if (!out || G <= 0 || n_total <= 0 || n_total >= 0x7fffffffLL || nnz < 0 || nnz >= 0x7fffffffLL)
        return RCM_ERR_INVALID_ARG;
    if (!goff || !rowptr || !perm_out || (nnz > 0 && !colidx)) return RCM_ERR_INVALID_ARG;
    *out = nullptr;
    rcm::BatchPlan* p = nullptr;
    const rcm_status st = rcm::batch_plan_create(G, n_total, nnz, goff, rowptr, colidx, perm_out, opts, &p);
    if (st != RCM_OK) return st;
    *out = new (std::nothrow) rcm_batch_plan{p};
    if (!*out) {
        rcm::batch_plan_destroy(p);
        return RCM_ERR_OOM;
    }
    return RCM_OK;
}

rcm_status rcm_batch_plan_launch(rcm_batch_plan* plan, rcm_stream_t stream) {
    if (!plan) return RCM_ERR_INVALID_ARG;
    return rcm::batch_plan_launch(plan->p, (cudaStream_t)stream);
}

rcm_status rcm_batch_plan_status(rcm_batch_plan* plan, rcm_stream_t stream) {
    if (!plan) return RCM_ERR_INVALID_ARG;
    return rcm::batch_plan_status(plan->p, (cudaStream_t)stream);
}

rcm_status rcm_batch_plan_destroy(rcm_batch_plan* plan) {
    if (!plan) return RCM_ERR_INVALID_ARG;
    rcm::batch_plan_destroy(plan->p);
    delete plan;
    return RCM_OK;
}

}  // extern "C"
