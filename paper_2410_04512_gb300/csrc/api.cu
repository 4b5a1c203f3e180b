// api.cu -- context, errors, device buffers, scans and kernel timing.
#include "sgp_internal.cuh"

#include <cuda.h>

#include <atomic>
#include <cstdlib>

sgp_status sgp_fail(sgp_ctx *ctx, sgp_status code, const char *fmt, ...)
{
    if (ctx) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof(buf), fmt, ap);
        va_end(ap);
        ctx->err = buf;
    }
    return code;
}

sgp_status buf_ensure(sgp_ctx *ctx, DBuf &b, size_t bytes)
{
    if (bytes == 0) bytes = 16;
    if (b.p && b.bytes >= bytes) return SGP_OK;
    if (b.p) {
        cudaFreeAsync(b.p, ctx->stream);
        b.p = nullptr;
        b.bytes = 0;
    }
    size_t want = (bytes + 255) & ~size_t(255);
    cudaError_t e = cudaMallocAsync(&b.p, want, ctx->stream);
    if (e != cudaSuccess) {
        b.p = nullptr;
        cudaGetLastError();
        return sgp_fail(ctx, SGP_ERR_OOM, "device allocation of %zu bytes failed: %s", want,
                        cudaGetErrorString(e));
    }
    b.bytes = want;
    return SGP_OK;
}

void buf_release(DBuf &b, cudaStream_t s)
{
    if (b.p) cudaFreeAsync(b.p, s);
    b.p = nullptr;
    b.bytes = 0;
}

sgp_status scratch_ensure(sgp_ctx *ctx, size_t bytes)
{
    if (ctx->d_scratch && ctx->d_scratch_bytes >= bytes) return SGP_OK;
    if (ctx->d_scratch) cudaFreeAsync(ctx->d_scratch, ctx->stream);
    ctx->d_scratch = nullptr;
    size_t want = (bytes + 4095) & ~size_t(4095);
    cudaError_t e = cudaMallocAsync(&ctx->d_scratch, want, ctx->stream);
    if (e != cudaSuccess) {
        ctx->d_scratch = nullptr;
        ctx->d_scratch_bytes = 0;
        cudaGetLastError();
        return sgp_fail(ctx, SGP_ERR_OOM, "scratch allocation of %zu bytes failed", want);
    }
    SGP_CUDA(ctx, cudaMemsetAsync(ctx->d_scratch, 0, want, ctx->stream));
    ctx->d_scratch_bytes = want;
    return SGP_OK;
}

// the pinned page of a context
constexpr size_t PINNED = 4096;

sgp_status read_back(sgp_ctx *ctx, void *host, const void *dev, size_t bytes)
{
    void *stage = ctx->h_stage;
    if (bytes > ctx->h_stage_bytes) {
        if (bytes > ctx->h_large_bytes) {
            if (ctx->h_large) cudaFreeHost(ctx->h_large);
            ctx->h_large = nullptr;
            ctx->h_large_bytes = 0;
            SGP_CUDA(ctx, cudaMallocHost(&ctx->h_large, bytes));
            ctx->h_large_bytes = bytes;
        }
        stage = ctx->h_large;
    }
    SGP_CUDA(ctx, cudaMemcpyAsync(stage, dev, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    SGP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    memcpy(host, stage, bytes);
    SGP_TRY(kt_collect(ctx));
    return SGP_OK;
}

// ---------------------------------------------------------------------------
// Exclusive scan of int32, out[0..n] with out[n] the total; in may be out.
// Short arrays in one thread block; longer ones in two launches: the sums of
// up to SCAN_BLOCKS chunks, then every block adds up the sums before its own
// chunk (a few per thread) and scans that.  A build runs some fifty scans, most
// of them short, so the launches count: a copy of the last input, the tiles,
// their totals, the addition and out[n] were five.  1e5 cells, factor: 2.10 -> 1.88 ms; 1e6: 4.38 -> 3.73.
// ---------------------------------------------------------------------------
constexpr int SCAN_ITEMS = 4, SCAN_TILE = SGP_BLOCK * SCAN_ITEMS, SCAN_BLOCKS = 1024, SCAN_ONE = 1024;

// exclusive scan of one value per thread of a block of BS; *total the sum
template <int BS>
__device__ __forceinline__ int32_t block_excl_scan(int32_t v, int32_t *sh, int32_t *total)
{
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (l >= o) x += y;
    }
    if (l == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        int32_t t = l < BS / 32 ? sh[l] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (l >= o) t += y;
        }
        if (l < BS / 32) sh[l] = t;
    }
    __syncthreads();
    const int32_t before = (w > 0 ? sh[w - 1] : 0) + x - v;
    *total = sh[BS / 32 - 1];
    __syncthreads();
    return before;
}

// [i0, i1) of the array from the running total `carry`; returns the new total
template <int BS>
__device__ __forceinline__ int32_t scan_range(const int32_t *in, int32_t *out, int64_t i0, int64_t i1, int32_t carry,
                                              int32_t *sh)
{
    for (int64_t t = i0; t < i1; t += BS * SCAN_ITEMS) {
        const int64_t base = t + (int64_t)threadIdx.x * SCAN_ITEMS;
        int32_t v[SCAN_ITEMS], s = 0, tot;
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) {
            v[k] = base + k < i1 ? in[base + k] : 0;
            s += v[k];
        }
        int32_t run = carry + block_excl_scan<BS>(s, sh, &tot);
#pragma unroll
        for (int k = 0; k < SCAN_ITEMS; ++k) {
            if (base + k < i1) out[base + k] = run;
            run += v[k];
        }
        carry += tot;
    }
    return carry;
}

__global__ void __launch_bounds__(SCAN_ONE) k_scan_one(const int32_t *in, int32_t *out, int64_t n)
{
    __shared__ int32_t sh[32];
    const int32_t total = scan_range<SCAN_ONE>(in, out, 0, n, 0, sh);
    if (threadIdx.x == 0) out[n] = total;
}
__global__ void __launch_bounds__(SGP_BLOCK) k_scan_sums(const int32_t *in, int64_t n, int64_t chunk, int32_t *sums)
{
    __shared__ int32_t sh[32];
    const int64_t i0 = blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    int32_t s = 0, total;
#pragma unroll 4
    for (int64_t i = i0 + threadIdx.x; i < i1; i += SGP_BLOCK) s += in[i];
    block_excl_scan<SGP_BLOCK>(s, sh, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}
__global__ void __launch_bounds__(SGP_BLOCK) k_scan_out(const int32_t *in, int32_t *out, int64_t n, int64_t chunk,
                                                        const int32_t *__restrict__ sums)
{
    __shared__ int32_t sh[32];
    int32_t s = 0, before;
#pragma unroll
    for (int k = 0; k < SCAN_BLOCKS / SGP_BLOCK; ++k) {
        const unsigned b = threadIdx.x + k * SGP_BLOCK;
        s += b < blockIdx.x ? sums[b] : 0;
    }
    block_excl_scan<SGP_BLOCK>(s, sh, &before);
    const int64_t i0 = blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    const int32_t total = scan_range<SGP_BLOCK>(in, out, i0, i1, before, sh);
    if (threadIdx.x == 0 && i1 == n) out[n] = total;
}

sgp_status scan_exclusive_i32(sgp_ctx *ctx, const int32_t *in, int32_t *out, int64_t n)
{
    if (n <= 0) {
        SGP_CUDA(ctx, cudaMemsetAsync(out, 0, sizeof(int32_t), ctx->stream));
        return SGP_OK;
    }
    // one block up to two of its tiles
    if (n <= 2 * SCAN_ONE * SCAN_ITEMS) {
        LAUNCH(ctx, k_scan_one, 1, SCAN_ONE, 0, in, out, n);
        return SGP_OK;
    }
    const int64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE, per = (tiles + SCAN_BLOCKS - 1) / SCAN_BLOCKS,
                  chunk = per * SCAN_TILE;
    const unsigned blocks = (unsigned)((n + chunk - 1) / chunk);
    if (!ctx->d_scan) SGP_CUDA(ctx, cudaMallocAsync(&ctx->d_scan, sizeof(int32_t) * SCAN_BLOCKS, ctx->stream));
    int32_t *sums = reinterpret_cast<int32_t *>(ctx->d_scan);
    LAUNCH(ctx, k_scan_sums, blocks, SGP_BLOCK, 0, in, n, chunk, sums);
    LAUNCH(ctx, k_scan_out, blocks, SGP_BLOCK, 0, in, out, n, chunk, (const int32_t *)sums);
    return SGP_OK;
}

// ---------------------------------------------------------------------------
// kernel timing
// ---------------------------------------------------------------------------
static cudaEvent_t ev_get(sgp_ctx *ctx)
{
    if (!ctx->ev_free.empty()) {
        cudaEvent_t e = ctx->ev_free.back();
        ctx->ev_free.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}

sgp_status kt_begin(sgp_ctx *ctx, int kclass, cudaEvent_t *ev)
{
    *ev = nullptr;
    if (!ctx->timing) return SGP_OK;
    if (ctx->capture_sink) {
        // inside a capture: an event-record node owned by the graph entry
        SGP_CUDA(ctx, cudaEventCreate(ev));
        SGP_CUDA(ctx, cudaEventRecordWithFlags(*ev, ctx->stream, cudaEventRecordExternal));
        return SGP_OK;
    }
    *ev = ev_get(ctx);
    SGP_CUDA(ctx, cudaEventRecord(*ev, ctx->stream));
    return SGP_OK;
}

sgp_status kt_end(sgp_ctx *ctx, int kclass, cudaEvent_t start)
{
    if (!ctx->timing || !start) return SGP_OK;
    if (ctx->capture_sink) {
        cudaEvent_t e = nullptr;
        SGP_CUDA(ctx, cudaEventCreate(&e));
        SGP_CUDA(ctx, cudaEventRecordWithFlags(e, ctx->stream, cudaEventRecordExternal));
        ctx->capture_sink->push_back(KtRec{kclass, start, e});
        return SGP_OK;
    }
    cudaEvent_t e = ev_get(ctx);
    SGP_CUDA(ctx, cudaEventRecord(e, ctx->stream));
    ctx->ev_pending[kclass].push_back(start);
    ctx->ev_pending[kclass].push_back(e);
    return SGP_OK;
}

// The SMs that a launch on the context's stream can have: the device's (an MPS
// client's share of them), or those of the green context the stream belongs to.
// The persistent solves wait for one another's blocks and take at most one per SM.
static bool stream_sms(sgp_ctx *ctx)
{
    if (cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess) return false;
    // the driver's functions, looked up once per process (0.1 ms)
    static const struct Green {
        decltype(&cuStreamGetGreenCtx) of = nullptr;
        decltype(&cuGreenCtxGetDevResource) resource = nullptr;
        Green()
        {
            void *f = nullptr, *g = nullptr;
            cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound, r = q;
            if (cudaGetDriverEntryPointByVersion("cuStreamGetGreenCtx", &f, CUDART_VERSION, cudaEnableDefault, &q) == cudaSuccess &&
                cudaGetDriverEntryPointByVersion("cuGreenCtxGetDevResource", &g, CUDART_VERSION, cudaEnableDefault, &r) == cudaSuccess &&
                q == cudaDriverEntryPointSuccess && r == cudaDriverEntryPointSuccess) {
                of = reinterpret_cast<decltype(of)>(f);
                resource = reinterpret_cast<decltype(resource)>(g);
            } else {
                cudaGetLastError();   // a driver without green contexts
            }
        }
    } green;
    CUgreenCtx g = nullptr;
    CUdevResource r{};
    if (green.of && green.of((CUstream)ctx->stream, &g) == CUDA_SUCCESS && g &&
        green.resource(g, &r, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS)
        ctx->num_sms = (int)r.sm.smCount;
    return ctx->num_sms > 0;
}

sgp_status resident_grid(sgp_ctx *ctx, const void *kernel, int block, int64_t want, unsigned *grid)
{
    int per_sm = 0;
    for (auto &kv : ctx->occupancy)
        if (kv.first == kernel) per_sm = kv.second;
    if (!per_sm) {
        SGP_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, 0));
        per_sm = std::max(per_sm, 1);
        ctx->occupancy.push_back({kernel, per_sm});
    }
    int64_t cap = (int64_t)ctx->num_sms * per_sm;
    *grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, cap));
    return SGP_OK;
}

// ---------------------------------------------------------------------------
// CUDA graph cache
// ---------------------------------------------------------------------------
uint64_t next_generation()
{
    static std::atomic<uint64_t> g{1};
    return g.fetch_add(1);
}

static void graph_free(GraphEntry *ge)
{
    if (ge->exec) cudaGraphExecDestroy(ge->exec);
    for (auto &r : ge->ev) {
        cudaEventDestroy(r.a);
        cudaEventDestroy(r.b);
    }
    delete ge;
}

void graph_release_all(sgp_ctx *ctx)
{
    for (GraphEntry *ge : ctx->graphs) graph_free(ge);
    ctx->graphs.clear();
}

sgp_status graph_lookup(sgp_ctx *ctx, const uint64_t *key, int nkey, GraphEntry **out)
{
    if (nkey > 32) return sgp_fail(ctx, SGP_ERR_INVALID_ARG, "graph key too long");
    ++ctx->graph_clock;
    for (GraphEntry *ge : ctx->graphs)
        if (ge->nkey == nkey && std::memcmp(ge->key, key, sizeof(uint64_t) * nkey) == 0) {
            ge->last_use = ctx->graph_clock;
            *out = ge;
            return SGP_OK;
        }
    const size_t max_entries = 6;
    if (ctx->graphs.size() >= max_entries) {
        auto lru = std::min_element(ctx->graphs.begin(), ctx->graphs.end(),
                                    [](GraphEntry *a, GraphEntry *b) { return a->last_use < b->last_use; });
        SGP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        graph_free(*lru);
        ctx->graphs.erase(lru);
    }
    GraphEntry *ge = new GraphEntry();
    std::memcpy(ge->key, key, sizeof(uint64_t) * nkey);
    ge->nkey = nkey;
    ge->last_use = ctx->graph_clock;
    ctx->graphs.push_back(ge);
    *out = ge;
    return SGP_OK;
}

sgp_status graph_begin(sgp_ctx *ctx, GraphEntry *ge, cudaStream_t *saved, int64_t *l0)
{
    if (!ctx->cap_stream) SGP_CUDA(ctx, cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking));
    *saved = ctx->stream;
    *l0 = ctx->launches;
    SGP_CUDA(ctx, cudaStreamBeginCapture(ctx->cap_stream, cudaStreamCaptureModeThreadLocal));
    ctx->stream = ctx->cap_stream;
    ctx->capture_sink = &ge->ev;
    return SGP_OK;
}

sgp_status graph_end(sgp_ctx *ctx, GraphEntry *ge, cudaStream_t saved, int64_t l0, sgp_status st)
{
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(ctx->cap_stream, &g);
    ctx->stream = saved;
    ctx->capture_sink = nullptr;
    ge->kernels = ctx->launches - l0;
    ctx->launches = l0;
    if (st != SGP_OK) {
        if (g) cudaGraphDestroy(g);
        return st;
    }
    if (e != cudaSuccess || !g)
        return sgp_fail(ctx, SGP_ERR_CUDA, "graph capture failed: %s", cudaGetErrorString(e));
    e = cudaGraphInstantiate(&ge->exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        ge->exec = nullptr;
        return sgp_fail(ctx, SGP_ERR_CUDA, "graph instantiation failed: %s", cudaGetErrorString(e));
    }
    return SGP_OK;
}

__global__ void k_while_cond(cudaGraphConditionalHandle h, const int *done, int *bodies, int max_bodies)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        const int b = *bodies + 1;
        *bodies = b;
        cudaGraphSetConditional(h, (*done == 0 && b < max_bodies) ? 1u : 0u);
    }
}

sgp_status graph_while_begin(sgp_ctx *ctx, GraphEntry *ge, cudaStream_t *saved, int64_t *l0, cudaGraph_t *g,
                             cudaGraphConditionalHandle *h)
{
    if (!ctx->cap_stream) SGP_CUDA(ctx, cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking));
    SGP_CUDA(ctx, cudaGraphCreate(g, 0));
    cudaError_t e = cudaGraphConditionalHandleCreate(h, *g, 1, cudaGraphCondAssignDefault);
    cudaGraphNodeParams cp{};
    cudaGraphNode_t node = nullptr;
    if (e == cudaSuccess) {
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = *h;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        e = cudaGraphAddNode(&node, *g, nullptr, nullptr, 0, &cp);
    }
    if (e == cudaSuccess)
        e = cudaStreamBeginCaptureToGraph(ctx->cap_stream, cp.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                          cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        cudaGraphDestroy(*g);
        *g = nullptr;
        return sgp_fail(ctx, SGP_ERR_CUDA, "conditional graph setup failed: %s", cudaGetErrorString(e));
    }
    *saved = ctx->stream;
    *l0 = ctx->launches;
    ctx->stream = ctx->cap_stream;
    ctx->capture_sink = nullptr;
    return SGP_OK;
}

sgp_status graph_while_end(sgp_ctx *ctx, GraphEntry *ge, cudaStream_t saved, int64_t l0, cudaGraph_t g,
                           cudaGraphConditionalHandle h, const int *done, int *bodies, int max_bodies,
                           sgp_status st)
{
    if (st == SGP_OK) {
        k_while_cond<<<1, 32, 0, ctx->cap_stream>>>(h, done, bodies, max_bodies);
        ctx->launches++;
    }
    cudaGraph_t body = nullptr;
    cudaError_t e = cudaStreamEndCapture(ctx->cap_stream, &body);
    if (e == cudaSuccess) e = cudaGetLastError();
    ctx->stream = saved;
    ge->kernels = ctx->launches - l0;
    ctx->launches = l0;
    if (st != SGP_OK || e != cudaSuccess) {
        cudaGraphDestroy(g);
        if (st != SGP_OK) return st;
        return sgp_fail(ctx, SGP_ERR_CUDA, "conditional graph capture failed: %s", cudaGetErrorString(e));
    }
    e = cudaGraphInstantiate(&ge->exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        ge->exec = nullptr;
        cudaGetLastError();
        return sgp_fail(ctx, SGP_ERR_CUDA, "conditional graph instantiation failed: %s", cudaGetErrorString(e));
    }
    return SGP_OK;
}

// After a replay has completed (the caller synchronised): add the replay's
// event-pair durations to the kernel-time totals.
sgp_status graph_collect_timing(sgp_ctx *ctx, GraphEntry *ge)
{
    if (!ctx->timing) return SGP_OK;
    for (auto &r : ge->ev) {
        float ms = 0.f;
        SGP_CUDA(ctx, cudaEventElapsedTime(&ms, r.a, r.b));
        ctx->kt_ms[r.cls] += ms;
        ctx->kt_n[r.cls] += 1;
    }
    return SGP_OK;
}

sgp_status kt_collect(sgp_ctx *ctx)
{
    for (int k = 0; k < SGP_KT_COUNT; ++k) {
        auto &v = ctx->ev_pending[k];
        for (size_t i = 0; i + 1 < v.size(); i += 2) {
            float ms = 0.f;
            SGP_CUDA(ctx, cudaEventElapsedTime(&ms, v[i], v[i + 1]));
            ctx->kt_ms[k] += ms;
            ctx->kt_n[k] += 1;
            ctx->ev_free.push_back(v[i]);
            ctx->ev_free.push_back(v[i + 1]);
        }
        v.clear();
    }
    return SGP_OK;
}

// ---------------------------------------------------------------------------
// C ABI: context
// ---------------------------------------------------------------------------
extern "C" {

const char *sgp_version(void) { return "sgp 0.1 sm_103a"; }

sgp_status sgp_create(sgp_ctx **out, int device, void *stream)
{
    if (!out) return SGP_ERR_INVALID_ARG;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
        cudaGetLastError();
        return SGP_ERR_INVALID_ARG;
    }
    if (cudaSetDevice(device) != cudaSuccess) return SGP_ERR_CUDA;
    sgp_ctx *ctx = new sgp_ctx();
    ctx->device = device;
    ctx->stream = reinterpret_cast<cudaStream_t>(stream);
    const char *ng = getenv("SGP_NO_GRAPHS");
    ctx->use_graphs = (ng && ng[0] == '1') ? 0 : 1;
    const char *lpr = getenv("SGP_SPMV_LPR");
    if (lpr) ctx->spmv_lpr = atoi(lpr);
    const char *nw = getenv("SGP_NO_WHILE");
    ctx->use_while = (nw && nw[0] == '1') ? 0 : 1;
    const char *np = getenv("SGP_NO_PDL");
    ctx->use_pdl = (np && np[0] == '1') ? 0 : 1;
    const char *tc = getenv("SGP_TAIL_CAP");
    if (tc) ctx->tail_cap = atoi(tc);
    const char *bc = getenv("SGP_BIN_CAP");
    if (bc) ctx->bin_cap = atoi(bc);
    const char *ns = getenv("SGP_NO_SMALL");
    if (ns && atoi(ns)) ctx->small_solve = 0;
    const char *nf = getenv("SGP_NO_FUSE");
    if (nf && atoi(nf)) ctx->fused = 0;
    const char *sk = getenv("SGP_SKEW_PACKETS");
    if (sk && atoi(sk)) ctx->skew = 1u << 20;
    if (scratch_ensure(ctx, 1 << 20) != SGP_OK || cudaMalloc(&ctx->d_flags, 4096) != cudaSuccess ||
        cudaMemset(ctx->d_flags, 0, 4096) != cudaSuccess ||
        cudaHostAlloc(&ctx->h_gave_up, PINNED, cudaHostAllocMapped) != cudaSuccess ||
        cudaHostGetDevicePointer(&ctx->d_gave_up, ctx->h_gave_up, 0) != cudaSuccess) {
        cudaGetLastError();
        if (ctx->d_scratch) cudaFree(ctx->d_scratch);
        if (ctx->d_flags) cudaFree(ctx->d_flags);
        if (ctx->h_gave_up) cudaFreeHost(ctx->h_gave_up);
        delete ctx;
        return SGP_ERR_OOM;
    }
    *ctx->h_gave_up = 0;
    ctx->h_stage = reinterpret_cast<char *>(ctx->h_gave_up) + 64;
    ctx->h_stage_bytes = PINNED - 64;
    if (noalloc_prepare(ctx) != SGP_OK || !stream_sms(ctx)) {
        cudaFree(ctx->d_scratch);
        cudaFree(ctx->d_flags);
        cudaFreeHost(ctx->h_gave_up);
        delete ctx;
        return SGP_ERR_CUDA;
    }
    *out = ctx;
    return SGP_OK;
}

void sgp_destroy(sgp_ctx *ctx)
{
    if (!ctx) return;
    cudaStreamSynchronize(ctx->stream);
    graph_release_all(ctx);
    if (ctx->cap_stream) cudaStreamDestroy(ctx->cap_stream);
    if (ctx->d_scratch) cudaFree(ctx->d_scratch);
    if (ctx->d_flags) cudaFree(ctx->d_flags);
    if (ctx->d_scan) cudaFree(ctx->d_scan);
    if (ctx->h_large) cudaFreeHost(ctx->h_large);
    if (ctx->h_gave_up) cudaFreeHost(ctx->h_gave_up);
    for (auto e : ctx->ev_free) cudaEventDestroy(e);
    for (int k = 0; k < SGP_KT_COUNT; ++k)
        for (auto e : ctx->ev_pending[k]) cudaEventDestroy(e);
    grid_release(ctx->grid_plain);
    grid_rows_release(ctx->grid_rows);
    if (ctx->grid_apply.p) cudaFree(ctx->grid_apply.p);
    delete ctx;
}

const char *sgp_last_error(const sgp_ctx *ctx) { return ctx ? ctx->err.c_str() : "no context"; }

sgp_status sgp_copy(sgp_ctx *ctx, void *dst, const void *src, int64_t bytes)
{
    if (!ctx || bytes < 0 || (bytes > 0 && (!dst || !src))) return SGP_ERR_INVALID_ARG;
    if (bytes == 0) return SGP_OK;
    SGP_CUDA(ctx, cudaMemcpyAsync(dst, src, (size_t)bytes, cudaMemcpyDeviceToDevice, ctx->stream));
    return SGP_OK;
}

sgp_status sgp_set_kernel_timing(sgp_ctx *ctx, int32_t enable)
{
    if (!ctx) return SGP_ERR_INVALID_ARG;
    ctx->timing = enable ? 1 : 0;
    return SGP_OK;
}

sgp_status sgp_kernel_time(sgp_ctx *ctx, int32_t kclass, double *total_ms, int64_t *launches,
                           int32_t reset)
{
    if (!ctx || kclass < 0 || kclass >= SGP_KT_COUNT) return SGP_ERR_INVALID_ARG;
    SGP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    SGP_TRY(kt_collect(ctx));
    if (total_ms) *total_ms = ctx->kt_ms[kclass];
    if (launches) *launches = ctx->kt_n[kclass];
    if (reset) {
        ctx->kt_ms[kclass] = 0;
        ctx->kt_n[kclass] = 0;
    }
    return SGP_OK;
}

sgp_status sgp_launch_count(sgp_ctx *ctx, int64_t *count, int32_t reset)
{
    if (!ctx) return SGP_ERR_INVALID_ARG;
    if (count) *count = ctx->launches;
    if (reset) ctx->launches = 0;
    return SGP_OK;
}

}  // extern "C"
