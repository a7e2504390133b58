// Context, store and tuple-set management behind the C ABI (include/tid.h).
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <atomic>
#include <new>

#include "lookback.cuh"
#include "ops.cuh"

namespace tid {

// ---------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------
static thread_local std::string g_err;

int fail(int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

int fail_cuda(cudaError_t e, const char *what) {
    cudaGetLastError();  // clear a non-sticky error so later calls can proceed
    if (e == cudaErrorMemoryAllocation) return fail(TID_ERR_OOM, "%s: out of device memory", what);
    return fail(TID_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

void clear_error() { g_err.clear(); }

// One GPU per process: launch shapes and shared-memory opt-ins are worked out
// once per process, on the device of its first context (or no-alloc scan).
static std::atomic<int> g_device{-1};

int sm_count() {
    static std::atomic<int> cached[64];  // zero: not yet queried
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) dev = 0;
    int v = dev < 64 ? cached[dev].load(std::memory_order_relaxed) : 0;
    if (v <= 0) {
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 1;
        if (dev < 64) cached[dev].store(v, std::memory_order_relaxed);
    }
    return v;
}

int claim_device(int device) {
    int first = -1;
    if (g_device.compare_exchange_strong(first, device) || first == device) return TID_OK;
    return fail(TID_ERR_ARG, "device %d: this process already runs on device %d (one GPU per process)", device,
                first);
}

int launch_check(const char *what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail_cuda(e, what);
    return TID_OK;
}

DeviceGuard::DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
}
DeviceGuard::~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
}

// ---------------------------------------------------------------------------
// memory
// ---------------------------------------------------------------------------
// Gives the held blocks back to the pool; false if there are none.
static bool drop_blocks(tid_ctx *ctx, bool all = false) {
    return ctx->blocks.drop([&](void *p) { cudaFreeAsync(p, ctx->stream); }, all);
}

// Asked once per call of the library (a capture begins and ends between calls): asked
// at every allocation and free it took eight plans on a small store 50 us of 2200.
void note_capture(tid_ctx *ctx) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool none = cudaStreamIsCapturing(ctx->stream, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone;
    ctx->in_graph.store(!none, std::memory_order_relaxed);
}

int dev_alloc(tid_ctx *ctx, void **p, size_t bytes) {
    *p = nullptr;
    const int64_t fa = ctx->fail_after.load(std::memory_order_relaxed);
    if (fa >= 0 && ctx->allocs.fetch_add(1, std::memory_order_relaxed) >= fa)
        return fail(TID_ERR_OOM, "device allocation refused (injected failure)");
    if (bytes == 0) bytes = 256;
    const bool in_graph = capturing(ctx);  // then the allocation is the graph's
    int cls = BlockCache::LARGE;
    if (bytes <= BlockCache::MAX_BLOCK && !in_graph) {
        cls = BlockCache::class_of(bytes);
        bytes = BlockCache::class_bytes(cls);
        if ((*p = ctx->blocks.take(cls))) return TID_OK;
    }
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, ctx->pool, ctx->stream);
    if (e == cudaErrorMemoryAllocation && drop_blocks(ctx)) {
        cudaGetLastError();
        e = cudaMallocFromPoolAsync(p, bytes, ctx->pool, ctx->stream);
    }
    if (e != cudaSuccess) {
        *p = nullptr;
        return fail_cuda(e, "device allocation");
    }
    if (!in_graph) ctx->blocks.add(*p, cls);
    return TID_OK;
}

void dev_free(tid_ctx *ctx, void *p) {
    if (!p) return;
    switch (ctx->blocks.put(p, capturing(ctx))) {
        case BlockCache::KEPT: break;
        case BlockCache::POOL: cudaFreeAsync(p, ctx->stream); break;
        case BlockCache::TWICE: ctx->freed_twice.store(true); break;
    }
}

// What a context keeps on the device between calls, neutral between launches: the
// finished-CTA counter of the row selections, the bounds of an extraction, the
// look-back's ticket and first status words.  One block, made with the context: an
// allocation made while a graph is captured is the graph's, unmapped until the
// graph runs, so it must not stay behind in the context.  (Called again by the
// first call that needs it only if the context itself was created under capture.)
int keep_scratch(tid_ctx *ctx) {
    std::lock_guard<std::mutex> lk(ctx->mu);
    if (ctx->kept) return TID_OK;
    constexpr size_t LB_FIRST = 1024;
    const size_t bytes = 3 * 256 + LB_FIRST * sizeof(unsigned long long);
    void *p = nullptr;
    TID_TRY(dev_alloc(ctx, &p, bytes));
    cudaError_t e = cudaMemsetAsync(p, 0, bytes, ctx->stream);
    if (e == cudaSuccess) {
        ctx->bounds_dev = (uint32_t *)((char *)p + 256);
        e = reset_bounds(ctx);
    }
    if (e != cudaSuccess) {
        ctx->bounds_dev = nullptr;
        dev_free(ctx, p);
        return fail_cuda(e, "context scratch");
    }
    ctx->sel_done = (unsigned *)p;
    ctx->lb_ticket = (unsigned *)((char *)p + 512);
    ctx->lb_status = (unsigned long long *)((char *)p + 768);
    ctx->lb_cap = LB_FIRST;
    ctx->kept = p;
    return TID_OK;
}

// The context's look-back scratch, grown on demand to >= `words` status words
// (new words are zeroed, i.e. "not ready" for every epoch) plus a ticket
// counter that is 0 between launches.  An array that a larger one replaces stays
// until the context goes: launches recorded in a graph have its address.  Under
// capture a larger array is the graph's, for this launch alone.
int ctx_scratch(tid_ctx *ctx, size_t words, LbScratch *sc) {
    const bool grows = words > ctx->lb_cap, in_graph = (grows || !ctx->kept) && capturing(ctx);
    if (!ctx->kept && !in_graph) TID_TRY(keep_scratch(ctx));
    sc->err = ctx->err_dev;
    sc->epoch = &ctx->epoch;
    if (words > ctx->lb_cap) {
        size_t want = 1024;
        while (want < words) want *= 2;
        void *p = nullptr;
        TID_TRY(dev_alloc(ctx, &p, want * sizeof(unsigned long long) + 256));
        TID_TRY_CUDA(cudaMemsetAsync(p, 0, want * sizeof(unsigned long long) + 256, ctx->stream),
                     "clear look-back scratch");
        sc->status = (unsigned long long *)p;
        sc->ticket = (unsigned int *)((char *)p + want * sizeof(unsigned long long));
        sc->cap = want;
        if (in_graph) return TID_OK;
        ctx->lb_grown[ctx->n_grown++] = p;
        ctx->lb_status = sc->status;
        ctx->lb_ticket = sc->ticket;
        ctx->lb_cap = want;
        return TID_OK;
    }
    sc->status = ctx->lb_status;
    sc->cap = ctx->lb_cap;
    sc->ticket = ctx->lb_ticket;
    return TID_OK;
}

// Look-back state for one launch of `num_tiles` tiles: a fresh epoch, so the
// status words of earlier launches read as "not ready".
int make_lookback(const LbScratch &sc, unsigned int num_tiles, Lookback *lb) {
    if (num_tiles > sc.cap) return fail(TID_ERR_ARG, "look-back scratch holds %zu tiles, %u needed", sc.cap, num_tiles);
    unsigned e = (*sc.epoch + 1) & ((1u << 30) - 1);
    if (e == 0) e = 1;
    *sc.epoch = e;
    lb->status = sc.status;
    lb->ticket = sc.ticket;
    lb->epoch = e;
    lb->num_tiles = num_tiles;
    lb->err = sc.err;
    return TID_OK;
}

int lookback_scratch(tid_ctx *ctx, unsigned int num_tiles, Lookback *lb) {
    std::lock_guard<std::mutex> lk(ctx->lb_mu);
    LbScratch sc{};
    TID_TRY(ctx_scratch(ctx, num_tiles, &sc));
    return make_lookback(sc, num_tiles, lb);
}

// ---------------------------------------------------------------------------
// row-count and bounds slots (mapped pinned host memory)
// ---------------------------------------------------------------------------
static constexpr int SLAB_SLOTS = 4096;

static void recycle(tid_ctx *ctx, const PendingSlot &p) {
    if (ctx->free_events.size() < MAX_FREE_EVENTS) ctx->free_events.push_back(p.ev);
    else cudaEventDestroy(p.ev);
    ctx->free_slots.push_back({p.slot.slab, p.slot.index});
}

// While a graph is captured in the default (global) mode, by this thread or by
// another, a query of an event is refused and ends that capture; in relaxed mode, the
// calling thread's own affair, it is allowed for events recorded outside a capture.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// The producer is known to be done: any other answer of the query (not ready, refused,
// a failed context) leaves the slot to it.
static bool producer_done(cudaEvent_t ev) {
    if (cudaEventQuery(ev) == cudaSuccess) return true;
    cudaGetLastError();  // no failure of a later launch
    return false;
}

static void sweep_pending(tid_ctx *ctx) {
    RelaxedCapture mode;
    auto &pend = ctx->pending;
    size_t w = 0;
    for (size_t i = 0; i < pend.size(); ++i) {
        if (producer_done(pend[i].ev)) recycle(ctx, pend[i]);
        else pend[w++] = pend[i];
    }
    pend.resize(w);
}

// The oldest pending slots whose producers are done, a few at a time (a program
// that frees sets far ahead of the GPU has thousands pending).
static void sweep_oldest(tid_ctx *ctx) {
    RelaxedCapture mode;
    auto &pend = ctx->pending;
    for (int i = 0; i < 4 && !pend.empty(); ++i) {
        if (!producer_done(pend.front().ev)) break;
        recycle(ctx, pend.front());
        pend.pop_front();
    }
}

static int slot_acquire(tid_ctx *ctx, Slot *s) {
    std::lock_guard<std::mutex> lk(ctx->mu);
    if (ctx->free_events.empty()) sweep_oldest(ctx);
    if (ctx->free_slots.empty()) sweep_pending(ctx);
    if (ctx->free_slots.empty()) {
        void *h = nullptr;
        TID_TRY_CUDA(cudaHostAlloc(&h, SLAB_SLOTS * sizeof(SlotWords), cudaHostAllocMapped),
                     "pinned slot slab");
        void *d = nullptr;
        cudaError_t e = cudaHostGetDevicePointer(&d, h, 0);
        if (e != cudaSuccess) {
            cudaFreeHost(h);
            return fail_cuda(e, "mapped slot slab");
        }
        const int slab = (int)ctx->slabs_host.size();
        ctx->slabs_host.push_back((SlotWords *)h);
        ctx->slabs_dev.push_back((SlotWords *)d);
        for (int i = SLAB_SLOTS - 1; i >= 0; --i) ctx->free_slots.push_back({slab, i});
    }
    auto si = ctx->free_slots.back();
    ctx->free_slots.pop_back();
    s->slab = si.first;
    s->index = si.second;
    s->words = ctx->slabs_host[si.first] + si.second;
    s->dev = &ctx->slabs_dev[si.first][si.second].rows;
    *(volatile int64_t *)&s->words->rows = -1;
    return TID_OK;
}

// ---------------------------------------------------------------------------
// sets
// ---------------------------------------------------------------------------
static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

int set_alloc(tid_ctx *ctx, int k, const int8_t *vars, int64_t cap, tid_set **out) {
    *out = nullptr;
    if (k < 1 || k > TID_MAX_COLS) return fail(TID_ERR_ARG, "set with %d columns", k);
    if (cap < 0) cap = 0;
    tid_set *s = new (std::nothrow) tid_set();
    if (!s) return fail(TID_ERR_OOM, "host allocation");
    s->ctx = ctx;
    s->k = k;
    for (int c = 0; c < k; ++c) s->vars[c] = vars[c];
    s->cap = cap;
    s->in_graph = capturing(ctx);
    const size_t colb = align_up((size_t)cap * sizeof(int32_t), 256);
    const size_t bytes = colb * (size_t)k + 256;
    int rc = dev_alloc(ctx, &s->block, bytes);
    if (rc != TID_OK) {
        delete s;
        return rc;
    }
    for (int c = 0; c < k; ++c) s->col[c] = (int32_t *)((char *)s->block + colb * c);
    s->d_rows = (int64_t *)((char *)s->block + colb * k);
    rc = slot_acquire(ctx, &s->slot);
    if (rc == TID_OK) {
        cudaError_t e = cudaSuccess;
        {
            std::lock_guard<std::mutex> lk(ctx->mu);
            if (!ctx->free_events.empty()) {
                s->ready = ctx->free_events.back();
                ctx->free_events.pop_back();
            }
        }
        if (!s->ready) e = cudaEventCreateWithFlags(&s->ready, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            s->ready = nullptr;
            rc = fail_cuda(e, "event");
        }
    }
    if (rc != TID_OK) {
        set_free(s);
        return rc;
    }
    *out = s;
    return TID_OK;
}

int set_view(tid_ctx *ctx, SharedBlock *sb, int32_t *col, int64_t *d_rows, int64_t rows, tid_set **out) {
    *out = nullptr;
    tid_set *s = new (std::nothrow) tid_set();
    if (!s) return fail(TID_ERR_OOM, "host allocation");
    s->ctx = ctx;
    s->k = 1;
    s->vars[0] = -1;
    s->cap = rows;
    s->col[0] = col;
    s->d_rows = d_rows;
    s->rows_known = rows;
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        s->shared = sb;
        ++sb->refs;
    }
    *out = s;
    return TID_OK;
}

int set_ready(tid_set *set) {
    if (!set->ready) return TID_OK;  // a view: its producer is waited for through the stream
    TID_TRY_CUDA(cudaEventRecord(set->ready, set->ctx->stream), "event record");
    return TID_OK;
}

cudaError_t reset_bounds(tid_ctx *ctx) {
    // 16 words of bounds, then the finished-CTA counter
    const size_t least = TID_MAX_COLS * sizeof(uint32_t);
    cudaError_t e = cudaMemsetAsync(ctx->bounds_dev, 0xFF, least, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->bounds_dev + TID_MAX_COLS, 0, 256 - least, ctx->stream);
    return e;
}

int check_ctx_error(tid_ctx *ctx) {
    if (ctx->freed_twice.exchange(false)) return fail(TID_ERR_CUDA, "a device block was freed twice");
    int e = *(volatile int *)ctx->err_host;
    if (e != 0) {
        *(volatile int *)ctx->err_host = 0;
        // a launch that gave up may leave the ticket counter off zero, and the
        // bounds with some of its CTAs' values
        if (ctx->lb_ticket) cudaMemsetAsync(ctx->lb_ticket, 0, sizeof(unsigned int), ctx->stream);
        if (ctx->bounds_dev) reset_bounds(ctx);
        if (e == TID_ERR_TIMEOUT) return fail(TID_ERR_TIMEOUT, "an in-kernel wait gave up");
        return fail(e, "kernel reported error %d", e);
    }
    return TID_OK;
}

struct SetCols {
    const int32_t *c[TID_MAX_COLS];
};

// n rows x k row-major from k columns: a thread writes one row, its loads in flight
// together (the columns come as arguments: a copy of their addresses to the device
// and a division per value cost more than the rows of a small set)
template <int K>
__global__ void __launch_bounds__(256) k_interleave(SetCols cols, int k, int64_t n, int32_t *__restrict__ out) {
    for (int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x; r < n; r += (int64_t)gridDim.x * 256) {
        int32_t v[K];
#pragma unroll
        for (int c = 0; c < K; ++c)
            if (c < k) v[c] = cols.c[c][r];
#pragma unroll
        for (int c = 0; c < K; ++c)
            if (c < k) out[r * k + c] = v[c];
    }
}

}  // namespace tid


// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
using namespace tid;

extern "C" const char *tid_last_error(void) { return g_err.c_str(); }

extern "C" int tid_ctx_create(int device, void *cuda_stream, tid_ctx **out) {
    clear_error();
    if (!out) return fail(TID_ERR_ARG, "tid_ctx_create: null out");
    *out = nullptr;
    int ndev = 0;
    TID_TRY_CUDA(cudaGetDeviceCount(&ndev), "cudaGetDeviceCount");
    if (device < 0 || device >= ndev) return fail(TID_ERR_ARG, "tid_ctx_create: no device %d", device);
    TID_TRY(claim_device(device));
    DeviceGuard g(device);
    tid_ctx *c = new (std::nothrow) tid_ctx();
    if (!c) return fail(TID_ERR_OOM, "host allocation");
    c->device = device;
    cudaError_t e = cudaSuccess;
    if (cuda_stream) {
        c->stream = (cudaStream_t)cuda_stream;
    } else {
        e = cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking);
        c->own_stream = true;
    }
    if (e == cudaSuccess) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        e = cudaMemPoolCreate(&c->pool, &props);
        if (e == cudaSuccess) {
            uint64_t thr = UINT64_MAX;
            cudaMemPoolSetAttribute(c->pool, cudaMemPoolAttrReleaseThreshold, &thr);
        }
    }
    void *h = nullptr;
    if (e == cudaSuccess) e = cudaHostAlloc(&h, 256, cudaHostAllocMapped);
    if (e == cudaSuccess) {
        c->err_host = (int *)h;
        *c->err_host = 0;
        void *d = nullptr;
        e = cudaHostGetDevicePointer(&d, h, 0);
        c->err_dev = (int *)d;
    }
    int rc = e == cudaSuccess ? TID_OK : fail_cuda(e, "tid_ctx_create");
    if (rc == TID_OK) note_capture(c);
    if (rc == TID_OK && !capturing(c)) rc = keep_scratch(c);
    if (rc != TID_OK) {
        if (c->err_host) cudaFreeHost(c->err_host);
        if (c->pool) cudaMemPoolDestroy(c->pool);
        if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
        delete c;
        return rc;
    }
    *out = c;
    return TID_OK;
}

extern "C" int tid_ctx_sync(tid_ctx *ctx) {
    clear_error();
    tid::Range nvtx_range("tid_ctx_sync");
    if (!ctx) return fail(TID_ERR_ARG, "tid_ctx_sync: null ctx");
    DeviceGuard g(ctx->device);
    TID_TRY_CUDA(cudaStreamSynchronize(ctx->stream), "stream synchronize");
    return check_ctx_error(ctx);
}

extern "C" int tid_ctx_destroy(tid_ctx *ctx) {
    clear_error();
    if (!ctx) return TID_OK;
    DeviceGuard g(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        for (const PendingSlot &p : ctx->pending) cudaEventDestroy(p.ev);
        ctx->pending.clear();
    }
    dev_free(ctx, ctx->kept);
    for (int i = 0; i < ctx->n_grown; ++i) dev_free(ctx, ctx->lb_grown[i]);
    drop_blocks(ctx, true);
    for (cudaEvent_t ev : ctx->free_events) cudaEventDestroy(ev);
    cudaStreamSynchronize(ctx->stream);
    for (auto *h : ctx->slabs_host) cudaFreeHost(h);
    if (ctx->err_host) cudaFreeHost(ctx->err_host);
    if (ctx->pool) cudaMemPoolDestroy(ctx->pool);
    if (ctx->own_stream) cudaStreamDestroy(ctx->stream);
    delete ctx;
    return TID_OK;
}

namespace {
// The second of two tiles, whose predecessor never reports: the look-back gives up
// after `limit` polls and sets TID_ERR_TIMEOUT.
__global__ void k_wait_for_tile(tid::Lookback lb, unsigned limit) { tid::lb_exclusive_prefix(lb, 1u, 1u, limit); }
}  // namespace

extern "C" int tid_ctx_test_bounded_wait(tid_ctx *ctx, int64_t polls) {
    clear_error();
    if (!ctx) return fail(TID_ERR_ARG, "tid_ctx_test_bounded_wait: null context");
    if (polls < 1 || polls > (int64_t)LB_SPIN_LIMIT)
        return fail(TID_ERR_ARG, "tid_ctx_test_bounded_wait: polls = %lld", (long long)polls);
    CallGuard g(ctx);
    Lookback lb{};
    TID_TRY(lookback_scratch(ctx, 2, &lb));
    k_wait_for_tile<<<1, 32, 0, ctx->stream>>>(lb, (unsigned)polls);
    TID_TRY(launch_check("k_wait_for_tile"));
    return tid_ctx_sync(ctx);
}

extern "C" int tid_ctx_inject_alloc_failure(tid_ctx *ctx, int64_t after) {
    clear_error();
    if (!ctx) return fail(TID_ERR_ARG, "tid_ctx_inject_alloc_failure: null context");
    ctx->allocs.store(0);
    ctx->fail_after.store(after < 0 ? -1 : after);
    return TID_OK;
}

namespace {
// *unsorted = 1 if some triple is smaller, in (s, p, o) order, than the one
// before it
__global__ void k_spo_unsorted(const int32_t *__restrict__ s, const int32_t *__restrict__ p,
                               const int32_t *__restrict__ o, int64_t n, int32_t *__restrict__ unsorted) {
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x + 1; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t s0 = s[i - 1], s1 = s[i];
        if (s0 != s1) {
            bad = bad || s0 > s1;
            continue;
        }
        const int32_t p0 = p[i - 1], p1 = p[i];
        bad = bad || p0 > p1 || (p0 == p1 && o[i - 1] > o[i]);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) *unsorted = 1;
}
}  // namespace

namespace tid {
bool store_spo_sorted(const tid_store *st) {
    if (st->spo_sorted < 0) {
        int32_t h = 1;
        DeviceGuard g(st->ctx->device);
        cudaError_t e = cudaMemcpyAsync(&h, st->d_unsorted, sizeof h, cudaMemcpyDeviceToHost, st->ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st->ctx->stream);
        if (e != cudaSuccess) return false;  // unknown: take the general path
        st->spo_sorted = h == 0 ? 1 : 0;
    }
    return st->spo_sorted == 1;
}
}  // namespace tid

extern "C" int tid_load(tid_ctx *ctx, const int32_t *s, const int32_t *p, const int32_t *o,
                        int64_t n, int where, int copy, tid_store **out) {
    clear_error();
    tid::Range nvtx_range("tid_load");
    if (!ctx || !out) return fail(TID_ERR_ARG, "tid_load: null argument");
    *out = nullptr;
    if (n < 0 || n > INT32_MAX) return fail(TID_ERR_ARG, "tid_load: n = %lld out of range", (long long)n);
    if (n > 0 && (!s || !p || !o)) return fail(TID_ERR_ARG, "tid_load: null column");
    if (where != TID_HOST && where != TID_DEVICE) return fail(TID_ERR_ARG, "tid_load: bad `where`");
    CallGuard g(ctx);
    tid_store *st = new (std::nothrow) tid_store();
    if (!st) return fail(TID_ERR_OOM, "host allocation");
    st->ctx = ctx;
    st->n = n;
    if (where == TID_DEVICE && !copy) {
        st->s = s;
        st->p = p;
        st->o = o;
    } else {
        const size_t colb = align_up((size_t)n * sizeof(int32_t), 256);
        int rc = dev_alloc(ctx, &st->owned, 3 * colb);
        if (rc != TID_OK) {
            delete st;
            return rc;
        }
        int32_t *base = (int32_t *)st->owned;
        int32_t *cs = base, *cp = (int32_t *)((char *)base + colb), *co = (int32_t *)((char *)base + 2 * colb);
        const cudaMemcpyKind kind = where == TID_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
        cudaError_t e = cudaSuccess;
        if (n > 0) {
            e = cudaMemcpyAsync(cs, s, (size_t)n * 4, kind, ctx->stream);
            if (e == cudaSuccess) e = cudaMemcpyAsync(cp, p, (size_t)n * 4, kind, ctx->stream);
            if (e == cudaSuccess) e = cudaMemcpyAsync(co, o, (size_t)n * 4, kind, ctx->stream);
        }
        if (e != cudaSuccess) {
            dev_free(ctx, st->owned);
            delete st;
            return fail_cuda(e, "tid_load copy");
        }
        st->s = cs;
        st->p = cp;
        st->o = co;
    }
    st->aligned16 = ((uintptr_t)st->s % 16 == 0) && ((uintptr_t)st->p % 16 == 0) &&
                    ((uintptr_t)st->o % 16 == 0);
    // the order check: one read of the store, queued like the copies
    int rc = dev_alloc(ctx, (void **)&st->d_unsorted, sizeof(int32_t));
    if (rc == TID_OK) {
        cudaError_t e = cudaMemsetAsync(st->d_unsorted, 0, sizeof(int32_t), ctx->stream);
        if (e != cudaSuccess) rc = fail_cuda(e, "tid_load");
    }
    if (rc == TID_OK && n > 1) {
        k_spo_unsorted<<<grid_for(n, 256, 8), 256, 0, ctx->stream>>>(st->s, st->p, st->o, n, st->d_unsorted);
        rc = launch_check("k_spo_unsorted");
    }
    if (rc != TID_OK) {
        if (st->d_unsorted) dev_free(ctx, st->d_unsorted);
        if (st->owned) dev_free(ctx, st->owned);
        delete st;
        return rc;
    }
    *out = st;
    return TID_OK;
}

extern "C" int tid_store_info(const tid_store *st, int64_t *n, const int32_t **s, const int32_t **p,
                              const int32_t **o) {
    clear_error();
    if (!st) return fail(TID_ERR_ARG, "tid_store_info: null store");
    if (n) *n = st->n;
    if (s) *s = st->s;
    if (p) *p = st->p;
    if (o) *o = st->o;
    return TID_OK;
}

extern "C" int tid_store_free(tid_store *st) {
    clear_error();
    if (!st) return TID_OK;
    CallGuard g(st->ctx);
    if (st->d_unsorted) dev_free(st->ctx, st->d_unsorted);
    if (st->owned) dev_free(st->ctx, st->owned);
    delete st;
    return TID_OK;
}

namespace tid {
int set_rows_host(tid_set *set, int64_t *rows) {
    if (set->rows_known < 0) {
        DeviceGuard g(set->ctx->device);
        TID_TRY_CUDA(cudaEventSynchronize(set->ready), "wait for set");
        TID_TRY(check_ctx_error(set->ctx));
        const int64_t r = *(volatile int64_t *)&set->slot.words->rows;
        if (r < 0) return fail(TID_ERR_CUDA, "row count was not produced");
        set->rows_known = r;
    }
    *rows = set->rows_known;
    return TID_OK;
}
int set_rows_host(const tid_set *set, int64_t *rows) { return set_rows_host(const_cast<tid_set *>(set), rows); }
}  // namespace tid

extern "C" int tid_set_rows(tid_set *set, int64_t *rows) {
    clear_error();
    tid::Range nvtx_range("tid_set_rows");
    if (!set || !rows) return fail(TID_ERR_ARG, "tid_set_rows: null argument");
    return set_rows_host(set, rows);
}

extern "C" int tid_set_info(const tid_set *set, int *cols, int64_t *capacity, const int8_t **var_ids,
                            int32_t *const **dev_cols, const int64_t **dev_rows) {
    clear_error();
    if (!set) return fail(TID_ERR_ARG, "tid_set_info: null set");
    if (cols) *cols = set->k;
    if (capacity) *capacity = set->cap;
    if (var_ids) *var_ids = set->vars;
    if (dev_cols) *dev_cols = set->col;
    if (dev_rows) *dev_rows = set->d_rows;
    return TID_OK;
}

extern "C" int tid_set_to_host(tid_set *set, int32_t *buf, int64_t cap_rows, int64_t *rows_out) {
    clear_error();
    tid::Range nvtx_range("tid_set_to_host");
    if (!set) return fail(TID_ERR_ARG, "tid_set_to_host: null set");
    int64_t rows = 0;
    TID_TRY(tid_set_rows(set, &rows));
    if (rows_out) *rows_out = rows;
    if (rows > cap_rows) return fail(TID_ERR_CAPACITY, "tid_set_to_host: %lld rows > %lld", (long long)rows, (long long)cap_rows);
    if (rows == 0) return TID_OK;
    if (!buf) return fail(TID_ERR_ARG, "tid_set_to_host: null buffer");
    tid_ctx *ctx = set->ctx;
    CallGuard g(ctx);
    const size_t bytes = (size_t)rows * set->k * sizeof(int32_t);
    if (set->k == 1) {
        TID_TRY_CUDA(cudaMemcpyAsync(buf, set->col[0], bytes, cudaMemcpyDeviceToHost, ctx->stream), "copy set");
    } else {
        void *tmp = nullptr;
        TID_TRY(dev_alloc(ctx, &tmp, bytes));
        SetCols sc{};
        for (int c = 0; c < set->k; ++c) sc.c[c] = set->col[c];
        const unsigned grid = grid_for(rows, 256);
        if (set->k <= 3) k_interleave<3><<<grid, 256, 0, ctx->stream>>>(sc, set->k, rows, (int32_t *)tmp);
        else k_interleave<TID_MAX_COLS><<<grid, 256, 0, ctx->stream>>>(sc, set->k, rows, (int32_t *)tmp);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(buf, tmp, bytes, cudaMemcpyDeviceToHost, ctx->stream);
        dev_free(ctx, tmp);
        if (e != cudaSuccess) return fail_cuda(e, "copy set");
    }
    TID_TRY_CUDA(cudaStreamSynchronize(ctx->stream), "copy set");
    return check_ctx_error(ctx);
}

namespace tid {
// frees a set without touching the error message (used on error paths too)
void set_free(tid_set *set) {
    if (!set) return;
    tid_ctx *ctx = set->ctx;
    DeviceGuard g(ctx->device);
    if (set->block) dev_free(ctx, set->block);
    if (set->shared) {
        SharedBlock *sb = set->shared;
        bool last;
        {
            std::lock_guard<std::mutex> lk(ctx->mu);
            last = --sb->refs == 0;
        }
        if (last) {
            note_capture(ctx);
            for (void *p : sb->ptr)
                if (p) dev_free(ctx, p);
            delete sb;
        }
    }
    if (set->slot.slab >= 0) {
        std::lock_guard<std::mutex> lk(ctx->mu);
        if (set->in_graph) {
            // every run of the graph writes the slot, for as long as the program
            // keeps the graph: it is never handed out again (nor is the event)
        } else if (set->ready) {
            // the producer may still be writing the slot: recycle it once done
            ctx->pending.push_back({set->slot, set->ready});
            set->ready = nullptr;
        } else {
            ctx->free_slots.push_back({set->slot.slab, set->slot.index});
        }
    }
    if (set->ready) cudaEventDestroy(set->ready);
    delete set;
}
}  // namespace tid

extern "C" int tid_set_free(tid_set *set) {
    clear_error();
    if (set && set->block) note_capture(set->ctx);
    tid::set_free(set);
    return TID_OK;
}
