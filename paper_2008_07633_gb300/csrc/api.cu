// Context, status, allocation and timing plumbing of libsfg.
#include <algorithm>
#include <cstdarg>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "sfg_internal.cuh"

sfg_status sfg_fail(sfg_ctx* ctx, sfg_status st, const char* fmt, ...) {
    if (ctx) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof buf, fmt, ap);
        va_end(ap);
        ctx->last_error = buf;
    }
    return st;
}

sfg_status sfg_cuda_fail(sfg_ctx* ctx, cudaError_t e, const char* where) {
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return sfg_fail(ctx, SFG_ENOMEM, "out of device memory in %s", where);
    }
    return sfg_fail(ctx, SFG_ECUDA, "CUDA error %d (%s) in %s", (int)e, cudaGetErrorString(e),
                    where);
}

// Counts an allocation; true when this one has to fail (SFG_FAULT_ALLOC).
static bool alloc_fails(sfg_ctx* ctx) {
    ctx->alloc_count++;
    return ctx->fail_alloc_at >= 0 && ctx->alloc_count == ctx->fail_alloc_at;
}

bool sfg_capturing(cudaStream_t stream) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &st) != cudaSuccess) {  // the legacy stream while another one is captured
        cudaGetLastError();
        return true;
    }
    return st != cudaStreamCaptureStatusNone;
}

constexpr size_t kKeptBlocks = 96;
constexpr int kKeptDevices = 64;
constexpr int64_t kKeptShare = 128, kKeptDeviceShare = 32;  // of a device's memory: a context's, all contexts' together

// What the contexts of one device keep together.
struct KeptDevice {
    std::mutex mu;  // guards the two lists
    std::once_flag once;
    std::atomic<int64_t> room{0};    // bytes that may still be kept
    int64_t all = 0;                 // the same before any is
    std::vector<sfg_ctx*> contexts;
    std::vector<void*> left;         // legacy blocks that lost their place while a capture forbade freeing them
    cudaStream_t frees = nullptr;    // the library's own: gives blocks back after their event, never on a user's stream
};
static KeptDevice kept_devices[kKeptDevices];

static KeptDevice& kept_device(const sfg_ctx* ctx) { return kept_devices[ctx->device]; }

// A context that is not registered (no room for its device's number, no event, no stream of the library's own)
// keeps nothing.
static void kept_register(sfg_ctx* ctx) {
    if (ctx->device >= kKeptDevices) return;
    KeptDevice& d = kept_device(ctx);
    std::call_once(d.once, [&d] {
        size_t unused = 0, total = 0;
        if (cudaMemGetInfo(&unused, &total) == cudaSuccess &&
            cudaStreamCreateWithFlags(&d.frees, cudaStreamNonBlocking) == cudaSuccess)
            d.room = d.all = (int64_t)total / kKeptDeviceShare;
        else cudaGetLastError();
    });
    if (!d.frees || cudaEventCreateWithFlags(&ctx->kept_event, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        ctx->kept_event = nullptr;
        return;
    }
    std::lock_guard<std::mutex> lock(d.mu);
    ctx->kept.reserve(kKeptBlocks);
    d.left.reserve(kKeptBlocks);
    d.contexts.push_back(ctx);
}

// From here on to sfg_scratch_settle: with the context's lock.
static SfgKept kept_remove(sfg_ctx* ctx, size_t i) {
    const SfgKept b = ctx->kept[i];
    kept_device(ctx).room.fetch_add((int64_t)b.bytes);
    ctx->kept_bytes -= (int64_t)b.bytes;
    ctx->kept.erase(ctx->kept.begin() + i);
    return b;
}

// Frees in the order of the legacy stream; not while another stream's capture forbids its use.
static void kept_free_legacy(sfg_ctx* ctx) {
    if (sfg_capturing(cudaStreamLegacy)) return;
    for (size_t i = ctx->kept.size(); i-- > 0;)
        if (ctx->kept[i].legacy) cudaFreeAsync(kept_remove(ctx, i).p, cudaStreamLegacy);
}

// Gives back what can be waited for without the context's stream, in the order of the event.
static void kept_release(sfg_ctx* ctx) {
    KeptDevice& d = kept_device(ctx);
    kept_free_legacy(ctx);
    bool first = true;
    for (size_t i = ctx->kept.size(); i-- > 0;) {
        if (!ctx->kept[i].settled) continue;
        if (first && cudaStreamWaitEvent(d.frees, ctx->kept_event, 0) != cudaSuccess) {
            cudaGetLastError();
            return;
        }
        first = false;
        cudaFreeAsync(kept_remove(ctx, i).p, d.frees);
    }
}

// The same in the order of the context's stream, which has to be alive and not captured.
static void kept_free(sfg_ctx* ctx) {
    kept_free_legacy(ctx);
    for (size_t i = ctx->kept.size(); i-- > 0;)
        if (!ctx->kept[i].legacy) cudaFreeAsync(kept_remove(ctx, i).p, ctx->stream);
}

// Blocks that lost their context or place while a capture forbade freeing them.
static void kept_free_left(KeptDevice& d) {  // with the device's lock
    if (d.left.empty() || sfg_capturing(cudaStreamLegacy)) return;
    for (void* p : d.left) cudaFreeAsync(p, cudaStreamLegacy);
    d.left.clear();
}

// An allocation has failed: everything that this context and those not in a call keep goes back to the pool.
static void kept_reclaim(sfg_ctx* ctx) {
    if (!ctx->kept_event) return;
    KeptDevice& d = kept_device(ctx);
    if (!sfg_capturing(ctx->stream)) kept_free(ctx);
    {
        std::lock_guard<std::mutex> lock(d.mu);
        kept_free_left(d);
        for (sfg_ctx* c : d.contexts) {
            if (c == ctx || c->kept_lock.exchange(1, std::memory_order_acquire)) continue;
            kept_release(c);
            c->kept_lock.store(0, std::memory_order_release);
        }
    }
    cudaStreamSynchronize(d.frees);
    if (!sfg_capturing(cudaStreamLegacy)) cudaStreamSynchronize(cudaStreamLegacy);
}

// The SMs that a stream's kernels can run on: those of its green context, if it has one, else the device's.
static int stream_sms(const sfg_ctx* ctx, cudaStream_t stream) {
    static PFN_cuStreamGetGreenCtx_v12040 green_of = nullptr;
    static PFN_cuGreenCtxGetDevResource_v12040 resource_of = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        auto find = [](const char* name) {
            void* p = nullptr;
            cudaDriverEntryPointQueryResult found;
            if (cudaGetDriverEntryPointByVersion(name, &p, 12040, cudaEnableDefault, &found) != cudaSuccess) {
                cudaGetLastError();
                return (void*)nullptr;
            }
            return found == cudaDriverEntryPointSuccess ? p : nullptr;
        };
        green_of = (PFN_cuStreamGetGreenCtx_v12040)find("cuStreamGetGreenCtx");
        resource_of = (PFN_cuGreenCtxGetDevResource_v12040)find("cuGreenCtxGetDevResource");
    });
    CUgreenCtx green = nullptr;
    CUdevResource r;
    if (!green_of || !resource_of || green_of((CUstream)stream, &green) != CUDA_SUCCESS || !green ||
        resource_of(green, &r, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS)
        return ctx->num_sms;
    return std::max(1, std::min(ctx->num_sms, (int)r.sm.smCount));
}

static void set_stream(sfg_ctx* ctx, cudaStream_t stream) {
    unsigned long long id = 0;
    const bool known = cudaStreamGetId(stream, &id) == cudaSuccess;
    if (!known) cudaGetLastError();
    if (ctx->kept_event && (!known || id != ctx->stream_id)) kept_release(ctx);
    ctx->stream = stream;
    ctx->stream_id = id;
    ctx->stream_sms = stream_sms(ctx, stream);
    ctx->on_legacy = stream == nullptr || stream == cudaStreamLegacy;
    ctx->stream_keeps = known && ctx->kept_event && stream != cudaStreamPerThread;
}

static sfg_status pool_alloc(sfg_ctx* ctx, void** p, size_t bytes) {
    cudaError_t e = ctx->alloc_count == ctx->fail_pool_at ? cudaErrorMemoryAllocation
                                                          : cudaMallocFromPoolAsync(p, bytes, ctx->pool, ctx->stream);
    if (e == cudaErrorMemoryAllocation) {
        // the contexts keep scratch and the pool freed memory; hand it back to the device and try once more
        cudaGetLastError();
        kept_reclaim(ctx);
        cudaStreamSynchronize(ctx->stream);
        cudaMemPoolTrimTo(ctx->pool, 0);
        e = cudaMallocFromPoolAsync(p, bytes, ctx->pool, ctx->stream);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return sfg_fail(ctx, SFG_ENOMEM, "cudaMallocFromPoolAsync(%zu bytes) failed: %s", bytes,
                        cudaGetErrorString(e));
    }
    return SFG_OK;
}

static sfg_status alloc_injected(sfg_ctx* ctx) {
    return sfg_fail(ctx, SFG_ENOMEM, "injected allocation failure (allocation %lld)", (long long)ctx->alloc_count);
}

sfg_status sfg_alloc(sfg_ctx* ctx, void** p, size_t bytes) {
    *p = nullptr;
    if (alloc_fails(ctx)) return alloc_injected(ctx);
    return pool_alloc(ctx, p, bytes);
}

sfg_status sfg_scratch_take(sfg_ctx* ctx, void** p, size_t* bytes) {
    *p = nullptr;
    if (alloc_fails(ctx)) return alloc_injected(ctx);
    size_t best = 0, size = SIZE_MAX;  // the smallest block that is large enough, if it is not much larger
    for (size_t i = 0; i < ctx->kept.size(); ++i) {
        const SfgKept& b = ctx->kept[i];
        if (b.legacy == ctx->on_legacy && b.bytes >= *bytes && b.bytes < size) best = i, size = b.bytes;
    }
    if (size <= *bytes + *bytes / 4 + 4096) {
        const SfgKept b = kept_remove(ctx, best);
        *p = b.p;
        *bytes = b.bytes;
        return SFG_OK;
    }
    return pool_alloc(ctx, p, *bytes);
}

// Keeps the block, the oldest ones making room; a block for which even all of the context's own would not make
// room goes back to the pool at once and leaves them where they are.
void sfg_scratch_give(sfg_ctx* ctx, void* p, size_t bytes) {
    KeptDevice& d = kept_device(ctx);
    const int64_t size = (int64_t)bytes, share = d.all / (kKeptShare / kKeptDeviceShare);
    if (size > share || size > d.room.load() + ctx->kept_bytes) return sfg_free(ctx, p);
    auto reserve = [&] {
        if (ctx->kept.size() >= kKeptBlocks || ctx->kept_bytes + size > share) return false;
        if (d.room.fetch_sub(size) >= size) return true;
        d.room.fetch_add(size);
        return false;
    };
    bool room = reserve();
    while (!room && !ctx->kept.empty()) {
        const SfgKept b = kept_remove(ctx, 0);
        if (b.legacy == ctx->on_legacy) {
            sfg_free(ctx, b.p);
        } else {
            std::lock_guard<std::mutex> lock(d.mu);
            d.left.push_back(b.p);
        }
        room = reserve();
    }
    if (!room) return sfg_free(ctx, p);
    ctx->kept.push_back({p, bytes, ctx->on_legacy, false});  // the list has its room from the start: nothing throws
    ctx->kept_bytes += size;
    ctx->kept_dirty = !ctx->on_legacy;
}

// At the end of a call: the context's event stands for the last use of everything it keeps. (Nothing is given
// back while the stream is being captured, so the record is never part of a graph.)
void sfg_scratch_settle(sfg_ctx* ctx) {
    ctx->kept_dirty = false;
    const bool ok = cudaEventRecord(ctx->kept_event, ctx->stream) == cudaSuccess;
    if (!ok) cudaGetLastError();
    for (size_t i = ctx->kept.size(); i-- > 0;) {
        if (ctx->kept[i].legacy) continue;
        if (ok) ctx->kept[i].settled = true;
        else sfg_free(ctx, kept_remove(ctx, i).p);
    }
}

void sfg_free(sfg_ctx* ctx, void* p) {
    if (p) cudaFreeAsync(p, ctx->stream);
}

// Status words of the grid barriers, one a context, in page-locked host memory that is never freed: a captured
// launch may be replayed after its context is gone (its word may then belong to a later context).
static std::mutex status_mu;
static std::vector<int*> status_free;

static int* status_take() {
    std::lock_guard<std::mutex> lock(status_mu);
    if (status_free.empty()) {
        constexpr int kWords = 1024;
        int* page = nullptr;
        if (cudaHostAlloc((void**)&page, sizeof(int) * kWords, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        for (int i = 0; i < kWords; ++i) status_free.push_back(page + i);
    }
    int* w = status_free.back();
    status_free.pop_back();
    *(volatile int*)w = 0;
    return w;
}

static void status_give(int* w) {
    std::lock_guard<std::mutex> lock(status_mu);
    if (w) status_free.push_back(w);
}

GridWait sfg_grid_wait(const sfg_ctx* ctx, const char* kernel) {
    if (ctx->fault_barrier && ctx->fault_grid == kernel) return GridWait{ctx->grid_status, 20000000ull, ctx->fault_barrier};
    return GridWait{ctx->grid_status, 2000000000ull, 0u};
}

sfg_status sfg_grid_check(sfg_ctx* ctx) {
    volatile int* w = ctx->grid_status;
    if (!*w) return SFG_OK;
    *w = 0;
    return sfg_fail(ctx, SFG_ETIMEOUT, "a launch whose CTAs wait for one another gave up: its results, or those of "
                                       "an earlier call that did not synchronise, are not valid");
}

sfg_status sfg_wait(sfg_ctx* ctx) {
    SFG_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    return sfg_grid_check(ctx);
}

sfg_status sfg_host_word(sfg_ctx* ctx, int slot, int** out) {
    if (!ctx->host_word)
        SFG_CUDA(ctx, cudaMallocHost((void**)&ctx->host_word, sizeof(int) * kSfgHostWords));
    *out = ctx->host_word + slot;
    return SFG_OK;
}

sfg_status sfg_check_dev(sfg_ctx* ctx, const void* p, const char* what) {
    if (!p) return sfg_fail(ctx, SFG_EINVAL, "%s is NULL", what);
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return sfg_fail(ctx, SFG_EINVAL, "%s is not a CUDA pointer", what);
    }
    if (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)
        return sfg_fail(ctx, SFG_EINVAL, "%s is not device memory", what);
    return SFG_OK;
}

static int grid_on(sfg_ctx* ctx, const void* kernel, int block, size_t smem, int64_t work_items, int sms) {
    // resident CTAs per SM, asked once per (kernel, block, shared memory) and context
    const auto key = std::make_tuple(kernel, block, smem);
    auto it = ctx->occupancy.find(key);
    int per_sm = 0;
    if (it != ctx->occupancy.end()) {
        per_sm = it->second;
    } else {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, smem) != cudaSuccess ||
            per_sm < 1) {
            cudaGetLastError();
            per_sm = 1;
        }
        ctx->occupancy.emplace(key, per_sm);
    }
    int64_t full = (int64_t)per_sm * sms;
    int64_t need = (work_items + block - 1) / block;
    if (need < 1) need = 1;
    return (int)(need < full ? need : full);
}

int sfg_grid(sfg_ctx* ctx, const void* kernel, int block, size_t smem, int64_t work_items) {
    return grid_on(ctx, kernel, block, smem, work_items, ctx->num_sms);
}

int sfg_coop_grid(sfg_ctx* ctx, const void* kernel, int block, int64_t work_items) {
    return grid_on(ctx, kernel, block, 0, work_items, ctx->stream_sms);
}

void sfg_tic(sfg_ctx* ctx, const char* name) {
    if (!ctx->timing) return;
    sfg_timer_rec r;
    r.name = name;
    for (int i = 0; i < 2; ++i) {
        cudaEvent_t ev;
        if (!ctx->event_pool.empty()) {
            ev = ctx->event_pool.back();
            ctx->event_pool.pop_back();
        } else if (cudaEventCreate(&ev) != cudaSuccess) {
            cudaGetLastError();
            return;
        }
        (i == 0 ? r.start : r.stop) = ev;
    }
    cudaEventRecord(r.start, ctx->stream);
    ctx->timers.push_back(r);
}

void sfg_toc(sfg_ctx* ctx) {
    if (!ctx->timing || ctx->timers.empty()) return;
    cudaEventRecord(ctx->timers.back().stop, ctx->stream);
}

uint32_t sfg_tune_key(int K, sfg_dtype dt, int bucket) {
    return ((uint32_t)K << 16) | ((uint32_t)dt << 8) | (uint32_t)bucket;
}

int sfg_degree_bucket(const sfg_graph* L) {
    const double avg = L->n > 0 ? (2.0 * (double)L->m) / (double)L->n : 0.0;
    int b = 0;
    while (b < 15 && (double)(2 << b) <= avg) ++b;  // bucket b: 2^b <= avg degree < 2^(b+1)
    return b;
}

int sfg_tuned_variant(const sfg_ctx* ctx, int K, sfg_dtype dt, const sfg_graph* L) {
    if (ctx->tune.empty()) return -1;
    auto it = ctx->tune.find(sfg_tune_key(K, dt, sfg_degree_bucket(L)));
    return it == ctx->tune.end() ? -1 : it->second;
}

void sfg_tune_record(sfg_ctx* ctx, int K, sfg_dtype dt, const sfg_graph* L, int variant) {
    ctx->tune[sfg_tune_key(K, dt, sfg_degree_bucket(L))] = variant;
}

int sfg_score_shape(const sfg_ctx* ctx, int K, sfg_dtype dt, const sfg_graph* L) {
    const int b = sfg_degree_bucket(L);
    if (!ctx->score_tune.empty()) {
        auto it = ctx->score_tune.find(sfg_tune_key(K, dt, b));
        if (it != ctx->score_tune.end()) return it->second;
    }
    return b <= 2 ? 0 : 1;
}

extern "C" {

// The library's memory pool on `device`: created on first use and kept for the life of the
// process, shared by every context on the device, with a release threshold that keeps freed
// memory mapped (the device's default pool returns everything at each synchronisation, and the
// next large block then pays for mapping it again). Graphs and networks may outlive the context
// that made them, so the pool is never destroyed; contexts only trim it.
static cudaMemPool_t device_pool(int device) {
    static std::mutex mu;
    static std::map<int, cudaMemPool_t> pools;
    std::lock_guard<std::mutex> lock(mu);
    auto it = pools.find(device);
    if (it != pools.end()) return it->second;
    cudaMemPoolProps pp = {};
    pp.allocType = cudaMemAllocationTypePinned;
    pp.handleTypes = cudaMemHandleTypeNone;
    pp.location.type = cudaMemLocationTypeDevice;
    pp.location.id = device;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &pp) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    uint64_t keep = UINT64_MAX;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    pools[device] = pool;
    return pool;
}

sfg_status sfg_ctx_create(sfg_ctx** out, int device, void* cuda_stream) {
    if (!out) return SFG_EINVAL;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
        cudaGetLastError();
        return SFG_EINVAL;
    }
    SfgDeviceGuard guard(device);
    sfg_ctx* c = new sfg_ctx();
    c->device = device;
    cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, device);
    if (c->num_sms < 1) c->num_sms = 1;
    if (const char* f = std::getenv("SFG_FAULT_ALLOC")) c->fail_alloc_at = std::atoll(f);
    if (const char* f = std::getenv("SFG_FAULT_POOL")) c->fail_pool_at = std::atoll(f);
    if (const char* f = std::getenv("SFG_BUILD_SORT")) c->build_sorts = std::atoi(f) != 0;
    if (const char* f = std::getenv("SFG_FAULT_MMA_WAIT")) c->withhold_mma = std::atoi(f) != 0;
    if (const char* f = std::getenv("SFG_FAULT_GRID_WAIT")) {
        const char* colon = std::strchr(f, ':');
        if (colon) {
            c->fault_grid.assign(f, colon - f);
            c->fault_barrier = (unsigned)std::atoi(colon + 1);
        }
    }
    c->pool = device_pool(device);
    c->grid_status = status_take();
    if (!c->pool || !c->grid_status) {
        status_give(c->grid_status);
        delete c;
        return SFG_ECUDA;
    }
    // The allocation-free entry points' file-scope scratch is resolved here, so that the module
    // that holds it is loaded (and its memory taken) when a context is created, never inside
    // one of those calls.
    if (sfg_noalloc_prepare(c) != SFG_OK) {
        status_give(c->grid_status);
        delete c;
        return SFG_ECUDA;
    }
    kept_register(c);
    set_stream(c, (cudaStream_t)cuda_stream);
    *out = c;
    return SFG_OK;
}

sfg_status sfg_ctx_trim(sfg_ctx* ctx) {
    if (!ctx) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    if (ctx->kept_event) {
        kept_free(ctx);
        std::lock_guard<std::mutex> lock(kept_device(ctx).mu);
        kept_free_left(kept_device(ctx));
    }
    SFG_TRY(sfg_wait(ctx));
    SFG_CUDA(ctx, cudaMemPoolTrimTo(ctx->pool, 0));
    return SFG_OK;
}

void sfg_ctx_destroy(sfg_ctx* ctx) {
    if (!ctx) return;
    SfgDeviceGuard guard(ctx->device);
    for (auto& r : ctx->timers) {
        cudaEventDestroy(r.start);
        cudaEventDestroy(r.stop);
    }
    for (auto e : ctx->event_pool) cudaEventDestroy(e);
    const bool capturing = sfg_capturing(ctx->stream);  // such a stream cannot be waited for
    if (ctx->host_word) {
        if (!capturing) cudaStreamSynchronize(ctx->stream);
        cudaFreeHost(ctx->host_word);
    }
    if (ctx->kept_event) {
        KeptDevice& d = kept_device(ctx);
        {   // no other context takes from this one any more
            std::lock_guard<std::mutex> lock(d.mu);
            d.contexts.erase(std::find(d.contexts.begin(), d.contexts.end(), ctx));
        }
        if (capturing) kept_release(ctx);
        else kept_free(ctx);
        std::lock_guard<std::mutex> lock(d.mu);
        while (!ctx->kept.empty()) d.left.push_back(kept_remove(ctx, 0).p);
        kept_free_left(d);
        cudaEventDestroy(ctx->kept_event);
    }
    // unused memory goes back to the device; memory of live graphs stays valid
    if (!capturing) cudaStreamSynchronize(ctx->stream);
    cudaMemPoolTrimTo(ctx->pool, 0);
    status_give(ctx->grid_status);
    delete ctx;
}

sfg_status sfg_ctx_set_stream(sfg_ctx* ctx, void* cuda_stream) {
    if (!ctx) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    set_stream(ctx, (cudaStream_t)cuda_stream);
    return SFG_OK;
}

const char* sfg_last_error(const sfg_ctx* ctx) { return ctx ? ctx->last_error.c_str() : ""; }

sfg_status sfg_ctx_timing(sfg_ctx* ctx, int on) {
    if (!ctx) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    SFG_TRY(sfg_wait(ctx));
    for (auto& r : ctx->timers) {
        ctx->event_pool.push_back(r.start);
        ctx->event_pool.push_back(r.stop);
    }
    ctx->timers.clear();
    ctx->timing = on != 0;
    return SFG_OK;
}

sfg_status sfg_ctx_kernel_time(sfg_ctx* ctx, const char* prefix, int64_t* launches_host,
                               double* ms_host) {
    if (!ctx || !prefix || !launches_host || !ms_host) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    SFG_TRY(sfg_wait(ctx));
    int64_t n = 0;
    double total = 0.0;
    size_t len = std::strlen(prefix);
    for (auto& r : ctx->timers) {
        if (std::strncmp(r.name, prefix, len) != 0) continue;
        float ms = 0.f;
        SFG_CUDA(ctx, cudaEventElapsedTime(&ms, r.start, r.stop));
        total += ms;
        ++n;
    }
    *launches_host = n;
    *ms_host = total;
    return SFG_OK;
}

sfg_status sfg_ctx_launches(const sfg_ctx* ctx, int64_t* launches_host) {
    if (!ctx || !launches_host) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    *launches_host = ctx->launches;
    return SFG_OK;
}

sfg_status sfg_autotune(sfg_ctx* ctx, const sfg_graph* L, int K, sfg_dtype storage,
                        int* variant_host, double* us_per_sweep_host) {
    if (!ctx) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    if (!L) return sfg_fail(ctx, SFG_EINVAL, "graph is NULL");
    if (!sfg_k_supported(K, storage))
        return sfg_fail(ctx, SFG_EUNSUPPORTED, "K=%d unsupported for dtype %d", K, (int)storage);
    return sfg_autotune_impl(ctx, L, K, storage, variant_host, us_per_sweep_host);
}

sfg_status sfg_tune_set(sfg_ctx* ctx, int K, sfg_dtype storage, int degree_bucket, int variant) {
    if (!ctx) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    if (degree_bucket < 0 || degree_bucket > 15 || variant < -1 || variant >= SFG_SWEEP_VARIANTS)
        return sfg_fail(ctx, SFG_EINVAL, "bad tuning entry");
    const uint32_t key = sfg_tune_key(K, storage, degree_bucket);
    if (variant < 0) ctx->tune.erase(key);
    else ctx->tune[key] = variant;
    return SFG_OK;
}

sfg_status sfg_tune_set_score(sfg_ctx* ctx, int K, sfg_dtype storage, int degree_bucket,
                              int shape) {
    if (!ctx) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    if (degree_bucket < 0 || degree_bucket > 15 || shape < -1 || shape >= SFG_SCORE_SHAPES)
        return sfg_fail(ctx, SFG_EINVAL, "bad tuning entry");
    const uint32_t key = sfg_tune_key(K, storage, degree_bucket);
    if (shape < 0) ctx->score_tune.erase(key);
    else ctx->score_tune[key] = shape;
    return SFG_OK;
}

sfg_status sfg_tune_table(const sfg_ctx* ctx, char* buf, int64_t cap, int64_t* len_host) {
    if (!ctx || !len_host) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    static const int tpi[SFG_SWEEP_VARIANTS] = {1, 2, 4, 1, 2, 4};
    static const int minb[SFG_SWEEP_VARIANTS] = {4, 4, 4, 3, 3, 3};
    std::map<uint32_t, std::pair<int, int>> keys;  // key -> (sweep variant, scorer shape)
    for (auto& kv : ctx->tune) keys[kv.first] = {kv.second, -1};
    for (auto& kv : ctx->score_tune) {
        auto it = keys.find(kv.first);
        if (it == keys.end()) keys[kv.first] = {-1, kv.second};
        else it->second.second = kv.second;
    }
    std::string j = "[";
    for (auto& kv : keys) {
        char item[224];
        const int v = kv.second.first, s = kv.second.second;
        snprintf(item, sizeof item,
                 "%s{\"K\": %u, \"dtype\": %u, \"degree_bucket\": %u, \"variant\": %d, "
                 "\"tiles_per_warp\": %d, \"ctas_per_sm\": %d, \"score_shape\": %d}",
                 j.size() > 1 ? ", " : "", kv.first >> 16, (kv.first >> 8) & 0xff, kv.first & 0xff,
                 v, v >= 0 ? tpi[v] : 0, v >= 0 ? minb[v] : 0, s);
        j += item;
    }
    j += "]";
    *len_host = (int64_t)j.size();
    if (buf && cap > 0) {
        const size_t n = std::min((size_t)cap - 1, j.size());
        memcpy(buf, j.data(), n);
        buf[n] = 0;
        if ((int64_t)j.size() >= cap) return SFG_ECAPACITY;
    }
    return SFG_OK;
}

}  // extern "C"
