// Internal declarations shared by the translation units of libsfg (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <cstdint>
#include <algorithm>
#include <atomic>
#include <cmath>
#include <map>
#include <cstdio>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/sfg.h"
#include "gridbar.cuh"

// ------------------------------------------------------------------------------------------------
// Context: device, borrowed stream, last error text, optional per-kernel event timers.
// ------------------------------------------------------------------------------------------------
struct sfg_timer_rec {
    const char* name;
    cudaEvent_t start, stop;
};

// A scratch block that a context keeps after the call that used it, free for work on its stream. legacy: used on the
// legacy default stream, which is always there. settled: the context's event has been recorded since the block was
// given back, so that its last use can be waited for without the stream.
struct SfgKept {
    void* p;
    size_t bytes;
    bool legacy;
    bool settled;
};

struct sfg_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    cudaMemPool_t pool = nullptr;          // the device's stream-ordered pool of the library
    int* host_word = nullptr;              // pinned host ints for flags read after a sync
    int num_sms = 0;
    int stream_sms = 0;                    // of them, those that the stream's kernels can run on
    std::string last_error;
    bool timing = false;
    std::vector<sfg_timer_rec> timers;     // recorded this session
    std::vector<cudaEvent_t> event_pool;   // free events
    int64_t launches = 0;                  // kernels launched through this context
    std::map<uint32_t, int> tune;          // (K, dtype, degree bucket) -> sweep variant
    std::map<uint32_t, int> score_tune;    // (K, dtype, degree bucket) -> scorer launch shape
    std::map<std::tuple<const void*, int, size_t>, int> occupancy;  // resident CTAs per SM
    // Scratch kept for the next call, oldest first. What is not marked legacy was used on the current stream. A call
    // on the context holds kept_lock throughout; another context that runs out of memory takes the blocks of
    // contexts that are not in a call (it never waits for the lock).
    std::atomic<int> kept_lock{0};
    int call_depth = 0;                    // entry points call one another
    std::vector<SfgKept> kept;
    int64_t kept_bytes = 0;
    bool kept_dirty = false;               // blocks given back since the event was recorded
    cudaEvent_t kept_event = nullptr;      // NULL: nothing is kept
    unsigned long long stream_id = 0;      // of the current stream: a handle can name another stream later
    bool stream_keeps = false;             // not the per-thread default stream, whose handle names many
    bool on_legacy = false;                // the current stream is the legacy default stream
    int64_t alloc_count = 0;               // for the allocation-failure injection hook
    int64_t fail_alloc_at = -1;            // SFG_FAULT_ALLOC=<n>: the n-th allocation fails
    int64_t fail_pool_at = -1;             // SFG_FAULT_POOL=<n>: the n-th finds the pool out of memory at
                                           // its first try, if it comes from the pool
    bool build_sorts = false;              // SFG_BUILD_SORT=1: graphs are built by the sort of all entries
    bool withhold_mma = false;             // SFG_FAULT_MMA_WAIT=1: tensor-core kernels issue no
                                           // MMA, so their bounded completion waits run out
    int* grid_status = nullptr;            // host word that grid barriers set when a wait runs out
    std::string fault_grid;                // SFG_FAULT_GRID_WAIT=<kernel>:<n>: the waits of that kernel's
    unsigned fault_barrier = 0;            // n-th barrier run out (after 20 ms)
};

struct sfg_graph {
    int device = -1;           // device that holds the arrays
    int32_t n = 0;
    int64_t m = 0;             // canonical edges
    double reach = INFINITY;   // mean |u - v| of the edges it was built from (of its supergraph's; infinite: not known)
    int32_t* eu = nullptr;     // [m] canonical edge endpoints, eu < ev, sorted
    int32_t* ev = nullptr;
    float* ew = nullptr;       // [m]
    int32_t* row_ptr = nullptr;// [n+1]
    int2* colval = nullptr;    // [2m] (column, float bits of the weight), rows sorted by column
    int32_t* eid = nullptr;    // [2m] canonical edge id of each CSR entry
    double* deg = nullptr;     // [n]
    double* invdeg = nullptr;  // [n] 1 / deg in FP64 (0 for isolated nodes)
    // Gauss-Seidel colouring, built on first use (color.cu): colour per node, the nodes sorted
    // by (colour, id), and colour c's nodes at gs_order[gs_off[c], gs_off[c + 1]).
    int32_t* gs_color = nullptr;
    int32_t* gs_order = nullptr;
    std::vector<int64_t> gs_off;
    // Rows with more entries than the sweep's heavy-row threshold, built on the first sweep
    // (smooth.cu): hv_n rows (-1 = not built yet) at hv_rows, row h's segments at
    // hv_seg[hv_soff[h], hv_soff[h + 1]), each (row, first entry, end entry, 0).
    int32_t hv_n = -1;
    int64_t hv_nseg = 0;
    bool hv_spread = false;    // hub rows, and the other rows' lengths vary widely (see k_heavy_mark)
    int32_t* hv_rows = nullptr;
    int32_t* hv_soff = nullptr;
    int4* hv_seg = nullptr;
    // The same rows grouped by Gauss-Seidel colour class (built on the first Gauss-Seidel
    // smoothing): gh_rows sorted by (colour, id), row k's segments at gh_seg[gh_soff[k],
    // gh_soff[k + 1]); colour c's rows at [gh_coff[c], gh_coff[c + 1]) and its segments at
    // [gh_scoff[c], gh_scoff[c + 1]).
    bool gh_ready = false;
    int32_t* gh_rows = nullptr;
    int32_t* gh_soff = nullptr;
    int4* gh_seg = nullptr;
    std::vector<int64_t> gh_coff, gh_scoff;
    cudaStream_t stream = nullptr;
};

// Every entry point runs with the context's device current and gives the caller's current device
// back when it returns (cudaSetDevice only when the two differ).
struct SfgDeviceGuard {
    int prev = -1;
    explicit SfgDeviceGuard(int device) {
        int cur = -1;
        if (device < 0 || cudaGetDevice(&cur) != cudaSuccess || cur == device) return;
        if (cudaSetDevice(device) == cudaSuccess) prev = cur;
        else cudaGetLastError();  // the entry point's own CUDA calls then report the failure
    }
    ~SfgDeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
    SfgDeviceGuard(const SfgDeviceGuard&) = delete;
    SfgDeviceGuard& operator=(const SfgDeviceGuard&) = delete;
};
void sfg_scratch_settle(sfg_ctx* ctx);
struct SfgCall {
    SfgDeviceGuard device;
    sfg_ctx* ctx;
    explicit SfgCall(sfg_ctx* c) : device(c->device), ctx(c) {
        if (c->call_depth++ == 0)
            while (c->kept_lock.exchange(1, std::memory_order_acquire)) {}  // held for some frees at most
    }
    explicit SfgCall(const sfg_ctx* c) : device(c->device), ctx(nullptr) {}
    ~SfgCall() {
        if (!ctx) return;
        if (ctx->kept_dirty) sfg_scratch_settle(ctx);
        if (--ctx->call_depth == 0) ctx->kept_lock.store(0, std::memory_order_release);
    }
    SfgCall(const SfgCall&) = delete;
    SfgCall& operator=(const SfgCall&) = delete;
};
#define SFG_DEVICE(ctx) SfgCall sfg_call_(ctx)

// ------------------------------------------------------------------------------------------------
// Status helpers. Every API entry point returns through these so the text lands in ctx.
// ------------------------------------------------------------------------------------------------
sfg_status sfg_fail(sfg_ctx* ctx, sfg_status st, const char* fmt, ...);
sfg_status sfg_cuda_fail(sfg_ctx* ctx, cudaError_t e, const char* where);

#define SFG_CUDA(ctx, call)                                                 \
    do {                                                                    \
        cudaError_t _e = (call);                                            \
        if (_e != cudaSuccess) return sfg_cuda_fail((ctx), _e, #call);      \
    } while (0)

#define SFG_TRY(call)                                                       \
    do {                                                                    \
        sfg_status _s = (call);                                             \
        if (_s != SFG_OK) return _s;                                        \
    } while (0)

#define SFG_LAUNCH_CHECK(ctx, name)                                         \
    do {                                                                    \
        cudaError_t _e = cudaGetLastError();                                \
        if (_e != cudaSuccess) return sfg_cuda_fail((ctx), _e, name);       \
    } while (0)

// Stream-ordered device allocation from the context's pool (cudaMallocAsync).
sfg_status sfg_alloc(sfg_ctx* ctx, void** p, size_t bytes);
void sfg_free(sfg_ctx* ctx, void* p);

// Scratch from the blocks the context keeps from its earlier calls, else from the pool; *bytes becomes the
// block's size. A kept block is reused on the stream it was used on only. What a context keeps is bounded
// (kKeptBlocks, and 1/128 of the device's memory; 1/32 over all contexts of a device) and goes back to the pool
// with sfg_ctx_trim, sfg_ctx_set_stream to another stream, sfg_ctx_destroy, and when an allocation of any
// context on the device fails. An event recorded at the end of each call stands for the last use, so that a
// change of stream never touches the old one: its owner may have destroyed it, work pending, and its handle
// may already name another stream (streams are told apart by their ids). The legacy default stream cannot be
// destroyed and needs no event, which a call of 50 us would feel (1-2 us).
// Why: the pool took 45-190 us for each of the four large blocks of an end-to-end call on the 128^3 grid, with the
// GPU idle, and about 1 us for each small one (GB300, all scratch from the pool / kept: that call
// 7,347 / 7,084 us, two-level 14,170 / 13,970, a 64 x 64 grid 257 / 241, a gradient over 65,536 rows 74 / 61).
sfg_status sfg_scratch_take(sfg_ctx* ctx, void** p, size_t* bytes);
void sfg_scratch_give(sfg_ctx* ctx, void* p, size_t bytes);
bool sfg_capturing(cudaStream_t stream);

// Scoped list of scratch allocations released (stream-ordered) at scope exit. A captured call takes and
// frees its own (nodes of the graph being captured); any other call goes through the kept blocks.
struct Scratch {
    sfg_ctx* ctx;
    bool keep;
    std::vector<std::pair<void*, size_t>> ptrs;  // size 0: not to be kept
    explicit Scratch(sfg_ctx* c) : ctx(c), keep(c->stream_keeps && !sfg_capturing(c->stream)) {}
    ~Scratch() {
        for (auto& q : ptrs) {
            if (!q.first) continue;
            if (keep && q.second > 0) sfg_scratch_give(ctx, q.first, q.second);
            else sfg_free(ctx, q.first);
        }
    }
    template <typename T>
    sfg_status get(T** p, size_t count) {
        void* q = nullptr;
        size_t bytes = count * sizeof(T) > 0 ? count * sizeof(T) : 16;
        SFG_TRY(keep ? sfg_scratch_take(ctx, &q, &bytes) : sfg_alloc(ctx, &q, bytes));
        ptrs.emplace_back(q, keep ? bytes : 0);
        *p = static_cast<T*>(q);
        return SFG_OK;
    }
    void adopt(void* p) { ptrs.emplace_back(p, 0); }  // take ownership from the caller
    void release(void* p) {  // hand ownership to the caller
        for (auto& q : ptrs)
            if (q.first == p) q.first = nullptr;
    }
};

// The context's pinned host ints (allocated on first use): a stream-ordered copy into one costs no
// synchronisation, and the host reads it after the next one. Slots: 1 pointer-jumping flag, 3
// breadth-first flag; from kSfgHostBuild on, 64-bit words read back together (a graph build's, a
// spanning forest's, a network's loss).
constexpr int kSfgHostBuild = 8, kSfgHostWords = 64;
sfg_status sfg_host_word(sfg_ctx* ctx, int slot, int** out);

// Kernel timing (no-ops unless ctx->timing).
void sfg_tic(sfg_ctx* ctx, const char* name);
void sfg_toc(sfg_ctx* ctx);

// Pointer checks: NULL or not device-accessible memory -> SFG_EINVAL.
sfg_status sfg_check_dev(sfg_ctx* ctx, const void* p, const char* what);

// Grid size for a grid-stride kernel: a whole number of waves over the SMs.
int sfg_grid(sfg_ctx* ctx, const void* kernel, int block, size_t smem, int64_t work_items);
// The same for a cooperative launch, whose CTAs have to be resident together: over the SMs of the stream.
int sfg_coop_grid(sfg_ctx* ctx, const void* kernel, int block, int64_t work_items);

static inline unsigned ceil_div_u(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

// ------------------------------------------------------------------------------------------------
// Device primitives (primitives.cu)
// ------------------------------------------------------------------------------------------------
// out[i] = sum_{j<i} in[j] for i in [0, n]; out has n + 1 entries (out[n] = total).
sfg_status sfg_scan_u8(sfg_ctx* ctx, const uint8_t* in, int64_t* out, int64_t n);
sfg_status sfg_scan_i32(sfg_ctx* ctx, const int32_t* in, int64_t* out, int64_t n);
sfg_status sfg_scan_i64(sfg_ctx* ctx, const int64_t* in, int64_t* out, int64_t n);
// Stable LSD radix sort of (key, val) pairs on the low `bits` bits of the keys. The sorted data
// ends in (*keys, *vals); the pointers may be swapped with the alternate buffers.
sfg_status sfg_radix_sort_pairs(sfg_ctx* ctx, uint64_t** keys, uint32_t** vals,
                                uint64_t** keys_alt, uint32_t** vals_alt, int64_t n, int bits);
// Wait for the context's stream: the last step of every entry point that is documented to synchronise, so
// that what it made may be used from any stream, and its inputs released, when it returns. Like every wait of
// the library it reports a grid barrier that has run out since the last one (sfg_grid_check: SFG_ETIMEOUT, once).
sfg_status sfg_wait(sfg_ctx* ctx);
sfg_status sfg_grid_check(sfg_ctx* ctx);
// The barrier limits of a cooperative launch of `kernel`.
GridWait sfg_grid_wait(const sfg_ctx* ctx, const char* kernel);
// Copy scalars back (synchronises the stream).
sfg_status sfg_read_i64(sfg_ctx* ctx, const int64_t* dev, int64_t* host);

// ------------------------------------------------------------------------------------------------
// Cross-unit helpers
// ------------------------------------------------------------------------------------------------
// Build an sfg_graph from an input edge list already on the device (validated or not).
sfg_status sfg_build_graph(sfg_ctx* ctx, int32_t n, int64_t m, const int32_t* u,
                           const int32_t* v, const float* w, bool validate, sfg_graph** out,
                           int32_t* fine2coarse_out);
// off_ids (may be NULL) receives the ids of the edges outside the mask, ascending, in an allocation
// of the context (at least m - kept entries) that the caller frees.
sfg_status sfg_subgraph_impl(sfg_ctx* ctx, const sfg_graph* g, const uint8_t* mask,
                             sfg_graph** out, int32_t** off_ids = nullptr);
// comp_out (optional, n entries): each node's component label, a node of that component.
// key_id (m entries, may be NULL): the id that breaks weight ties for edge e (default e), with
// key_inv its inverse; a relabelled copy of a graph passes its original edge ids, so that its
// forest is the original graph's forest edge for edge.
sfg_status sfg_mst_impl(sfg_ctx* ctx, const sfg_graph* g, const uint8_t* allow, uint8_t* mask,
                        int64_t* n_tree, int32_t* comp_out = nullptr,
                        const int32_t* key_id = nullptr, const int32_t* key_inv = nullptr);
sfg_status sfg_smooth_impl(sfg_ctx* ctx, const sfg_graph* L, int K, int steps, double omega,
                           uint64_t seed, sfg_dtype storage, void* X_out);
// sg, sp (may be NULL): per-column scales applied to raw blocks (projection folded in).
sfg_status sfg_score_impl(sfg_ctx* ctx, const sfg_graph* LG, const void* XG, const void* XP,
                          int K, sfg_dtype storage, const int32_t* ids, int64_t ne,
                          sfg_score_mode mode, float* out, const float* sg = nullptr,
                          const float* sp = nullptr);
sfg_status sfg_score_batched_impl(sfg_ctx* ctx, const sfg_graph* LG, const void* XG,
                                  const void* XP, int K, sfg_dtype storage, const int32_t* ids,
                                  int64_t ne, sfg_score_mode mode, float* out, const float* sg,
                                  const float* sp, const int32_t* node_off, int ngraphs);
// orig_local (n entries, may be NULL): the graph-local node id whose seeded row row r carries
// (default r - node_off[g]), for unions whose nodes were reordered.
sfg_status sfg_filter_score_batched_impl(sfg_ctx* ctx, const sfg_graph* U, const sfg_graph* PU,
                                         const int32_t* orig_local,
                                         int ng, const int32_t* node_off, int K, int steps,
                                         double omega, uint64_t seed, sfg_dtype storage,
                                         const int32_t* ids, int64_t ne, sfg_score_mode mode,
                                         float* scores);
// Top-k per segment: of the candidates [seg_off[s], seg_off[s+1]) of segment s the k_dev[s] largest
// get mask[id] = 1.
sfg_status sfg_topk_segmented_mark(sfg_ctx* ctx, const float* scores, const int32_t* ids,
                                   int64_t ne, int nseg, const int64_t* seg_off,
                                   const int64_t* k_dev, uint8_t* mask);
typedef struct sfg_mlp sfg_mlp;
sfg_status sfg_mlp_forward_impl(sfg_ctx* ctx, const sfg_mlp* net, const float* feats, int64_t ne,
                                float* out);
sfg_status sfg_mlp_check_impl(sfg_ctx* ctx, const sfg_mlp* net);
sfg_status sfg_edge_features_impl(sfg_ctx* ctx, const sfg_graph* LG, const sfg_graph* LP, int K,
                                  int steps, double omega, uint64_t seed, sfg_dtype storage,
                                  const int32_t* ids, int64_t ne, float* feats);
sfg_status sfg_filter_score_impl(sfg_ctx* ctx, const sfg_graph* LG, const sfg_graph* LP, int K,
                                 int steps, double omega, uint64_t seed, sfg_dtype storage,
                                 const int32_t* ids, int64_t ne, sfg_score_mode mode,
                                 float* scores);
sfg_status sfg_topk_impl(sfg_ctx* ctx, const float* scores, const int32_t* ids, int64_t ne,
                         int64_t k, int32_t* out);
sfg_status sfg_coarsen_impl(sfg_ctx* ctx, const sfg_graph* L, const void* X, int K,
                            sfg_dtype storage, int32_t* agg, int32_t* f2c, int32_t* nc,
                            sfg_graph** coarse);
sfg_status sfg_backward_impl(sfg_ctx* ctx, const sfg_graph* fine, const int32_t* agg,
                             const int32_t* f2c, const sfg_graph* coarse, const uint8_t* pmask_c,
                             uint8_t* pmask_f);
void sfg_graph_free(sfg_graph* g);
// Device arrays of a graph with n nodes and m canonical edges (contents unset).
sfg_status sfg_alloc_graph(sfg_ctx* ctx, int32_t n, int64_t m, sfg_graph** out);
bool sfg_k_supported(int K, sfg_dtype dt);
// Tile-shape tuning table of a context (see sfg_autotune). Variant -1 = none recorded.
int sfg_degree_bucket(const sfg_graph* L);
uint32_t sfg_tune_key(int K, sfg_dtype dt, int bucket);
int sfg_tuned_variant(const sfg_ctx* ctx, int K, sfg_dtype dt, const sfg_graph* L);
void sfg_tune_record(sfg_ctx* ctx, int K, sfg_dtype dt, const sfg_graph* L, int variant);
// Launch shape of the scorer for graphs like L: the recorded one, else 0 (one tile per warp
// iteration, four CTAs per SM) below an average degree of 8 and 1 (two tiles, two CTAs) above.
int sfg_score_shape(const sfg_ctx* ctx, int K, sfg_dtype dt, const sfg_graph* L);
// Times both scorer shapes on every edge of L with X as both blocks and records the faster.
sfg_status sfg_score_autotune_impl(sfg_ctx* ctx, const sfg_graph* L, int K, sfg_dtype storage,
                                   const void* X);
sfg_status sfg_autotune_impl(sfg_ctx* ctx, const sfg_graph* L, int K, sfg_dtype storage,
                             int* best, double* us);

// splitmix64 (Steele, Lea & Flood 2014), host and device.
__host__ __device__ inline uint64_t sfg_splitmix64(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
// kappa(L_G, L_P) for P = the masked edges of G (kappa.cu); info6 (nullable) as sfg_kappa's.
sfg_status sfg_kappa_impl(sfg_ctx* ctx, const sfg_graph* G, const uint8_t* mask, int steps,
                          uint64_t seed, double* kappa, double* info6);
// Build the Gauss-Seidel colouring of L once (cached on the graph; color.cu).
sfg_status sfg_gs_prepare(sfg_ctx* ctx, const sfg_graph* L);
// Rows with more than SFG_HEAVY_ROW entries and their SFG_HEAVY_SEG-entry segments (hv_* of the
// graph), built once per graph (smooth.cu); the sweep and the spanning-forest rounds use them.
constexpr int32_t SFG_HEAVY_ROW = 256, SFG_HEAVY_SEG = 128;
sfg_status sfg_heavy_prepare(sfg_ctx* ctx, const sfg_graph* L);
// Give P (a subgraph of G on the same nodes) G's colouring, which is proper for P too.
sfg_status sfg_gs_inherit(sfg_ctx* ctx, const sfg_graph* P, const sfg_graph* G);
// y_p = d_p - omega * (weight to nodes after p in (colour, id) order): the weights of the
// quantity y^T x that the colour-ordered SOR sweep conserves (color.cu).
__global__ void k_gs_weights(int32_t n, const int32_t* __restrict__ row_ptr,
                             const int2* __restrict__ colval, const int32_t* __restrict__ color,
                             const double* __restrict__ deg, double omega, double* __restrict__ y);
__global__ void k_gs_weights_heavy(int32_t nh, const int32_t* __restrict__ hrow,
                                   const int32_t* __restrict__ row_ptr, const int2* __restrict__ colval,
                                   const int32_t* __restrict__ color, double omega, double* __restrict__ y);
sfg_status sfg_smooth_gs_impl(sfg_ctx* ctx, const sfg_graph* L, int K, int steps, double omega,
                              uint64_t seed, sfg_dtype storage, void* X_out);
sfg_status sfg_pointer_jump(sfg_ctx* ctx, int32_t n, int32_t* parent);
sfg_status sfg_count_mask(sfg_ctx* ctx, const uint8_t* mask, int64_t m, int64_t* count_host);
sfg_status sfg_affinity_impl(sfg_ctx* ctx, const sfg_graph* L, const void* X, int K,
                             sfg_dtype storage, double* delta);
// Resolve (once per device, with ctx's device current) the device address of the file-scope
// scratch of the allocation-free entry points (noalloc.cu); called by sfg_ctx_create.
sfg_status sfg_noalloc_prepare(sfg_ctx* ctx);
