// Graph canonicalisation and the CSR Laplacian (Sec. 2.1: A(p,q) = w(p,q), D(p,p) = sum_t w(p,t),
// L = D - A; Sec. 4: positive weights).
//
// By rows (the usual path): every directed entry (column, input position) is placed in its row by
// a counting pass and each row is then sorted on chip, so an entry crosses HBM a few times instead
// of once per radix digit (see build_by_rows; rows too long for that are sorted among themselves). By sort
// (2m >= 2^31, or too much in such rows): one stable radix sort of the 2m directed entries keyed by (row, column).
// Both give the CSR rows sorted by column with parallel edges merged by an FP64 sum in input order
// rounded once to FP32; the upper-triangle entries, in order, are the canonical edge list (edge id
// = rank among them), and a lower-triangle entry takes the id of its mirror.
#include <cmath>
#include <type_traits>

#include "sfg_internal.cuh"
#include "dot64.cuh"

namespace {

constexpr int kBlock = 256;

__global__ void k_lap_expand(int32_t n, int64_t m, const int32_t* __restrict__ u,
                             const int32_t* __restrict__ v, const float* __restrict__ w, int bits,
                             uint64_t sent, uint64_t* __restrict__ keys,
                             uint32_t* __restrict__ vals, int* __restrict__ err) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = u[e], b = v[e];
        const float ww = w[e];
        const bool bad = a < 0 || a >= n || b < 0 || b >= n || !isfinite(ww) || !(ww > 0.0f);
        if (bad) atomicOr(err, 1);
        uint64_t k0 = sent, k1 = sent;
        if (!bad && a != b) {
            k0 = ((uint64_t)a << bits) | (uint64_t)b;
            k1 = ((uint64_t)b << bits) | (uint64_t)a;
        }
        keys[2 * e] = k0;
        keys[2 * e + 1] = k1;
        vals[2 * e] = (uint32_t)e;
        vals[2 * e + 1] = (uint32_t)e;
    }
}

__global__ void k_lap_heads(const uint64_t* __restrict__ keys, int64_t len, uint64_t sent,
                            uint8_t* __restrict__ head) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = keys[i];
        head[i] = (k != sent) && (i == 0 || keys[i - 1] != k);
    }
}

__global__ void k_lap_runs(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                           const float* __restrict__ w, int64_t len, const uint8_t* __restrict__ head,
                           const int64_t* __restrict__ run_off, int bits,
                           int32_t* __restrict__ row_of_run, int2* __restrict__ colval,
                           uint8_t* __restrict__ upper) {
    const uint64_t cmask = (1ull << bits) - 1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!head[i]) continue;
        const uint64_t k = keys[i];
        // parallel edges: FP64 sum in input order, rounded once; a coarse graph's hub pair can have
        // thousands, so eight entries are loaded at a time
        double s = (double)w[vals[i]];
        if (i + 1 < len && keys[i + 1] == k)
            for (int64_t t = i + 1;; t += 8) {
                uint64_t kk[8];
                float ww[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int64_t j = min(t + q, len - 1);
                    kk[q] = t + q < len ? keys[j] : ~k;
                    ww[q] = w[vals[j]];
                }
                int q = 0;
#pragma unroll
                for (int b = 0; b < 8; ++b)
                    if (q == b && kk[b] == k) {
                        s += (double)ww[b];
                        q = b + 1;
                    }
                if (q < 8) break;
            }
        const int64_t j = run_off[i];
        const int32_t row = (int32_t)(k >> bits), col = (int32_t)(k & cmask);
        row_of_run[j] = row;
        colval[j] = make_int2(col, __float_as_int((float)s));
        upper[j] = row < col;
    }
}

__global__ void k_lap_rowptr(const int32_t* __restrict__ row_of_run, int64_t nnz, int32_t n,
                             int32_t* __restrict__ row_ptr) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j <= nnz;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t prev = j > 0 ? row_of_run[j - 1] : -1;
        const int32_t cur = j < nnz ? row_of_run[j] : n;
        for (int32_t r = prev + 1; r <= cur; ++r) row_ptr[r] = (int32_t)j;
    }
}

__global__ void k_lap_upper(const int2* __restrict__ colval, const int32_t* __restrict__ row_of_run,
                            const uint8_t* __restrict__ upper, const int64_t* __restrict__ up_off,
                            int64_t nnz, int32_t* __restrict__ eu, int32_t* __restrict__ ev,
                            float* __restrict__ ew, int32_t* __restrict__ eid) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nnz;
         j += (int64_t)gridDim.x * blockDim.x) {
        if (!upper[j]) continue;
        const int64_t e = up_off[j];
        const int2 cv = colval[j];
        eu[e] = row_of_run[j];
        ev[e] = cv.x;
        ew[e] = __int_as_float(cv.y);
        eid[j] = (int32_t)e;
    }
}

__global__ void k_lap_lower(const int2* __restrict__ colval, const int32_t* __restrict__ row_of_run,
                            const uint8_t* __restrict__ upper, const int32_t* __restrict__ row_ptr,
                            int64_t nnz, int32_t* __restrict__ eid) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nnz;
         j += (int64_t)gridDim.x * blockDim.x) {
        if (upper[j]) continue;
        const int32_t r = row_of_run[j], c = colval[j].x;  // entry (r, c), c < r: mirror (c, r)
        int32_t lo = row_ptr[c], hi = row_ptr[c + 1];
        while (lo < hi) {
            const int32_t mid = (lo + hi) >> 1;
            if (colval[mid].x < r) lo = mid + 1; else hi = mid;
        }
        eid[j] = eid[lo];
    }
}

// Degrees of the rows of at most hmax entries (longer rows: k_lap_deg_heavy): FP64 sum in column order, one thread a row.
__global__ void k_lap_deg(const int32_t* __restrict__ row_ptr, const int2* __restrict__ colval,
                          int32_t n, int32_t hmax, double* __restrict__ deg, double* __restrict__ invdeg) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = row_ptr[p], b = row_ptr[p + 1];
        if (b - a > hmax) continue;
        double s = 0.0;
        for (int32_t j = a; j < b; ++j) s += (double)__int_as_float(colval[j].y);
        deg[p] = s;
        invdeg[p] = s > 0.0 ? 1.0 / s : 0.0;
    }
}

// Whether FP64 sums of cnt FP32 weights whose exponent fields span [lo, hi] are exact in any order:
// every partial sum is a multiple of the smallest weight's unit below 2^53 of them.
__device__ __forceinline__ bool sums_exact(int lo, int hi, int cnt) {
    const int lg = cnt > 1 ? 32 - __clz(cnt - 1) : 0;
    return 24 + (hi - lo) + lg <= 53;
}
__device__ __forceinline__ int exponent_of(float w) { return max(1, (int)((__float_as_uint(w) >> 23) & 0xffu)); }

// A weight widened without the FP64 pipe (dot64.cuh), which the additions need.
__device__ __forceinline__ double widen_weight(float w) { return is_normal32(w) ? widen_normal(w) : (double)w; }

// FP64 sum of a row's weights in column order by one warp, 32 entries at a time. Where all of them are multiples of
// the unit of the sum so far and the new sum stays in its binade, no addition rounds, whatever the order: the lanes
// add them as a tree. Else each lane's weight is added in turn. (An FP64 addition takes a warp about 75 clocks, so
// a chain of them is what bounds this: a row of 30,000 entries took 1.2 ms in turn, one thread that loads and
// widens as it adds 2.0 ms.) A tail of zeros changes no sum of positive weights.
__device__ __forceinline__ double ordered_degree(const int2* __restrict__ row, int32_t len) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    float next = lane < len ? __int_as_float(row[lane].y) : 0.f;
    for (int32_t j0 = 0; j0 < len; j0 += 32) {
        const int lo = __reduce_min_sync(0xffffffffu, j0 + lane < len ? exponent_of(next) : 255);
        const double w = widen_weight(next);
        const int32_t j = j0 + 32 + lane;
        next = j < len ? __int_as_float(row[j].y) : 0.f;
        const int es = __double2hiint(s) >> 20;  // s >= 0: its exponent field
        if (lo + 925 >= es) {  // lowest unit 2^(lo - 150) against 2^(es - 1075)
            double t = w;
#pragma unroll
            for (int q = 16; q > 0; q >>= 1) t += __shfl_xor_sync(0xffffffffu, t, q);
            t = s + __shfl_sync(0xffffffffu, t, 0);
            if (__double2hiint(t) >> 20 == es) {
                s = t;
                continue;
            }
        }
#pragma unroll
        for (int q = 0; q < 32; ++q) s += __shfl_sync(0xffffffffu, w, q);
    }
    return s;
}

// Degrees of the listed rows that have more than SFG_HEAVY_ROW entries, one CTA a row: in parallel
// where every order gives the column order's bits, else one warp in order.
__global__ void __launch_bounds__(kBlock) k_lap_deg_heavy(int32_t nh, const int32_t* __restrict__ hrow,
                                                          const int32_t* __restrict__ row_ptr,
                                                          const int2* __restrict__ colval,
                                                          double* __restrict__ deg, double* __restrict__ invdeg) {
    __shared__ int slo, shi;
    __shared__ double ws[kBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int32_t h = blockIdx.x; h < nh; h += gridDim.x) {
        const int32_t p = hrow[h], a = row_ptr[p], b = row_ptr[p + 1];
        if (b - a <= SFG_HEAVY_ROW) continue;
        if (threadIdx.x == 0) {
            slo = 255;
            shi = 0;
        }
        __syncthreads();
        int lo = 255, hi = 0;
        double s = 0.0;
        for (int32_t j = a + threadIdx.x; j < b; j += kBlock) {
            const float w = __int_as_float(colval[j].y);
            lo = min(lo, exponent_of(w));
            hi = max(hi, exponent_of(w));
            s += (double)w;
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
        if (lane == 0) {
            atomicMin(&slo, lo);
            atomicMax(&shi, hi);
            ws[warp] = s;
        }
        __syncthreads();
        const bool exact = sums_exact(slo, shi, b - a);
        if (!exact && warp == 0) s = ordered_degree(colval + a, b - a);
        if (threadIdx.x == 0) {
            if (exact) {
                s = 0.0;
                for (int q = 0; q < kBlock / 32; ++q) s += ws[q];
            }
            deg[p] = s;
            invdeg[p] = s > 0.0 ? 1.0 / s : 0.0;
        }
        __syncthreads();
    }
}

__global__ void k_lap_f2c(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                          int64_t len, uint64_t sent, const int64_t* __restrict__ run_off,
                          const uint8_t* __restrict__ upper, const int64_t* __restrict__ up_off,
                          int32_t* __restrict__ f2c) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (keys[i] == sent) continue;
        const int64_t j = run_off[i + 1] - 1;  // run holding position i
        if (upper[j]) f2c[vals[i]] = (int32_t)up_off[j];
    }
}

// ---- canonical form by rows -------------------------------------------------------------------
// What bounds it: 4-byte and 8-byte accesses at random rows (counting, placing, mirrors), so the
// passes are few: count, place, sort rows, index. Rows are sorted where their entries fit on chip: up
// to kRowSmall entries, four rows a warp, and up to kRowWarp, one row a warp, each entry ranked
// against its row in shared memory (quadratic, but no barrier but the warp's); up to kRowMid, kRowBig
// and kRowCap entries, one CTA of 128, 256 or 1,024 threads a row, bitonic (three classes, because a
// CTA's shared memory is its class's largest row: rows of 257-4,096 entries in one class of 48 KB took
// 302 us on the Chung-Lu graph below, about 270 in two). The keys (column, input position) are unique, so the
// order does not depend on the order in which atomics placed them. Measured against the radix path,
// which moves 24 bytes an entry for each of 5-6 digits (GB300, kernels of one build): 2^20-node
// Chung-Lu graph (15.7M entries) 2.54 -> 1.75 ms, 128^3 grid (12.5M entries) 1.47 -> 0.57 ms. What is
// left of the first is the 390 us of counting (atomics on random rows) and 346 us of placing.
constexpr int kRowSmall = 32, kRowWarp = 256, kRowMid = 1024, kRowBig = 4096, kRowCap = 16384;

// Words the build reads back: input error, rows of the five larger classes, raw entries of the longest class, merged
// rows over SFG_HEAVY_ROW, raw entries, merged entries, canonical edges; rows left to k_deg_ordered, of up to
// kRowWarp entries and longer; summed |u - v|.
enum { kWErr, kWWarp, kWMid, kWBig, kWLarge, kWLong, kWLongRaw, kWHeavy, kWRaw, kWNnz, kWEdges, kWDegShort, kWDegLong, kWReach, kWCount };

// Raw row lengths and each entry's place within its row (slot.x in row u, slot.y in row v; -1 for
// self-loops and bad edges). A warp whose edges all share an endpoint (a hub's edges in a sorted
// list) adds once; MATCH: lanes that share an endpoint always add once (coarse graphs, whose sorted
// lists hold runs of parallel edges and hubs of thousands of entries).
template <bool MATCH>
__global__ void __launch_bounds__(kBlock)
    k_row_count(int32_t n, int64_t m, const int32_t* __restrict__ u, const int32_t* __restrict__ v,
                const float* __restrict__ w, int32_t* __restrict__ cnt, int2* __restrict__ slot,
                unsigned long long* __restrict__ words) {
    constexpr int Q = 4;
    __shared__ unsigned long long s_reach;
    const int lane = threadIdx.x & 31;
    unsigned long long reach = 0;
    if (threadIdx.x == 0) s_reach = 0ull;
    auto place = [&](int32_t r, bool ok) {
        if (MATCH) {
            const unsigned peers = __match_any_sync(0xffffffffu, ok ? r : -1);
            const int first = __ffs(peers) - 1;
            int32_t at = 0;
            if (ok && lane == first) at = atomicAdd(&cnt[r], __popc(peers));
            at = __shfl_sync(0xffffffffu, at, first) + __popc(peers & ((1u << lane) - 1u));
            return ok ? at : -1;
        }
        const int32_t r0 = __shfl_sync(0xffffffffu, r, 0);
        if (__all_sync(0xffffffffu, ok && r == r0)) {
            int32_t at = 0;
            if (lane == 0) at = atomicAdd(&cnt[r], 32);
            return __shfl_sync(0xffffffffu, at, 0) + lane;
        }
        return ok ? atomicAdd(&cnt[r], 1) : -1;
    };
    for (int64_t i0 = (int64_t)blockIdx.x * (kBlock * Q); i0 < m; i0 += (int64_t)gridDim.x * (kBlock * Q)) {
        int32_t a[Q], b[Q];
        bool bad = false;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t e = i0 + q * kBlock + threadIdx.x;
            a[q] = b[q] = -1;
            if (e < m) {
                a[q] = u[e];
                b[q] = v[e];
                const float ww = w[e];
                if (a[q] < 0 || a[q] >= n || b[q] < 0 || b[q] >= n || !isfinite(ww) || !(ww > 0.0f)) {
                    bad = true;
                    a[q] = b[q] = -1;
                }
            }
        }
        if (bad) atomicOr(words + kWErr, 1ull);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t e = i0 + q * kBlock + threadIdx.x;
            const bool ok = a[q] >= 0 && a[q] != b[q];
            const int32_t x = place(a[q], ok), y = place(b[q], ok);
            if (e < m) slot[e] = make_int2(x, y);
            reach += (unsigned)abs(a[q] - b[q]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) reach += __shfl_xor_sync(0xffffffffu, reach, o);
    if (lane == 0 && reach) atomicAdd(&s_reach, reach);
    __syncthreads();
    if (threadIdx.x == 0 && s_reach) atomicAdd(words + kWReach, s_reach);
}

// The rows of the five larger classes (in no particular order) and the raw entries of the longest.
__global__ void k_row_classify(int32_t n, const int32_t* __restrict__ cnt, int32_t* __restrict__ lwarp,
                               int32_t* __restrict__ mid, int32_t* __restrict__ big, int32_t* __restrict__ large,
                               int32_t* __restrict__ longest, unsigned long long* __restrict__ words) {
    for (int64_t r0 = (int64_t)blockIdx.x * kBlock; r0 < n; r0 += (int64_t)gridDim.x * kBlock) {
        const int64_t r = r0 + threadIdx.x;
        const int32_t c = r < n ? cnt[r] : 0;
        const bool w = c > kRowSmall && c <= kRowWarp;
        const unsigned ws = __ballot_sync(0xffffffffu, w);
        if (ws) {
            const int lane = threadIdx.x & 31, first = __ffs(ws) - 1;
            unsigned long long at = 0;
            if (lane == first) at = atomicAdd(words + kWWarp, (unsigned long long)__popc(ws));
            at = __shfl_sync(0xffffffffu, at, first);
            if (w) lwarp[at + __popc(ws & ((1u << lane) - 1u))] = (int32_t)r;
        }
        if (c > kRowWarp) {
            if (c <= kRowMid) mid[atomicAdd(words + kWMid, 1ull)] = (int32_t)r;
            else if (c <= kRowBig) big[atomicAdd(words + kWBig, 1ull)] = (int32_t)r;
            else if (c <= kRowCap) large[atomicAdd(words + kWLarge, 1ull)] = (int32_t)r;
            else {
                longest[atomicAdd(words + kWLong, 1ull)] = (int32_t)r;
                atomicAdd(words + kWLongRaw, (unsigned long long)c);
            }
        }
    }
}

__global__ void __launch_bounds__(kBlock)
    k_row_place(int64_t m, const int32_t* __restrict__ u, const int32_t* __restrict__ v,
                const int2* __restrict__ slot, const int64_t* __restrict__ off, uint64_t* __restrict__ raw) {
    constexpr int Q = 4;  // edges in flight a thread: slot and endpoints, then both offsets, then the stores
    for (int64_t i0 = (int64_t)blockIdx.x * (kBlock * Q) + threadIdx.x; i0 < m; i0 += (int64_t)gridDim.x * (kBlock * Q)) {
        int2 at[Q];
        int32_t a[Q], b[Q];
        int64_t oa[Q], ob[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t e = i0 + q * kBlock;
            at[q] = e < m ? slot[e] : make_int2(-1, -1);
            a[q] = e < m ? u[e] : 0;
            b[q] = e < m ? v[e] : 0;
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            oa[q] = at[q].x >= 0 ? off[a[q]] + at[q].x : -1;
            ob[q] = at[q].x >= 0 ? off[b[q]] + at[q].y : -1;
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const uint32_t e = (uint32_t)(i0 + q * kBlock);
            if (oa[q] < 0) continue;
            raw[oa[q]] = ((uint64_t)(uint32_t)b[q] << 32) | e;
            raw[ob[q]] = ((uint64_t)(uint32_t)a[q] << 32) | e;
        }
    }
}

// Per-row results at the row's raw offset: rcv / re / rrow = merged entries (column, weight), the
// first input position of each and its row (-1 past the row's merged entries); rpos[e] = raw-space
// place of input edge e's entry in its upper row; and the row's merged length, entries above the
// diagonal, degree and its reciprocal.
struct RowOut {
    int2* rcv;
    int32_t* re;
    int32_t* rrow;
    int32_t* rpos;
    int32_t* nnz;
    int32_t* up;
    double* deg;
    double* invdeg;
    int32_t* oshort;  // rows left to k_deg_ordered
    int32_t* olong;
    unsigned long long* words;
};

__device__ __forceinline__ void row_degree(const RowOut& o, int64_t r, double s) {
    o.deg[r] = s;
    o.invdeg[r] = s > 0.0 ? 1.0 / s : 0.0;
}

__device__ __forceinline__ void row_finish(const RowOut& o, int64_t r, int32_t nnz, int32_t up, double s, bool exact) {
    o.nnz[r] = nnz;
    o.up[r] = up;
    if (exact) {
        row_degree(o, r, s);
    } else {
        const bool longer = nnz > kRowWarp;
        (longer ? o.olong : o.oshort)[atomicAdd(o.words + (longer ? kWDegLong : kWDegShort), 1ull)] = (int32_t)r;
    }
    if (nnz > SFG_HEAVY_ROW) atomicAdd(o.words + kWHeavy, 1ull);
}

__device__ __forceinline__ int32_t key_col(uint64_t k) { return (int32_t)(k >> 32); }
__device__ __forceinline__ uint32_t key_pos(uint64_t k) { return (uint32_t)k; }

__device__ __forceinline__ void row_entry(const RowOut& o, int64_t p, int32_t r, uint64_t k, float w) {
    o.rcv[p] = make_int2(key_col(k), __float_as_int(w));
    o.re[p] = (int32_t)key_pos(k);
    o.rrow[p] = r;
}

// FP64 sum over the run of equal columns that starts at sorted position i (end b), input order.
__device__ __forceinline__ float run_weight(const uint64_t* key, const float* sw, int i, int b) {
    const int32_t c = key_col(key[i]);
    double s = (double)sw[i];
    for (int t = i + 1; t < b && key_col(key[t]) == c; ++t) s += (double)sw[t];
    return (float)s;
}

// Four consecutive rows a warp (one or two entries a lane on meshes); rows longer than kRowSmall
// are left to the kernels below. The degrees come last, one lane a row of the CTA's 32: an FP64
// instruction holds the pipe for 16 clocks whether one lane needs it or all (with eight rows a
// warp adding their own degrees the 128^3 grid took 410 us here, bound by that).
constexpr int kRowsPerWarp = 4, kRowWarps = kBlock / 32;
__global__ void __launch_bounds__(kBlock, 5)
    k_rows_small(int32_t n, const int32_t* __restrict__ cnt, const int64_t* __restrict__ off,
                 const uint64_t* __restrict__ raw, const float* __restrict__ w, RowOut o) {
    constexpr int CAP = kRowsPerWarp * kRowSmall, PER = CAP / 32;
    __shared__ uint64_t skey[kRowWarps][CAP];
    __shared__ float ssw[kRowWarps][CAP];
    __shared__ int32_t sstart[kRowWarps][kRowsPerWarp + 1];
    __shared__ unsigned sdup[kRowWarps];
    static_assert(kRowWarps * kRowsPerWarp == 32, "one warp adds the degrees");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t* key = skey[warp];
    float* sw = ssw[warp];
    int32_t* start = sstart[warp];
    const int64_t r0 = ((int64_t)blockIdx.x * kRowWarps + warp) * kRowsPerWarp;
    // lane l < kRowsPerWarp: row r0 + l
    const int64_t rl = r0 + lane;
    const bool have = lane < kRowsPerWarp && rl < n;
    int32_t c = have ? cnt[rl] : 0;
    const int64_t ol = have ? off[rl] : 0;
    const bool longer = c > kRowSmall;
    if (longer) c = 0;
    int32_t inc = c;
#pragma unroll
    for (int d = 1; d < kRowsPerWarp; d <<= 1) {
        const int32_t q = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += q;
    }
    if (lane < kRowsPerWarp) start[lane] = inc - c;
    if (lane == kRowsPerWarp - 1) start[kRowsPerWarp] = inc;
    __syncwarp();
    const int total = start[kRowsPerWarp];
    uint64_t mine[PER];
    float wv[PER];
    int lr[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        if (q * 32 >= total) break;  // warp-uniform
        const int i = q * 32 + lane;
        int l = 0;
#pragma unroll
        for (int s = kRowsPerWarp / 2; s > 0; s >>= 1)
            if (start[l + s] <= i) l += s;
        const int64_t base = __shfl_sync(0xffffffffu, ol, l);
        lr[q] = l;
        mine[q] = ~0ull;
        wv[q] = 0.f;
        if (i < total) {
            mine[q] = raw[base + (i - start[l])];
            key[i] = mine[q];
        }
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        if (q * 32 >= total) break;
        if (q * 32 + lane < total) wv[q] = w[key_pos(mine[q])];
    }
    __syncwarp();
    int to[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        if (q * 32 >= total) break;
        const int a = start[lr[q]], b = start[lr[q] + 1];
        int rank = 0;
        if (q * 32 + lane < total)
            for (int t = a; t < b; ++t) rank += key[t] < mine[q];
        to[q] = a + rank;
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        if (q * 32 >= total) break;
        if (q * 32 + lane < total) {
            key[to[q]] = mine[q];
            sw[to[q]] = wv[q];
        }
    }
    __syncwarp();
    unsigned dups = 0;  // rows of this warp that hold parallel edges
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        if (q * 32 >= total) break;
        const int i = q * 32 + lane;
        if (i < total && i > start[lr[q]] && key_col(key[i - 1]) == key_col(key[i])) dups |= 1u << lr[q];
    }
    dups = __reduce_or_sync(0xffffffffu, dups);
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        if (q * 32 >= total) break;
        const int i = q * 32 + lane;
        const int64_t base = __shfl_sync(0xffffffffu, ol, lr[q]);
        if (i >= total) continue;
        const int a = start[lr[q]], b = start[lr[q] + 1];
        const int32_t r = (int32_t)(r0 + lr[q]);
        const uint64_t k = key[i];
        const int32_t cc = key_col(k);
        int at = i - a;
        bool head = true;
        float ww = sw[i];
        if (dups >> lr[q] & 1u) {  // place among the merged entries: runs started up to here, less one
            at = 0;
            for (int t = a + 1; t <= i; ++t) at += key_col(key[t - 1]) != key_col(key[t]);
            head = i == a || key_col(key[i - 1]) != cc;
            if (head) ww = run_weight(key, sw, i, b);
        }
        if (head) row_entry(o, base + at, r, k, ww);
        if (cc > r) o.rpos[key_pos(k)] = (int32_t)(base + at);
    }
    if (lane == 0) sdup[warp] = dups;
    __syncthreads();
    // degree (FP64, column order), merged length and upper entries
    const int64_t r = (int64_t)blockIdx.x * 32 + lane;
    if (warp != 0 || r >= n || cnt[r] > kRowSmall) return;
    const int w4 = lane / kRowsPerWarp, l4 = lane % kRowsPerWarp;
    const int a = sstart[w4][l4], b = sstart[w4][l4 + 1];
    const bool merge = sdup[w4] >> l4 & 1u;
    key = skey[w4];
    sw = ssw[w4];
    double s = 0.0;
    int32_t nnz = 0, up = 0;
    for (int t = a; t < b;) {
        const int32_t cc = key_col(key[t]);
        float ww = sw[t];
        int e = t + 1;
        if (merge) {
            ww = run_weight(key, sw, t, b);
            while (e < b && key_col(key[e]) == cc) ++e;
        }
        s += (double)ww;
        ++nnz;
        up += cc > (int32_t)r;
        t = e;
    }
    for (int t = nnz; t < b - a; ++t) o.rrow[off[r] + t] = -1;
    row_finish(o, r, nnz, up, s, true);
}

// One warp a listed row of at most kRowWarp raw entries.
__global__ void __launch_bounds__(kBlock)
    k_rows_warp(int32_t nrows, const int32_t* __restrict__ rows, const int32_t* __restrict__ cnt,
                const int64_t* __restrict__ off, const uint64_t* __restrict__ raw,
                const float* __restrict__ w, RowOut o) {
    constexpr int PER = kRowWarp / 32;
    __shared__ __align__(16) uint64_t skey[kRowWarps][kRowWarp];
    __shared__ float ssw[kRowWarps][kRowWarp];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t* key = skey[warp];
    float* sw = ssw[warp];
    for (int32_t h = blockIdx.x * kRowWarps + warp; h < nrows; h += gridDim.x * kRowWarps) {
        const int32_t r = rows[h], d = cnt[r];
        const int64_t base = off[r];
        uint64_t mine[PER];
        float wv[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int i = q * 32 + lane;
            mine[q] = i < d ? raw[base + i] : ~0ull;
            key[i] = mine[q];  // past the end: larger than every key
        }
#pragma unroll
        for (int q = 0; q < PER; ++q) wv[q] = q * 32 + lane < d ? w[key_pos(mine[q])] : 0.f;
        __syncwarp();
        int rank[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) rank[q] = 0;
        for (int t = 0; t < d; t += 2) {  // two keys a load, the same for every lane
            const ulonglong2 kk = *reinterpret_cast<const ulonglong2*>(key + t);
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                if (q * 32 >= d) break;  // warp-uniform
                rank[q] += (int)(kk.x < mine[q]) + (int)(kk.y < mine[q]);
            }
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < PER; ++q)
            if (q * 32 + lane < d) {
                key[rank[q]] = mine[q];
                sw[rank[q]] = wv[q];
            }
        __syncwarp();
        int nnz = 0, up = 0, lo = 255, hi = 0;
        double s = 0.0;
        for (int i0 = 0; i0 < d; i0 += 32) {
            const int i = i0 + lane;
            bool head = false, upper = false;
            uint64_t k = 0;
            if (i < d) {
                k = key[i];
                head = i == 0 || key_col(key[i - 1]) != key_col(k);
                upper = key_col(k) > r;
            }
            const unsigned hb = __ballot_sync(0xffffffffu, head);
            const int at = nnz + __popc(hb & ((2u << lane) - 1u)) - 1;
            if (head) {
                const float ww = run_weight(key, sw, i, d);
                row_entry(o, base + at, r, k, ww);
                const int ex = exponent_of(ww);
                lo = min(lo, ex);
                hi = max(hi, ex);
                s += (double)ww;
            }
            if (upper) o.rpos[key_pos(k)] = (int32_t)(base + at);
            nnz += __popc(hb);
            up += __popc(__ballot_sync(0xffffffffu, head && upper));
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        const bool exact = sums_exact(lo, hi, nnz);
        if (exact) {
#pragma unroll
            for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
        }
        for (int i = nnz + lane; i < d; i += 32) o.rrow[base + i] = -1;
        if (lane == 0) row_finish(o, r, nnz, up, s, exact);
        __syncwarp();  // the next row reuses shared memory
    }
}

// One CTA a listed row of at most CAP raw entries: bitonic sort of the keys in shared memory.
// The degree is the FP64 sum in column order; where every partial sum is exact (sums_exact), any
// order gives the same bits and the CTA adds in parallel, else k_deg_ordered adds in order.
template <int THREADS, int CAP>
__global__ void __launch_bounds__(THREADS)
    k_rows_cta(int32_t nrows, const int32_t* __restrict__ rows, const int32_t* __restrict__ cnt,
               const int64_t* __restrict__ off, const uint64_t* __restrict__ raw,
               const float* __restrict__ w, RowOut o) {
    extern __shared__ __align__(16) unsigned char s_rows[];
    uint64_t* key = reinterpret_cast<uint64_t*>(s_rows);
    float* sw = reinterpret_cast<float*>(key + CAP);
    __shared__ int32_t wsum[THREADS / 32];
    __shared__ double dsum[THREADS / 32];
    __shared__ int32_t smin, smax, scarry, sup;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int32_t h = blockIdx.x; h < nrows; h += gridDim.x) {
        const int32_t r = rows[h], d = cnt[r];
        const int64_t base = off[r];
        int N = 64;
        while (N < d) N <<= 1;  // <= CAP
        for (int i = tid; i < N; i += THREADS) key[i] = i < d ? raw[base + i] : ~0ull;
        if (tid == 0) {
            smin = 255;
            smax = 0;
            scarry = 0;
            sup = 0;
        }
        __syncthreads();
        for (int k = 2; k <= N; k <<= 1)
            for (int j = k >> 1; j > 0;) {
                if (j >= 2) {  // two steps (distances j and j / 2) on four keys in registers
                    const int g = j >> 1;
                    for (int t = tid; t < N / 4; t += THREADS) {
                        const int i = ((t & ~(g - 1)) << 2) | (t & (g - 1));
                        const bool asc = (i & k) == 0;
                        uint64_t x0 = key[i], x1 = key[i + g], x2 = key[i + j], x3 = key[i + j + g];
                        auto order = [&](uint64_t& a, uint64_t& b) {
                            if ((a > b) == asc) {
                                const uint64_t q = a;
                                a = b;
                                b = q;
                            }
                        };
                        order(x0, x2);
                        order(x1, x3);
                        order(x0, x1);
                        order(x2, x3);
                        key[i] = x0;
                        key[i + g] = x1;
                        key[i + j] = x2;
                        key[i + j + g] = x3;
                    }
                    j >>= 2;
                } else {
                    for (int t = tid; t < N / 2; t += THREADS) {
                        const int i = 2 * t;
                        const uint64_t a = key[i], b = key[i + 1];
                        if ((a > b) == ((i & k) == 0)) {
                            key[i] = b;
                            key[i + 1] = a;
                        }
                    }
                    j = 0;
                }
                __syncthreads();
            }
        for (int i = tid; i < d; i += THREADS) sw[i] = w[key_pos(key[i])];
        __syncthreads();
        // merged entries, THREADS positions at a time: place = runs started before
        for (int i0 = 0; i0 < d; i0 += THREADS) {
            const int i = i0 + tid;
            bool head = false, upper = false;
            uint64_t k = 0;
            float ww = 0.f;
            if (i < d) {
                k = key[i];
                head = i == 0 || key_col(key[i - 1]) != key_col(k);
                upper = key_col(k) > r;
                if (head) ww = run_weight(key, sw, i, d);
            }
            const unsigned hb = __ballot_sync(0xffffffffu, head);
            const unsigned ub = __ballot_sync(0xffffffffu, head && upper);
            if (lane == 0) wsum[warp] = __popc(hb);
            __syncthreads();
            int before = scarry;
            for (int q = 0; q < warp; ++q) before += wsum[q];
            const int at = before + __popc(hb & ((2u << lane) - 1u)) - 1;
            if (head) {
                sw[at] = ww;  // at <= i: every run that starts in this stretch has been read
                const int ex = exponent_of(ww);
                atomicMin(&smin, ex);
                atomicMax(&smax, ex);
                row_entry(o, base + at, r, k, ww);
            }
            if (i < d && upper) o.rpos[key_pos(k)] = (int32_t)(base + at);
            if (lane == 0 && ub) atomicAdd(&sup, __popc(ub));
            __syncthreads();
            if (tid == THREADS - 1) scarry = before + __popc(hb);
            __syncthreads();
        }
        const int nnz = scarry;
        for (int i = nnz + tid; i < d; i += THREADS) o.rrow[base + i] = -1;
        double s = 0.0;
        const bool exact = sums_exact(smin, smax, nnz);
        if (exact) {
            for (int i = tid; i < nnz; i += THREADS) s += (double)sw[i];
#pragma unroll
            for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
            if (lane == 0) dsum[warp] = s;
            __syncthreads();
            s = 0.0;
            if (tid == 0)
                for (int q = 0; q < THREADS / 32; ++q) s += dsum[q];
        }
        if (tid == 0) row_finish(o, r, nnz, sup, s, exact);
        __syncthreads();  // the next row reuses shared memory
    }
}

// Degrees that have to be added in column order, once all rows are sorted: a lane a row up to kRowWarp entries (32
// rows share each FP64 instruction), a warp a longer row. Added by one thread of the warp or CTA that sorted the row,
// while the others waited, they made the build of a 2^20-node Chung-Lu graph with weights exp(3 N(0, 1))
// 3,041 us instead of 2,038 (2,783 with the radix sort of all entries and one thread a row).
__global__ void __launch_bounds__(kBlock) k_deg_ordered(const int64_t* __restrict__ off, RowOut o) {
    const int64_t t0 = (int64_t)blockIdx.x * kBlock + threadIdx.x, nt = (int64_t)gridDim.x * kBlock;
    const int64_t shorter = (int64_t)o.words[kWDegShort], longer = (int64_t)o.words[kWDegLong];
    for (int64_t i = t0 / 32; i < longer; i += nt / 32) {
        const int32_t r = o.olong[i];
        const double s = ordered_degree(o.rcv + off[r], o.nnz[r]);
        if ((threadIdx.x & 31) == 0) row_degree(o, r, s);
    }
    for (int64_t i = t0; i < shorter; i += nt) {
        const int32_t r = o.oshort[i], len = o.nnz[r];
        const int2* row = o.rcv + off[r];
        double s = 0.0;
        for (int32_t j0 = 0; j0 < len; j0 += 8) {
            float w[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) w[q] = j0 + q < len ? __int_as_float(row[j0 + q].y) : 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) s += widen_weight(w[q]);
        }
        row_degree(o, r, s);
    }
}

// ---- rows of more than kRowCap raw entries ----
// Their entries are gathered from the raw rows as keys (place in the list of rows, column, input position) and sorted
// by the radix sort, which moves these rows only. While a list with one such row took the sort of all entries,
// after it had been counted by rows, it took as long as or longer than with the sort alone: a 2^25-node random
// graph of 2^28 edges and a row of 20,000 entries 117.5 ms (107.8 with the sort alone, now 72.2), a 2^20-node
// Chung-Lu graph with such a row 2,713 us, now 1,946.
// pb, cb: bits of an input position and of a column; i0: first listed row of this sort.
struct LongRows {
    int32_t i0, cb, pb;
    const int32_t* rows;
    const int64_t* start;  // of each listed row's entries among those of all listed rows
    const int64_t* off;
};

__global__ void k_long_counts(int32_t nrows, const int32_t* __restrict__ rows, const int32_t* __restrict__ cnt,
                              int32_t* __restrict__ len) {
    for (int32_t i = blockIdx.x * kBlock + threadIdx.x; i < nrows; i += gridDim.x * kBlock) len[i] = cnt[rows[i]];
}

__global__ void k_long_gather(int64_t len, int32_t nrows, LongRows a, const uint64_t* __restrict__ raw,
                              uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
    const int64_t s0 = a.start[a.i0];
    for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < len; p += (int64_t)gridDim.x * kBlock) {
        int32_t lo = 0, hi = nrows;  // last row that starts at or before p
        while (hi - lo > 1) {
            const int32_t mid = (lo + hi) >> 1;
            if (a.start[a.i0 + mid] - s0 <= p) lo = mid; else hi = mid;
        }
        const uint64_t k = raw[a.off[a.rows[a.i0 + lo]] + (p - (a.start[a.i0 + lo] - s0))];
        keys[p] = ((uint64_t)lo << (a.cb + a.pb)) | (k >> 32 << a.pb) | (k & 0xffffffffull);
        vals[p] = 0u;
    }
}

__global__ void k_long_heads(int64_t len, int32_t pb, const uint64_t* __restrict__ keys, uint8_t* __restrict__ head) {
    for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < len; p += (int64_t)gridDim.x * kBlock)
        head[p] = p == 0 || keys[p - 1] >> pb != keys[p] >> pb;
}

// Merged entries and the raw places of the upper ones, as the row kernels write them.
__global__ void k_long_write(int64_t len, LongRows a, const uint64_t* __restrict__ keys,
                             const uint8_t* __restrict__ head, const int64_t* __restrict__ run,
                             const float* __restrict__ w, RowOut o) {
    const int64_t s0 = a.start[a.i0];
    const uint64_t pmask = (1ull << a.pb) - 1ull, cmask = (1ull << a.cb) - 1ull;
    for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < len; p += (int64_t)gridDim.x * kBlock) {
        const uint64_t k = keys[p], kc = k >> a.pb;
        const int32_t i = a.i0 + (int32_t)(k >> (a.cb + a.pb)), r = a.rows[i], c = (int32_t)(kc & cmask);
        const int64_t at = a.off[r] + (run[p + 1] - 1 - run[a.start[i] - s0]);
        if (c > r) o.rpos[k & pmask] = (int32_t)at;
        if (!head[p]) continue;
        double s = (double)w[k & pmask];  // input order, eight entries in flight
        for (int64_t t = p + 1; t < len && keys[t] >> a.pb == kc; t += 8) {
            float ww[8];
            int take = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint64_t kk = keys[min(t + q, len - 1)];
                if (t + q < len && kk >> a.pb == kc) take = q + 1;  // the run's entries are consecutive
                ww[q] = w[kk & pmask];
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < take) s += (double)ww[q];
            if (take < 8) break;
        }
        row_entry(o, at, r, ((uint64_t)(uint32_t)c << 32) | (k & pmask), (float)s);
    }
}

// One CTA a row: merged length, upper entries, the degree where it may be added in any order, and the rest of the
// raw row marked unused.
__global__ void __launch_bounds__(kBlock)
    k_long_finish(int32_t nrows, LongRows a, const int32_t* __restrict__ cnt, const int64_t* __restrict__ run,
                  RowOut o) {
    __shared__ int slo, shi;
    __shared__ double ws[kBlock / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int32_t i = a.i0 + blockIdx.x; i < a.i0 + nrows; i += gridDim.x) {
        const int32_t r = a.rows[i], d = cnt[r];
        const int64_t base = a.off[r], b = a.start[i] - a.start[a.i0];
        const int32_t nnz = (int32_t)(run[b + d] - run[b]);
        if (tid == 0) {
            slo = 255;
            shi = 0;
        }
        __syncthreads();
        int lo = 255, hi = 0;
        double s = 0.0;
        for (int32_t j = tid; j < nnz; j += kBlock) {
            const float ww = __int_as_float(o.rcv[base + j].y);
            lo = min(lo, exponent_of(ww));
            hi = max(hi, exponent_of(ww));
            s += (double)ww;
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
        if (lane == 0) {
            atomicMin(&slo, lo);
            atomicMax(&shi, hi);
            ws[warp] = s;
        }
        __syncthreads();
        for (int32_t j = nnz + tid; j < d; j += kBlock) o.rrow[base + j] = -1;
        if (tid == 0) {
            int32_t first = 0, end = nnz;  // first merged entry above the diagonal
            while (first < end) {
                const int32_t mid = (first + end) >> 1;
                if (o.rcv[base + mid].x > r) end = mid; else first = mid + 1;
            }
            s = 0.0;
            for (int q = 0; q < kBlock / 32; ++q) s += ws[q];
            row_finish(o, r, nnz, nnz - first, s, sums_exact(slo, shi, nnz));
        }
        __syncthreads();  // the next row reuses shared memory
    }
}

// row_ptr; D[c] such that an edge whose upper entry sits at raw place p of row c has id p + D[c]; and
// move[r], from a row's raw places to its final ones.
__global__ void k_row_index(int32_t n, const int64_t* __restrict__ off, const int64_t* __restrict__ row_off,
                            const int64_t* __restrict__ up_off, const int32_t* __restrict__ nnz,
                            const int32_t* __restrict__ up, int32_t* __restrict__ row_ptr,
                            int32_t* __restrict__ D, int32_t* __restrict__ move,
                            unsigned long long* __restrict__ words) {
    for (int64_t r = (int64_t)blockIdx.x * kBlock + threadIdx.x; r <= n; r += (int64_t)gridDim.x * kBlock) {
        row_ptr[r] = (int32_t)row_off[r];
        if (r < n) {
            D[r] = (int32_t)(up_off[r] - (int64_t)(nnz[r] - up[r]) - off[r]);
            move[r] = (int32_t)(row_off[r] - off[r]);
        } else {
            words[kWRaw] = (unsigned long long)off[n];
            words[kWNnz] = (unsigned long long)row_off[n];
            words[kWEdges] = (unsigned long long)up_off[n];
        }
    }
}

// Edge ids, the edge list and, where anything was merged or dropped, the entries themselves at their final places
// (else the sorted rows are the CSR rows). An upper entry's id comes from its own place, a lower entry's
// from its mirror's.
__global__ void __launch_bounds__(kBlock)
    k_entries_write(int64_t listed, const unsigned long long* __restrict__ words, const int32_t* __restrict__ rrow, const int2* __restrict__ rcv,
                    const int32_t* __restrict__ re, const int32_t* __restrict__ rpos,
                    const int32_t* __restrict__ D, const int32_t* __restrict__ move, int2* __restrict__ colval,
                    int32_t* __restrict__ eid, int32_t* __restrict__ eu, int32_t* __restrict__ ev,
                    float* __restrict__ ew) {
    constexpr int Q = 4;  // entries in flight a thread
    const int64_t len = (int64_t)words[kWRaw];  // raw places end where the rows do: self-loops were never placed
    const bool moved = (int64_t)words[kWNnz] != listed;
    for (int64_t j0 = (int64_t)blockIdx.x * (kBlock * Q) + threadIdx.x; j0 < len; j0 += (int64_t)gridDim.x * (kBlock * Q)) {
        int32_t r[Q], e[Q], id[Q];
        int2 cv[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t j = j0 + q * kBlock;
            r[q] = j < len ? rrow[j] : -1;
            cv[q] = j < len ? rcv[j] : make_int2(0, 0);
            e[q] = j < len ? re[j] : 0;
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            id[q] = 0;
            if (r[q] < 0) continue;
            const int32_t place = cv[q].x > r[q] ? (int32_t)(j0 + q * kBlock) : rpos[e[q]];
            id[q] = place + D[min(r[q], cv[q].x)];
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if (r[q] < 0) continue;
            int64_t dst = j0 + q * kBlock;
            if (moved) {
                dst += move[r[q]];
                colval[dst] = cv[q];
            }
            eid[dst] = id[q];
            if (cv[q].x > r[q]) {
                eu[id[q]] = r[q];
                ev[id[q]] = cv[q].x;
                ew[id[q]] = __int_as_float(cv[q].y);
            }
        }
    }
}

// Edges that were not placed (self-loops, and edges that an unvalidated list may hold with a weight that is not
// finite, such as merged weights past the FP32 range) belong to no canonical edge.
__global__ void k_row_f2c(int64_t m, const int32_t* __restrict__ u, const int32_t* __restrict__ v,
                          const int2* __restrict__ slot, const int32_t* __restrict__ rpos,
                          const int32_t* __restrict__ D, int32_t* __restrict__ f2c) {
    for (int64_t e = (int64_t)blockIdx.x * kBlock + threadIdx.x; e < m; e += (int64_t)gridDim.x * kBlock)
        f2c[e] = slot[e].x < 0 ? -1 : rpos[e] + D[min(u[e], v[e])];
}

// ---- subgraph ----------------------------------------------------------------------------------
// Kept edges and kept entries as one bit each with a running count per 32-bit word: an item's place
// in the subgraph is its word's count plus the bits below it, so the scans run over 1/32 of the
// items and the ranks of 12.5M entries are 3 MB of L2-resident words instead of 100 MB of 64-bit
// offsets. Bound by reading the entries. On the spanning forest of the 128^3 grid the kernels of one
// subgraph (with its degrees and the list of the other edges) and four host waits took about 0.55 ms of
// an end-to-end call, of which 0.24 ms are gone.
__device__ __forceinline__ int64_t bit_rank(const unsigned* __restrict__ bits, const int64_t* __restrict__ woff,
                                            int64_t i) {
    const int64_t w = i >> 5;
    return woff[w] + __popc(bits[w] & ((1u << (i & 31)) - 1u));
}

// IDS: item i is kept when mask[ids[i]] is set, else when mask[i] is. Whole words of 32 items a warp.
template <bool IDS>
__global__ void k_sub_bits(int64_t count, const int32_t* __restrict__ ids, const uint8_t* __restrict__ mask,
                           unsigned* __restrict__ bits, int32_t* __restrict__ pop) {
    constexpr int Q = 4;
    const int lane = threadIdx.x & 31;
    const int64_t nwords = (count + 31) / 32;
    const int64_t w0 = ((int64_t)blockIdx.x * kBlock + threadIdx.x) >> 5, nw = (int64_t)gridDim.x * (kBlock / 32);
    for (int64_t wb = w0 * Q; wb < nwords; wb += nw * Q) {
        int64_t at[Q];
        bool keep[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int64_t i = (wb + q) * 32 + lane;
            at[q] = i < count ? (IDS ? (int64_t)ids[i] : i) : -1;
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) keep[q] = at[q] >= 0 && mask[at[q]] != 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const unsigned b = __ballot_sync(0xffffffffu, keep[q]);
            if (lane == 0 && wb + q < nwords) {
                bits[wb + q] = b;
                pop[wb + q] = __popc(b);
            }
        }
    }
}

// The kept edges, and (out != NULL) the ids of the others in ascending order.
__global__ void k_sub_edges(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                            const float* __restrict__ ew, const unsigned* __restrict__ bits,
                            const int64_t* __restrict__ woff, int64_t m, int32_t* __restrict__ su,
                            int32_t* __restrict__ sv, float* __restrict__ sw, int32_t* __restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = bit_rank(bits, woff, e);
        if (bits[e >> 5] >> (e & 31) & 1u) {
            su[t] = eu[e]; sv[t] = ev[e]; sw[t] = ew[e];
        } else if (out) {
            out[e - t] = (int32_t)e;
        }
    }
}

__global__ void k_sub_csr(const int2* __restrict__ colval, const int32_t* __restrict__ eid,
                          const unsigned* __restrict__ jbits, const int64_t* __restrict__ jwoff,
                          const unsigned* __restrict__ ebits, const int64_t* __restrict__ ewoff, int64_t nnz,
                          int2* __restrict__ scv, int32_t* __restrict__ seid) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nnz;
         j += (int64_t)gridDim.x * blockDim.x) {
        if (!(jbits[j >> 5] >> (j & 31) & 1u)) continue;
        const int64_t t = bit_rank(jbits, jwoff, j);
        scv[t] = colval[j];
        seid[t] = (int32_t)bit_rank(ebits, ewoff, eid[j]);
    }
}

__global__ void k_sub_rowptr(const int32_t* __restrict__ row_ptr, const unsigned* __restrict__ jbits,
                             const int64_t* __restrict__ jwoff, int64_t nnz, int32_t n,
                             int32_t* __restrict__ srp) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p <= n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = row_ptr[p];
        srp[p] = (int32_t)(j < nnz ? bit_rank(jbits, jwoff, j) : jwoff[(nnz + 31) / 32]);
    }
}

__global__ void k_split_colval(const int2* __restrict__ cv, int64_t nnz, int32_t* __restrict__ col,
                               float* __restrict__ val) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nnz;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int2 x = cv[j];
        if (col) col[j] = x.x;
        if (val) val[j] = __int_as_float(x.y);
    }
}

int bits_for(int32_t n) {
    int b = 1;
    while (b < 31 && (1ll << b) < (int64_t)n) ++b;
    return b;
}

template <typename K>
int grid_of(sfg_ctx* ctx, K kernel, int64_t work) {
    return sfg_grid(ctx, (const void*)kernel, kBlock, 0, work);
}

}  // namespace

void sfg_graph_free(sfg_graph* g) {
    if (!g) return;
    SfgDeviceGuard guard(g->device);
    cudaStream_t s = g->stream;
    void* ptrs[] = {g->eu, g->ev, g->ew, g->row_ptr, g->colval, g->eid, g->deg, g->invdeg,
                    g->gs_color, g->gs_order, g->hv_rows, g->hv_soff, g->hv_seg, g->gh_rows, g->gh_soff, g->gh_seg};
    for (void* p : ptrs)
        if (p) cudaFreeAsync(p, s);
    delete g;
}

// Allocate the arrays of a graph with n nodes and m canonical edges.
sfg_status sfg_alloc_graph(sfg_ctx* ctx, int32_t n, int64_t m, sfg_graph** out) {
    sfg_graph* g = new sfg_graph();
    g->device = ctx->device;
    g->n = n;
    g->m = m;
    g->stream = ctx->stream;
    sfg_status st = SFG_OK;
    auto A = [&](void** p, size_t bytes) {
        if (st == SFG_OK) st = sfg_alloc(ctx, p, bytes > 0 ? bytes : 16);
    };
    A((void**)&g->eu, sizeof(int32_t) * m);
    A((void**)&g->ev, sizeof(int32_t) * m);
    A((void**)&g->ew, sizeof(float) * m);
    A((void**)&g->row_ptr, sizeof(int32_t) * ((size_t)n + 1));
    A((void**)&g->colval, sizeof(int2) * 2 * m);
    A((void**)&g->eid, sizeof(int32_t) * 2 * m);
    A((void**)&g->deg, sizeof(double) * n);
    A((void**)&g->invdeg, sizeof(double) * n);
    if (st != SFG_OK) {
        sfg_graph_free(g);
        return st;
    }
    *out = g;
    return SFG_OK;
}

// Degrees of a graph whose rows are in place, hub rows last: building the sweep's heavy-row lists (here, so that later
// calls, which may be captured into a CUDA graph, never synchronise for them) can wait for the host, and
// the other rows' degrees are queued by then.
static sfg_status row_degrees(sfg_ctx* ctx, sfg_graph* g) {
    if (g->n > 0) {
        k_lap_deg<<<grid_of(ctx, k_lap_deg, g->n), kBlock, 0, ctx->stream>>>(g->row_ptr, g->colval, g->n, SFG_HEAVY_ROW,
                                                                             g->deg, g->invdeg);
        ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_lap_deg");
    }
    SFG_TRY(sfg_heavy_prepare(ctx, g));
    if (g->hv_n > 0) {
        k_lap_deg_heavy<<<std::min(g->hv_n, 8 * ctx->num_sms), kBlock, 0, ctx->stream>>>(g->hv_n, g->hv_rows, g->row_ptr,
                                                                                         g->colval, g->deg, g->invdeg);
        ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_lap_deg_heavy");
    }
    return SFG_OK;
}

// Canonical form by one radix sort of the directed entries: lists whose 2m entries do not fit int32 places, and lists
// whose longest rows hold much of them (build_by_rows).
static sfg_status build_by_sort(sfg_ctx* ctx, int32_t n, int64_t m, const int32_t* u, const int32_t* v,
                                const float* w, bool validate, sfg_graph** out, int32_t* f2c) {
    *out = nullptr;
    const int bits = bits_for(n);
    const uint64_t sent = (bits * 2 >= 64) ? ~0ull : ((1ull << (2 * bits)) - 1);
    const int64_t len = 2 * m;
    Scratch s(ctx);
    uint64_t *keys, *keys2;
    uint32_t *vals, *vals2;
    int* err;
    uint8_t* head;
    int64_t* run_off;
    SFG_TRY(s.get(&keys, len));
    SFG_TRY(s.get(&keys2, len));
    SFG_TRY(s.get(&vals, len));
    SFG_TRY(s.get(&vals2, len));
    SFG_TRY(s.get(&err, 1));
    SFG_TRY(s.get(&head, len));
    SFG_TRY(s.get(&run_off, len + 1));
    SFG_CUDA(ctx, cudaMemsetAsync(err, 0, sizeof(int), ctx->stream));
    if (m > 0) {
        k_lap_expand<<<grid_of(ctx, k_lap_expand, m), kBlock, 0, ctx->stream>>>(
            n, m, u, v, w, bits, sent, keys, vals, err); ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_lap_expand");
    }
    if (validate) {
        int herr = 0;
        SFG_CUDA(ctx, cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        SFG_TRY(sfg_wait(ctx));
        if (herr)
            return sfg_fail(ctx, SFG_EINVAL,
                            "edge list: endpoint outside [0, n) or weight not finite and > 0");
    }
    SFG_TRY(sfg_radix_sort_pairs(ctx, &keys, &vals, &keys2, &vals2, len, 2 * bits));
    int64_t nnz = 0;
    if (len > 0) {
        k_lap_heads<<<grid_of(ctx, k_lap_heads, len), kBlock, 0, ctx->stream>>>(keys, len, sent, head); ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_lap_heads");
        SFG_TRY(sfg_scan_u8(ctx, head, run_off, len));
        SFG_TRY(sfg_read_i64(ctx, run_off + len, &nnz));
    }
    if (nnz >= (1ll << 31)) return sfg_fail(ctx, SFG_EINVAL, "too many edges for int32 CSR");
    int32_t* row_of_run;
    int2* colval_tmp;
    uint8_t* upper;
    int64_t* up_off;
    SFG_TRY(s.get(&row_of_run, nnz));
    SFG_TRY(s.get(&colval_tmp, nnz));
    SFG_TRY(s.get(&upper, nnz));
    SFG_TRY(s.get(&up_off, nnz + 1));
    int64_t mc = 0;
    if (nnz > 0) {
        k_lap_runs<<<grid_of(ctx, k_lap_runs, len), kBlock, 0, ctx->stream>>>(
            keys, vals, w, len, head, run_off, bits, row_of_run, colval_tmp, upper); ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_lap_runs");
        SFG_TRY(sfg_scan_u8(ctx, upper, up_off, nnz));
        SFG_TRY(sfg_read_i64(ctx, up_off + nnz, &mc));
    }
    sfg_graph* g = nullptr;
    SFG_TRY(sfg_alloc_graph(ctx, n, mc, &g));
    if (nnz > 0)
        SFG_CUDA(ctx, cudaMemcpyAsync(g->colval, colval_tmp, sizeof(int2) * nnz,
                                      cudaMemcpyDeviceToDevice, ctx->stream));
    k_lap_rowptr<<<grid_of(ctx, k_lap_rowptr, nnz + 1), kBlock, 0, ctx->stream>>>(row_of_run, nnz,
                                                                                   n, g->row_ptr); ++ctx->launches;
    SFG_LAUNCH_CHECK(ctx, "k_lap_rowptr");
    if (nnz > 0) {
        k_lap_upper<<<grid_of(ctx, k_lap_upper, nnz), kBlock, 0, ctx->stream>>>(
            g->colval, row_of_run, upper, up_off, nnz, g->eu, g->ev, g->ew, g->eid); ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_lap_upper");
        k_lap_lower<<<grid_of(ctx, k_lap_lower, nnz), kBlock, 0, ctx->stream>>>(
            g->colval, row_of_run, upper, g->row_ptr, nnz, g->eid); ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_lap_lower");
    }
    {
        const sfg_status ds = row_degrees(ctx, g);
        if (ds != SFG_OK) {
            sfg_graph_free(g);
            return ds;
        }
    }
    if (f2c && m > 0) {
        SFG_CUDA(ctx, cudaMemsetAsync(f2c, 0xff, sizeof(int32_t) * m, ctx->stream));
        if (nnz > 0) {
            k_lap_f2c<<<grid_of(ctx, k_lap_f2c, len), kBlock, 0, ctx->stream>>>(
                keys, vals, len, sent, run_off, upper, up_off, f2c); ++ctx->launches;
            SFG_LAUNCH_CHECK(ctx, "k_lap_f2c");
        }
    }
    *out = g;
    return SFG_OK;
}

// The rows of more than kRowCap raw entries: count of them in `longest`, total entries. The row's place in the list
// shares the 64-bit key with its column and position, so 64 rows (over a million entries) go in one sort, fewer on the
// largest graphs.
static sfg_status long_rows(sfg_ctx* ctx, int32_t n, int64_t m, int32_t count, int64_t total, const int32_t* longest,
                            const int32_t* cnt, const int64_t* off, const uint64_t* raw, const float* w,
                            const RowOut& o) {
    Scratch s(ctx);
    int32_t* len;
    int64_t *start, *run;
    uint64_t *keys, *keys2;
    uint32_t *vals, *vals2;
    uint8_t* head;
    SFG_TRY(s.get(&len, count));
    SFG_TRY(s.get(&start, (size_t)count + 1));
    k_long_counts<<<grid_of(ctx, k_long_counts, count), kBlock, 0, ctx->stream>>>(count, longest, cnt, len);
    ++ctx->launches;
    SFG_TRY(sfg_scan_i32(ctx, len, start, count));
    LongRows a{0, bits_for(n), 1, longest, start, off};
    while ((1ll << a.pb) < m) ++a.pb;
    const int32_t per = 1 << std::min(64 - a.cb - a.pb, 6);  // cb <= 31 and pb <= 30
    std::vector<int64_t> bounds(1, 0);
    if (count <= per) {
        bounds.push_back(total);
    } else {
        std::vector<int64_t> host((size_t)count + 1);
        SFG_CUDA(ctx, cudaMemcpyAsync(host.data(), start, sizeof(int64_t) * host.size(), cudaMemcpyDeviceToHost,
                                      ctx->stream));
        SFG_TRY(sfg_wait(ctx));
        for (int64_t i = per; i < (int64_t)count + per; i += per) bounds.push_back(host[std::min<int64_t>(i, count)]);
    }
    int64_t most = 0;
    for (size_t q = 1; q < bounds.size(); ++q) most = std::max(most, bounds[q] - bounds[q - 1]);
    SFG_TRY(s.get(&keys, most));
    SFG_TRY(s.get(&keys2, most));
    SFG_TRY(s.get(&vals, most));
    SFG_TRY(s.get(&vals2, most));
    SFG_TRY(s.get(&head, most));
    SFG_TRY(s.get(&run, most + 1));
    for (size_t q = 0; q + 1 < bounds.size(); ++q) {
        a.i0 = (int32_t)q * per;
        const int32_t rows = std::min(per, count - a.i0);
        const int64_t entries = bounds[q + 1] - bounds[q];
        k_long_gather<<<grid_of(ctx, k_long_gather, entries), kBlock, 0, ctx->stream>>>(entries, rows, a, raw, keys, vals);
        SFG_LAUNCH_CHECK(ctx, "k_long_gather");
        SFG_TRY(sfg_radix_sort_pairs(ctx, &keys, &vals, &keys2, &vals2, entries,
                                     a.cb + a.pb + (rows > 1 ? bits_for(rows) : 0)));
        k_long_heads<<<grid_of(ctx, k_long_heads, entries), kBlock, 0, ctx->stream>>>(entries, a.pb, keys, head);
        SFG_TRY(sfg_scan_u8(ctx, head, run, entries));
        k_long_write<<<grid_of(ctx, k_long_write, entries), kBlock, 0, ctx->stream>>>(entries, a, keys, head, run, w, o);
        k_long_finish<<<std::min(rows, 4 * ctx->num_sms), kBlock, 0, ctx->stream>>>(rows, a, cnt, run, o);
        ctx->launches += 4;
        SFG_LAUNCH_CHECK(ctx, "k_long_write");
    }
    return SFG_OK;
}

// Lists of up to so many edges get arrays for all of them before the merged sizes are known (a second wait of the
// host otherwise, 5-15 us of idle GPU); more than a quarter left unused goes back.
constexpr int64_t kEarlyEdges = 1 << 24;

static sfg_status fit_edges(sfg_ctx* ctx, sfg_graph* g, int64_t room, int64_t mc, int64_t entries) {
    if (mc >= room - room / 4) return SFG_OK;
    auto fit = [&](auto** p, int64_t count) -> sfg_status {
        void* q = nullptr;
        SFG_TRY(sfg_alloc(ctx, &q, sizeof(**p) * (size_t)count + 16));
        const cudaError_t e = cudaMemcpyAsync(q, *p, sizeof(**p) * (size_t)count, cudaMemcpyDeviceToDevice, ctx->stream);
        sfg_free(ctx, *p);
        *p = static_cast<std::remove_reference_t<decltype(*p)>>(q);
        return e == cudaSuccess ? SFG_OK : sfg_cuda_fail(ctx, e, "graph arrays");
    };
    SFG_TRY(fit(&g->eu, mc));
    SFG_TRY(fit(&g->ev, mc));
    SFG_TRY(fit(&g->ew, mc));
    SFG_TRY(fit(&g->colval, entries));
    return fit(&g->eid, entries);
}

// Canonical form by rows (see k_row_count). *fits = false (and nothing built) when rows of more than kRowCap raw
// entries hold over a quarter of them: the sort of all entries then moves little more than theirs. (GPU time from the
// list, by rows / by the sort: one row of 500,000 of 6.9M entries 1,590 / 1,800 us, one of 2M of 4M 2,770 / 2,390.)
// Two host waits: the input check with the sizes of the row classes, and the merged sizes (see kEarlyEdges).
static sfg_status build_by_rows(sfg_ctx* ctx, int32_t n, int64_t m, const int32_t* u, const int32_t* v,
                                const float* w, bool validate, sfg_graph** out, int32_t* f2c, bool* fits) {
    *out = nullptr;
    *fits = true;
    const int64_t len = 2 * m;
    Scratch s(ctx);
    int32_t *cnt, *lwarp, *mid, *big, *large, *longest, *re, *rrow, *rpos, *nnz, *up, *D, *move, *oshort, *olong;
    int2 *slot, *rcv;
    uint64_t* raw;
    int64_t *off, *row_off, *up_off;
    unsigned long long* words;
    SFG_TRY(s.get(&cnt, n));
    SFG_TRY(s.get(&lwarp, n));
    SFG_TRY(s.get(&mid, (size_t)(len / kRowWarp) + 1));  // longer rows are at most so many
    SFG_TRY(s.get(&big, (size_t)(len / kRowMid) + 1));
    SFG_TRY(s.get(&large, (size_t)(len / kRowBig) + 1));
    SFG_TRY(s.get(&longest, (size_t)(len / kRowCap) + 1));
    SFG_TRY(s.get(&slot, m));
    SFG_TRY(s.get(&words, kWCount));
    int* hw32 = nullptr;
    SFG_TRY(sfg_host_word(ctx, kSfgHostBuild, &hw32));
    unsigned long long* hw = reinterpret_cast<unsigned long long*>(hw32);
    SFG_CUDA(ctx, cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (size_t)n, ctx->stream));
    SFG_CUDA(ctx, cudaMemsetAsync(words, 0, sizeof(unsigned long long) * kWCount, ctx->stream));
    if (m > 0) {
        auto* count = validate ? k_row_count<false> : k_row_count<true>;
        count<<<grid_of(ctx, count, (m + 3) / 4), kBlock, 0, ctx->stream>>>(n, m, u, v, w, cnt, slot, words);
        k_row_classify<<<grid_of(ctx, k_row_classify, n), kBlock, 0, ctx->stream>>>(n, cnt, lwarp, mid, big, large, longest,
                                                                                        words);
        ctx->launches += 2;
        SFG_LAUNCH_CHECK(ctx, "k_row_count");
    }
    SFG_CUDA(ctx, cudaMemcpyAsync(hw, words, sizeof(unsigned long long) * kWCount, cudaMemcpyDeviceToHost,
                                  ctx->stream));
    SFG_TRY(sfg_wait(ctx));
    if (validate && hw[kWErr])
        return sfg_fail(ctx, SFG_EINVAL,
                        "edge list: endpoint outside [0, n) or weight not finite and > 0");
    const int32_t nwarp = (int32_t)hw[kWWarp], nmid = (int32_t)hw[kWMid], nbig = (int32_t)hw[kWBig], nlarge = (int32_t)hw[kWLarge],
                  nlong = (int32_t)hw[kWLong];
    const int64_t long_raw = (int64_t)hw[kWLongRaw];
    if (long_raw > len / 4) {
        *fits = false;
        return SFG_OK;
    }

    sfg_graph* g = new sfg_graph();
    struct Owner { sfg_graph* g; ~Owner() { sfg_graph_free(g); } } own{g};
    g->device = ctx->device;
    g->n = n;
    g->stream = ctx->stream;
    SFG_TRY(sfg_alloc(ctx, (void**)&g->row_ptr, sizeof(int32_t) * ((size_t)n + 1)));
    SFG_TRY(sfg_alloc(ctx, (void**)&g->deg, sizeof(double) * (size_t)n));
    SFG_TRY(sfg_alloc(ctx, (void**)&g->invdeg, sizeof(double) * (size_t)n));
    SFG_TRY(s.get(&off, (size_t)n + 1));
    SFG_TRY(s.get(&row_off, (size_t)n + 1));
    SFG_TRY(s.get(&up_off, (size_t)n + 1));
    SFG_TRY(s.get(&raw, len));
    SFG_TRY(s.get(&rcv, len));
    SFG_TRY(s.get(&re, len));
    SFG_TRY(s.get(&rrow, len));
    SFG_TRY(s.get(&rpos, m));
    SFG_TRY(s.get(&nnz, n));
    SFG_TRY(s.get(&up, n));
    SFG_TRY(s.get(&D, n));
    SFG_TRY(s.get(&move, n));
    SFG_TRY(sfg_scan_i32(ctx, cnt, off, n));
    if (m > 0) {
        k_row_place<<<grid_of(ctx, k_row_place, (m + 3) / 4), kBlock, 0, ctx->stream>>>(m, u, v, slot, off, raw);
        ++ctx->launches;
    }
    SFG_TRY(s.get(&oshort, (size_t)(len / kRowSmall) + 1));
    SFG_TRY(s.get(&olong, (size_t)(len / kRowWarp) + 1));
    const RowOut ro{rcv, re, rrow, rpos, nnz, up, g->deg, g->invdeg, oshort, olong, words};
    k_rows_small<<<ceil_div_u(n, kRowsPerWarp * kRowWarps), kBlock, 0, ctx->stream>>>(n, cnt, off, raw, w, ro);
    ++ctx->launches;
    if (nwarp > 0) {
        k_rows_warp<<<sfg_grid(ctx, (const void*)k_rows_warp, kBlock, 0, (int64_t)nwarp * 32), kBlock, 0, ctx->stream>>>(
            nwarp, lwarp, cnt, off, raw, w, ro);
        ++ctx->launches;
    }
    auto rows_cta = [&](auto* k, int threads, int cap, int32_t count, const int32_t* list) -> sfg_status {
        const size_t sm = (size_t)cap * (sizeof(uint64_t) + sizeof(float));  // up to 192 KB: opt in once
        const auto key = std::make_tuple((const void*)k, -threads, sm);
        if (ctx->occupancy.find(key) == ctx->occupancy.end()) {
            SFG_CUDA(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
            ctx->occupancy.emplace(key, 1);
        }
        k<<<sfg_grid(ctx, (const void*)k, threads, sm, (int64_t)count * threads), threads, sm, ctx->stream>>>(
            count, list, cnt, off, raw, w, ro);
        ++ctx->launches;
        return SFG_OK;
    };
    if (nmid > 0) SFG_TRY(rows_cta(k_rows_cta<128, kRowMid>, 128, kRowMid, nmid, mid));
    if (nbig > 0) SFG_TRY(rows_cta(k_rows_cta<256, kRowBig>, 256, kRowBig, nbig, big));
    if (nlarge > 0) SFG_TRY(rows_cta(k_rows_cta<1024, kRowCap>, 1024, kRowCap, nlarge, large));
    if (nlong > 0) SFG_TRY(long_rows(ctx, n, m, nlong, long_raw, longest, cnt, off, raw, w, ro));
    if (nwarp + nmid + nbig + nlarge + nlong > 0) {
        k_deg_ordered<<<4 * ctx->num_sms, kBlock, 0, ctx->stream>>>(off, ro);
        ++ctx->launches;
    }
    SFG_LAUNCH_CHECK(ctx, "k_rows");
    SFG_TRY(sfg_scan_i32(ctx, nnz, row_off, n));
    SFG_TRY(sfg_scan_i32(ctx, up, up_off, n));
    k_row_index<<<grid_of(ctx, k_row_index, (int64_t)n + 1), kBlock, 0, ctx->stream>>>(
        n, off, row_off, up_off, nnz, up, g->row_ptr, D, move, words);
    ++ctx->launches;
    SFG_LAUNCH_CHECK(ctx, "k_row_index");
    // A new list gets room for all its entries, so that the host need not wait for the merged sizes before the last
    // kernel can be queued: the one wait left is that for the whole build.
    const bool early = validate && m <= kEarlyEdges;
    int64_t entries = len, mc = m;
    auto read_sizes = [&]() -> sfg_status {
        SFG_CUDA(ctx, cudaMemcpyAsync(hw, words, sizeof(unsigned long long) * kWCount, cudaMemcpyDeviceToHost, ctx->stream));
        SFG_TRY(sfg_wait(ctx));
        entries = (int64_t)hw[kWNnz];
        mc = (int64_t)hw[kWEdges];
        return SFG_OK;
    };
    if (!early) SFG_TRY(read_sizes());
    SFG_TRY(sfg_alloc(ctx, (void**)&g->eu, sizeof(int32_t) * mc + 16));
    SFG_TRY(sfg_alloc(ctx, (void**)&g->ev, sizeof(int32_t) * mc + 16));
    SFG_TRY(sfg_alloc(ctx, (void**)&g->ew, sizeof(float) * mc + 16));
    SFG_TRY(sfg_alloc(ctx, (void**)&g->eid, sizeof(int32_t) * entries + 16));
    int2* moved = nullptr;  // the entries if they are moved
    if (early || entries != len || len == 0) SFG_TRY(s.get(&moved, (size_t)entries + 2));
    if (entries > 0) {
        k_entries_write<<<grid_of(ctx, k_entries_write, (len + 3) / 4), kBlock, 0, ctx->stream>>>(
            len, words, rrow, rcv, re, rpos, D, move, moved, g->eid, g->eu, g->ev, g->ew);
        ++ctx->launches;
    }
    if (f2c && m > 0) {
        k_row_f2c<<<grid_of(ctx, k_row_f2c, m), kBlock, 0, ctx->stream>>>(m, u, v, slot, rpos, D, f2c);
        ++ctx->launches;
    }
    SFG_LAUNCH_CHECK(ctx, "k_entries_write");
    if (early) SFG_TRY(read_sizes());
    g->colval = entries != len || len == 0 ? moved : rcv;
    s.release(g->colval);
    if (early) SFG_TRY(fit_edges(ctx, g, m, mc, entries));
    g->m = mc;
    g->reach = m > 0 ? (double)hw[kWReach] / (double)m : 0.0;
    // the sweep's heavy-row lists are built with the graph, so that later calls (which may be
    // captured into a CUDA graph) never synchronise for them
    if (hw[kWHeavy] == 0) {
        g->hv_nseg = 0;
        g->hv_n = 0;
    }
    SFG_TRY(sfg_heavy_prepare(ctx, g));
    own.g = nullptr;
    *out = g;
    return SFG_OK;
}

sfg_status sfg_build_graph(sfg_ctx* ctx, int32_t n, int64_t m, const int32_t* u, const int32_t* v,
                           const float* w, bool validate, sfg_graph** out, int32_t* f2c) {
    if (n > 0 && m < (1ll << 30) && !ctx->build_sorts) {
        bool fits = false;
        SFG_TRY(build_by_rows(ctx, n, m, u, v, w, validate, out, f2c, &fits));
        if (fits) return SFG_OK;
    }
    return build_by_sort(ctx, n, m, u, v, w, validate, out, f2c);
}

// 36 bytes an edge at most stay unused (2.4 MB); a second wait costs 10 of 65 us.
constexpr int64_t kEarlySubEdges = 1 << 16;

sfg_status sfg_subgraph_impl(sfg_ctx* ctx, const sfg_graph* g, const uint8_t* mask,
                             sfg_graph** out, int32_t** off_ids) {
    *out = nullptr;
    if (off_ids) *off_ids = nullptr;
    const int64_t m = g->m, nnz = 2 * m, ewords = (m + 31) / 32, jwords = (nnz + 31) / 32;
    Scratch s(ctx);
    unsigned *ebits, *jbits;
    int32_t *epop, *jpop;
    int64_t *ewoff, *jwoff;
    SFG_TRY(s.get(&ebits, ewords));
    SFG_TRY(s.get(&jbits, jwords));
    SFG_TRY(s.get(&epop, ewords));
    SFG_TRY(s.get(&jpop, jwords));
    SFG_TRY(s.get(&ewoff, ewords + 1));
    SFG_TRY(s.get(&jwoff, jwords + 1));
    // Small subgraphs get room for all of g's edges, so that the one host wait is that for the whole build.
    const bool early = !off_ids && m <= kEarlySubEdges;
    int64_t ms = early ? m : 0;
    if (m > 0) {
        k_sub_bits<false><<<grid_of(ctx, k_sub_bits<false>, (m + 3) / 4), kBlock, 0, ctx->stream>>>(m, nullptr, mask, ebits, epop);
        SFG_TRY(sfg_scan_i32(ctx, epop, ewoff, ewords));
        k_sub_bits<true><<<grid_of(ctx, k_sub_bits<true>, (nnz + 3) / 4), kBlock, 0, ctx->stream>>>(nnz, g->eid, mask, jbits, jpop);
        SFG_TRY(sfg_scan_i32(ctx, jpop, jwoff, jwords));
        ctx->launches += 2;
        SFG_LAUNCH_CHECK(ctx, "k_sub_bits");
        if (!early) SFG_TRY(sfg_read_i64(ctx, ewoff + ewords, &ms));
    } else {
        SFG_CUDA(ctx, cudaMemsetAsync(jwoff, 0, sizeof(int64_t), ctx->stream));
    }
    sfg_graph* p = nullptr;
    SFG_TRY(sfg_alloc_graph(ctx, g->n, ms, &p));
    struct Owner { sfg_graph* g; ~Owner() { sfg_graph_free(g); } } own{p};
    p->reach = g->reach;
    int32_t* rest = nullptr;
    if (off_ids) SFG_TRY(s.get(&rest, m - ms));
    if (m > 0) {
        k_sub_edges<<<grid_of(ctx, k_sub_edges, m), kBlock, 0, ctx->stream>>>(
            g->eu, g->ev, g->ew, ebits, ewoff, m, p->eu, p->ev, p->ew, rest); ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_sub_edges");
        k_sub_csr<<<grid_of(ctx, k_sub_csr, nnz), kBlock, 0, ctx->stream>>>(
            g->colval, g->eid, jbits, jwoff, ebits, ewoff, nnz, p->colval, p->eid); ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_sub_csr");
    }
    k_sub_rowptr<<<grid_of(ctx, k_sub_rowptr, (int64_t)g->n + 1), kBlock, 0, ctx->stream>>>(
        g->row_ptr, jbits, jwoff, nnz, g->n, p->row_ptr); ++ctx->launches;
    SFG_LAUNCH_CHECK(ctx, "k_sub_rowptr");
    if (g->hv_n == 0) {  // rows only lose entries: no heavy row here either
        p->hv_nseg = 0;
        p->hv_n = 0;
    }
    SFG_TRY(row_degrees(ctx, p));
    if (early && m > 0) SFG_TRY(sfg_read_i64(ctx, ewoff + ewords, &p->m));
    if (off_ids) {
        s.release(rest);
        *off_ids = rest;
    }
    own.g = nullptr;
    *out = p;
    return SFG_OK;
}

// The build's last kernels are still at work when the builders return: no graph leaves the library before
// they have finished.
static sfg_status wait_for_graph(sfg_ctx* ctx, sfg_graph** out) {
    const sfg_status st = sfg_wait(ctx);
    if (st != SFG_OK) {
        sfg_graph_free(*out);
        *out = nullptr;
    }
    return st;
}

extern "C" {

sfg_status sfg_laplacian(sfg_ctx* ctx, int32_t n, int64_t m, const int32_t* u, const int32_t* v,
                         const float* w, sfg_graph** out) {
    if (!ctx || !out) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    *out = nullptr;
    if (n < 1) return sfg_fail(ctx, SFG_EINVAL, "n must be >= 1 (got %d)", n);
    if (m < 0 || m >= (1ll << 31)) return sfg_fail(ctx, SFG_EINVAL, "m out of range");
    if (m > 0) {
        SFG_TRY(sfg_check_dev(ctx, u, "u"));
        SFG_TRY(sfg_check_dev(ctx, v, "v"));
        SFG_TRY(sfg_check_dev(ctx, w, "w"));
    }
    SFG_TRY(sfg_build_graph(ctx, n, m, u, v, w, true, out, nullptr));
    return wait_for_graph(ctx, out);
}

void sfg_graph_destroy(sfg_graph* g) { sfg_graph_free(g); }

sfg_status sfg_graph_info(const sfg_graph* g, int32_t* n_host, int64_t* m_host) {
    if (!g) return SFG_EINVAL;
    if (n_host) *n_host = g->n;
    if (m_host) *m_host = g->m;
    return SFG_OK;
}

sfg_status sfg_graph_edges(sfg_ctx* ctx, const sfg_graph* g, int32_t* u, int32_t* v, float* w) {
    if (!ctx || !g) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    if (g->m == 0) return SFG_OK;
    if (u) SFG_CUDA(ctx, cudaMemcpyAsync(u, g->eu, 4 * g->m, cudaMemcpyDeviceToDevice, ctx->stream));
    if (v) SFG_CUDA(ctx, cudaMemcpyAsync(v, g->ev, 4 * g->m, cudaMemcpyDeviceToDevice, ctx->stream));
    if (w) SFG_CUDA(ctx, cudaMemcpyAsync(w, g->ew, 4 * g->m, cudaMemcpyDeviceToDevice, ctx->stream));
    return SFG_OK;
}

sfg_status sfg_graph_csr(sfg_ctx* ctx, const sfg_graph* g, int32_t* row_ptr, int32_t* col,
                         float* val, int32_t* eid, double* deg) {
    if (!ctx || !g) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    const int64_t nnz = 2 * g->m;
    if (row_ptr)
        SFG_CUDA(ctx, cudaMemcpyAsync(row_ptr, g->row_ptr, 4 * ((size_t)g->n + 1),
                                      cudaMemcpyDeviceToDevice, ctx->stream));
    if (deg)
        SFG_CUDA(ctx, cudaMemcpyAsync(deg, g->deg, 8 * (size_t)g->n, cudaMemcpyDeviceToDevice,
                                      ctx->stream));
    if (nnz == 0) return SFG_OK;
    if (eid)
        SFG_CUDA(ctx, cudaMemcpyAsync(eid, g->eid, 4 * nnz, cudaMemcpyDeviceToDevice, ctx->stream));
    if (col || val) {
        k_split_colval<<<grid_of(ctx, k_split_colval, nnz), kBlock, 0, ctx->stream>>>(g->colval, nnz,
                                                                                      col, val); ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_split_colval");
    }
    return SFG_OK;
}

sfg_status sfg_graph_subgraph(sfg_ctx* ctx, const sfg_graph* g, const uint8_t* mask,
                              sfg_graph** out) {
    if (!ctx || !g || !out) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    *out = nullptr;
    if (g->m > 0) SFG_TRY(sfg_check_dev(ctx, mask, "mask"));
    SFG_TRY(sfg_subgraph_impl(ctx, g, mask, out));
    return wait_for_graph(ctx, out);
}

}  // extern "C"
