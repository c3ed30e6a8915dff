// Maximum-weight spanning forest (the spanning-tree backbone of Sec. 3.1 / 3.4, where the paper
// approximates a low-stretch tree by a maximum spanning tree).
//
// Boruvka rounds under the strict order (weight descending, edge id ascending): every edge key is
// (FP32 weight bits << 32) | ~id, unique and ordered like that order, so the forest is unique and
// equal to Kruskal's. A round: (1) each component takes the largest key among edges leaving it,
// (2) marks that edge and hooks to the component across it, the smaller label of a mutual pair
// staying a root, (3) nodes are relabelled with the roots of the hook forest (flattened by pointer jumping
// first where a path is long). Rounds repeat until no component has an outgoing edge. All rounds run in
// one cooperative launch.
#include "gridbar.cuh"
#include "sfg_internal.cuh"

namespace {

constexpr int kBlock = 256;

__global__ void k_mst_init(int32_t n, int32_t* __restrict__ comp) {
    for (int64_t p = (int64_t)blockIdx.x * kBlock + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * kBlock)
        comp[p] = (int32_t)p;
}

// What bounds a round: a node's largest key leaving its component is a gather of its neighbours'
// labels, 8 + 4 + 4 bytes an entry. An edge inside a component stays inside for good, so a node
// keeps its best edge and looks through its row again only when that edge has become internal, and
// never again once no edge leaves; a component's maximum is compared before the 64-bit atomicMax, so
// most nodes of a large component only read it. Hooking and jumping go over a list of the labels that
// are left, and relabelling climbs the hooks itself, so a round has three phases. Separate round kernels
// that rescanned every row took 1,490 us and 11 host waits on the 128^3 grid and 200 us and 7 waits on a
// 64 x 64 grid.
//
// Items are the rows [0, n), rows longer than SFG_HEAVY_ROW excepted, and then the fixed segments
// of those rows. A warp takes kMstTiles x 32 items at once (the tiles a whole grid apart, so that the hubs
// of a graph numbered by degree spread over the warps), one lane each checking the kept edges. The
// items to look through again go through shared memory: up to kMstLong entries to four 8-lane groups,
// kMstItems at a time, longer ones to the whole warp, four entries a lane in flight. Rows of up to
// kMstSorted entries are looked through once: the first round ranks their entries by key, one lane a
// row, and later rounds only step on while the current entry is internal, one lane a row and kMstAhead
// entries at once (the order is one 64-bit word a row: 4 bits a remaining entry, best first, above a 4-bit
// count). Every step is a chain of dependent loads, so the chains in flight set the time. Kernel time on
// the 128^3 grid and a 64 x 64 grid: every row in 8-lane groups each time 1,220 and 95 us, four tiles in
// flight and label lists 1,080 and 90, short rows stepped 880 and 72, two tiles and five entries ahead 826
// and 64 (one tile: 913 and 61). With hub rows in 8-lane groups a coarsened power-law graph, whose
// consecutive hub rows then shared a warp, took longer than the separate kernels (two-level sparsify of a
// 249,480-node Chung-Lu graph 9.6 ms instead of 6.9).
constexpr int kMstTiles = 2, kMstLong = 32, kMstSorted = 15, kMstAhead = 5;
constexpr int kMstLanes = 8, kMstGroups = 32 / kMstLanes, kMstItems = 4;

// Words of one launch: barrier count, rounds that ran out, edges taken, last pointer-jumping pass with work left,
// lengths of the two label lists.
enum { kMwBar, kMwErr, kMwTree, kMwJump, kMwLabels0, kMwLabels1, kMwCount };

struct MstArgs {
    int32_t n;
    int64_t nseg;
    const int32_t* row_ptr;
    const int4* seg;
    const int2* colval;
    const int32_t* eid;
    const int32_t* eu;
    const int32_t* ev;
    const uint8_t* allow;
    const int32_t* key_id;
    const int32_t* key_inv;
    int32_t* comp;              // written by the kernel from here on
    int32_t* parent;
    unsigned long long* best;   // per component label
    unsigned long long* ckey;   // per item: its kept edge's key and the node across it (-1: none left)
    int32_t* cnbr;
    unsigned long long* order;  // per row: the remaining entries of a short row (0: not a short row)
    int32_t* labels[2];         // labels of the components that still had an edge, this round's and the next's
    uint8_t* mask;
    unsigned long long* words;
    GridWait wait;
};

// Pointer jumping in place: every node climbs up to kHops parents and stores the ancestor it
// reached. Other threads' stores are read as they land: every stored value is an ancestor of its
// node, so any mix of old and new values is a valid forest with the same roots, and a node whose
// ancestors were already shortened climbs further.
constexpr int kHops = 8;
__device__ __forceinline__ bool jump_node(volatile int32_t* par, int64_t r) {  // true: not at a root yet
    int32_t p = par[r];
#pragma unroll 1
    for (int h = 0; h < kHops; ++h) {
        const int32_t pp = par[p];
        if (pp == p) break;
        p = pp;
    }
    par[r] = p;
    return par[p] != p;
}

// Offer a key to a component: the maximum so far is read first (from L2), so that most nodes of a large
// component only read. Folding a warp's offers first (by match and reduce, or along runs of lanes) cost
// more than the atomics it saved on every graph tried.
__device__ __forceinline__ void mst_offer(unsigned long long* best, int32_t c, unsigned long long key) {
    if (key > __ldcg(best + c)) atomicMax(best + c, key);
}

// Leaves the number of a jumping pass that has work left: the word is read first and one lane a warp writes. While
// every thread with work left added its atomic to this one word, the forest of a ring whose weights increase
// along it (one chain of hooks) took 273 us on 65,536 nodes and 1,057 on 2M; so it takes 74 and 457 (separate
// launches 196 and 790).
__device__ __forceinline__ void mst_left(unsigned long long* words, bool left, unsigned long long pass) {
    if (!__any_sync(0xffffffffu, left)) return;
    if ((threadIdx.x & 31) == 0 && *(volatile unsigned long long*)(words + kMwJump) < pass) atomicMax(words + kMwJump, pass);
}

__global__ void __launch_bounds__(kBlock, 4) k_mst(MstArgs A) {
    constexpr int LIST = kMstTiles * 32;
    __shared__ uint8_t s_list[kBlock / 32][LIST];
    __shared__ int32_t s_a[kBlock / 32][LIST], s_b[kBlock / 32][LIST], s_c[kBlock / 32][LIST];
    __shared__ unsigned long long s_rank[kBlock / 32][kMstSorted][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane % kMstLanes, grp = lane / kMstLanes;
    const int64_t t0 = (int64_t)blockIdx.x * kBlock + threadIdx.x, nt = (int64_t)gridDim.x * kBlock;
    const int64_t items = (int64_t)A.n + A.nseg;
    const GridBar bar{reinterpret_cast<unsigned*>(A.words + kMwBar), A.wait};
    unsigned passed = 0;
    for (int64_t p = t0; p < A.n; p += nt) {
        A.comp[p] = (int32_t)p;
        A.best[p] = 0ull;
    }
    if (!grid_barrier(bar, passed)) return;
    unsigned long long tree = 0, jump_pass = 0;
    // each round at least halves the number of components that still have outgoing edges
    for (int round = 0; round < 64; ++round) {
        // (1) the largest key leaving each component
        for (int64_t base = t0 - lane; base < items; base += nt * kMstTiles) {
            int32_t nb[kMstTiles], row[kMstTiles], cp[kMstTiles];
#pragma unroll
            for (int q = 0; q < kMstTiles; ++q) {
                const int64_t i = base + q * nt + lane;
                nb[q] = i < items ? (round == 0 ? 0 : A.cnbr[i]) : -1;
                row[q] = (int32_t)i;
                if (i >= A.n && nb[q] >= 0) row[q] = A.seg[i - A.n].x;
            }
#pragma unroll
            for (int q = 0; q < kMstTiles; ++q) {
                cp[q] = nb[q] >= 0 ? A.comp[row[q]] : -1;
                // the label across the kept edge (round 0: nothing kept, look)
                nb[q] = nb[q] >= 0 ? (round == 0 ? cp[q] : A.comp[nb[q]]) : -1;
            }
            // short rows whose kept entry has become internal: step on
            bool offer[kMstTiles];
            if (round > 0) {
                unsigned long long w[kMstTiles];  // remaining entries after the current one, best first
                int32_t first[kMstTiles], left[kMstTiles], j[kMstTiles];
                bool step[kMstTiles], any = false;
#pragma unroll
                for (int q = 0; q < kMstTiles; ++q) {
                    const int64_t i = base + q * nt + lane;
                    offer[q] = cp[q] >= 0 && nb[q] != cp[q];
                    step[q] = cp[q] >= 0 && !offer[q] && i < A.n;
                    w[q] = step[q] ? A.order[i] : 0ull;
                    first[q] = step[q] ? A.row_ptr[i] : 0;
                    step[q] = w[q] != 0ull;
                    left[q] = (int)(w[q] & 15ull) - 1;
                    w[q] >>= 8;
                    any |= step[q];
                    j[q] = step[q] ? -2 : -1;  // -2: looking, or found nothing
                }
                while (any) {  // kMstAhead entries of every row at once: one turn is two loads deep
                    any = false;
                    int32_t col[kMstTiles][kMstAhead];
#pragma unroll
                    for (int q = 0; q < kMstTiles; ++q)
#pragma unroll
                        for (int d = 0; d < kMstAhead; ++d)
                            col[q][d] = step[q] && d < left[q] ? A.colval[first[q] + (int32_t)((w[q] >> (4 * d)) & 15ull)].x : -1;
#pragma unroll
                    for (int q = 0; q < kMstTiles; ++q)
#pragma unroll
                        for (int d = 0; d < kMstAhead; ++d)
                            if (col[q][d] >= 0) col[q][d] = A.comp[col[q][d]] != cp[q] ? 1 : 0;
#pragma unroll
                    for (int q = 0; q < kMstTiles; ++q)
                        if (step[q]) {
                            int drop = kMstAhead;
#pragma unroll
                            for (int d = kMstAhead - 1; d >= 0; --d)
                                if (col[q][d] != 0) drop = d;  // external (1), or past the last one (-1)
                            w[q] >>= 4 * drop;
                            left[q] -= drop;
                            const bool found = drop < kMstAhead && left[q] > 0;
                            if (found) j[q] = first[q] + (int32_t)(w[q] & 15ull);
                            step[q] = !found && left[q] > 0;
                            any |= step[q];
                        }
                }
#pragma unroll
                for (int q = 0; q < kMstTiles; ++q) {
                    const int64_t i = base + q * nt + lane;
                    if (j[q] >= 0) {
                        const int2 cv = A.colval[j[q]];
                        const int32_t e = A.eid[j[q]];
                        const uint32_t id = A.key_id ? (uint32_t)A.key_id[e] : (uint32_t)e;
                        A.order[i] = (w[q] << 4) | (unsigned long long)left[q];
                        A.cnbr[i] = cv.x;
                        A.ckey[i] = ((unsigned long long)(uint32_t)cv.y << 32) | (unsigned long long)(~id);
                        offer[q] = true;
                    } else if (j[q] == -2) {
                        A.cnbr[i] = -1;  // its last entry is internal
                        cp[q] = -1;
                    }
                }
            }
            int cnt = 0, longs = 0;  // short items from the front of the lists, long ones from the back
#pragma unroll
            for (int q = 0; q < kMstTiles; ++q) {
                const int64_t i = base + q * nt + lane;
                bool need = cp[q] >= 0 && !(round > 0 && offer[q]);
                if (round > 0 && cp[q] >= 0 && offer[q]) mst_offer(A.best, cp[q], A.ckey[i]);
                int32_t a = 0, b = 0;
                if (need) {
                    if (i < A.n) {
                        a = A.row_ptr[i];
                        b = A.row_ptr[i + 1];
                        if (b - a > SFG_HEAVY_ROW) b = a;  // looked through by segments
                    } else {
                        const int4 sg = A.seg[i - A.n];
                        a = sg.y;
                        b = sg.z;
                    }
                }
                if (round == 0) {  // short rows: rank their entries (every allowed entry leaves its node)
                    const bool shortrow = need && i < A.n && b - a <= kMstSorted;
                    const int len = shortrow ? b - a : 0;
                    int live = 0;
                    unsigned long long top = 0ull, word = 0ull;
                    int32_t across = -1;
                    for (int x0 = 0; x0 < len; x0 += 4) {
                        int2 cv[4];
                        int32_t e[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (x0 + u < len) {
                                cv[u] = A.colval[a + x0 + u];
                                e[u] = A.eid[a + x0 + u];
                            }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (x0 + u < len) {
                                unsigned long long key = 0ull;
                                if (!A.allow || A.allow[e[u]]) {
                                    const uint32_t id = A.key_id ? (uint32_t)A.key_id[e[u]] : (uint32_t)e[u];
                                    key = ((unsigned long long)(uint32_t)cv[u].y << 32) | (unsigned long long)(~id);
                                    ++live;
                                    if (key > top) {
                                        top = key;
                                        across = cv[u].x;
                                    }
                                }
                                s_rank[warp][x0 + u][lane] = key;
                            }
                    }
                    for (int x = 0; x < len; ++x) {
                        const unsigned long long key = s_rank[warp][x][lane];
                        if (key == 0ull) continue;
                        int rank = 0;
                        for (int y = 0; y < len; ++y) rank += s_rank[warp][y][lane] > key;
                        word |= (unsigned long long)x << (4 * rank + 4);
                    }
                    if (shortrow) {
                        A.order[i] = live ? word | (unsigned long long)live : 0ull;
                        A.cnbr[i] = across;
                        A.ckey[i] = top;
                        if (top) atomicMax(A.best + cp[q], top);
                        need = false;
                    } else if (need && i < A.n) {
                        A.order[i] = 0ull;
                    }
                    if (!need) a = b = 0;
                }
                const bool big = b - a > kMstLong;
                const unsigned low = (1u << lane) - 1u;
                const unsigned todo = __ballot_sync(0xffffffffu, need && !big), wide = __ballot_sync(0xffffffffu, big);
                if (need) {
                    const int at = big ? LIST - 1 - (longs + __popc(wide & low)) : cnt + __popc(todo & low);
                    s_list[warp][at] = (uint8_t)(q * 32 + lane);
                    s_a[warp][at] = a;
                    s_b[warp][at] = b;
                    s_c[warp][at] = cp[q];
                }
                cnt += __popc(todo);
                longs += __popc(wide);
            }
            __syncwarp();
            for (int k0 = 0; k0 < cnt; k0 += kMstGroups * kMstItems) {
                int32_t ra[kMstItems], rb[kMstItems], rc[kMstItems], across[kMstItems], e[kMstItems];
                int2 cv[kMstItems];
                unsigned long long top[kMstItems];
#pragma unroll
                for (int u = 0; u < kMstItems; ++u) {
                    const int k = k0 + u * kMstGroups + grp;
                    ra[u] = rb[u] = rc[u] = 0;
                    if (k < cnt) {
                        ra[u] = s_a[warp][k];
                        rb[u] = s_b[warp][k];
                        rc[u] = s_c[warp][k];
                    }
                    const int32_t j = ra[u] + sub;
                    cv[u] = j < rb[u] ? A.colval[j] : make_int2(-1, 0);
                    e[u] = j < rb[u] ? A.eid[j] : 0;
                }
#pragma unroll
                for (int u = 0; u < kMstItems; ++u) {
                    top[u] = 0ull;
                    across[u] = -1;
                    for (int32_t j = ra[u] + sub;;) {
                        if (cv[u].x >= 0 && A.comp[cv[u].x] != rc[u] && (!A.allow || A.allow[e[u]])) {
                            const uint32_t id = A.key_id ? (uint32_t)A.key_id[e[u]] : (uint32_t)e[u];
                            const unsigned long long key = ((unsigned long long)(uint32_t)cv[u].y << 32) |
                                                           (unsigned long long)(~id);
                            if (key > top[u]) {
                                top[u] = key;
                                across[u] = cv[u].x;
                            }
                        }
                        j += kMstLanes;
                        if (j >= rb[u]) break;
                        cv[u] = A.colval[j];
                        e[u] = A.eid[j];
                    }
                }
#pragma unroll
                for (int u = 0; u < kMstItems; ++u) {
                    unsigned long long m = top[u];
#pragma unroll
                    for (int o = 1; o < kMstLanes; o <<= 1) {
                        const unsigned long long q = __shfl_xor_sync(0xffffffffu, m, o);
                        m = q > m ? q : m;
                    }
                    const int k = k0 + u * kMstGroups + grp;
                    if (k >= cnt) continue;
                    const int64_t it = base + (s_list[warp][k] >> 5) * nt + (s_list[warp][k] & 31);
                    if (m == 0ull) {
                        if (sub == 0) A.cnbr[it] = -1;
                    } else if (top[u] == m) {  // keys are unique: one lane holds it
                        A.cnbr[it] = across[u];
                        A.ckey[it] = m;
                        mst_offer(A.best, rc[u], m);
                    }
                }
            }
            for (int k = LIST - longs; k < LIST; ++k) {
                const int32_t a = s_a[warp][k], b = s_b[warp][k], c = s_c[warp][k];
                unsigned long long top = 0ull;
                int32_t across = -1;
                for (int32_t j0 = a; j0 < b; j0 += 128) {
                    int2 cv[4];
                    int32_t e[4], other[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int32_t j = j0 + u * 32 + lane;
                        cv[u] = j < b ? A.colval[j] : make_int2(-1, 0);
                        e[u] = j < b ? A.eid[j] : 0;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) other[u] = cv[u].x >= 0 ? A.comp[cv[u].x] : c;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (other[u] == c || (A.allow && !A.allow[e[u]])) continue;
                        const uint32_t id = A.key_id ? (uint32_t)A.key_id[e[u]] : (uint32_t)e[u];
                        const unsigned long long key = ((unsigned long long)(uint32_t)cv[u].y << 32) |
                                                       (unsigned long long)(~id);
                        if (key > top) {
                            top = key;
                            across = cv[u].x;
                        }
                    }
                }
                unsigned long long m = top;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned long long q = __shfl_xor_sync(0xffffffffu, m, o);
                    m = q > m ? q : m;
                }
                const int64_t it = base + (s_list[warp][k] >> 5) * nt + (s_list[warp][k] & 31);
                if (m == 0ull) {
                    if (lane == 0) A.cnbr[it] = -1;
                } else if (top == m) {
                    A.cnbr[it] = across;
                    A.ckey[it] = m;
                    mst_offer(A.best, c, m);
                }
            }
            __syncwarp();
        }
        if (!grid_barrier(bar, passed)) return;
        // (2) hooks across the chosen edges; round 0: every node is a label
        const int32_t* list = A.labels[round & 1];
        const int64_t nlab = round == 0 ? (int64_t)A.n
                                        : (int64_t)*(volatile unsigned long long*)(A.words + kMwLabels0 + (round & 1));
        if (blockIdx.x == 0 && threadIdx.x == 0) A.words[kMwLabels0 + ((round + 1) & 1)] = 0ull;
        unsigned taken = 0;
        for (int64_t i = t0; i < nlab; i += nt) {
            const int32_t r = round == 0 ? (int32_t)i : list[i];
            const unsigned long long k = A.best[r];
            int32_t up = r;
            if (k != 0ull) {
                const uint32_t id = ~(uint32_t)(k & 0xffffffffull);
                const uint32_t e = A.key_inv ? (uint32_t)A.key_inv[id] : id;
                A.mask[e] = 1;
                const int32_t c0 = A.comp[A.eu[e]], c1 = A.comp[A.ev[e]];
                const int32_t other = c0 == r ? c1 : c0;
                if (!(A.best[other] == k && r < other)) {
                    up = other;
                    ++taken;
                }
            }
            A.parent[r] = up;
        }
        taken = __reduce_add_sync(0xffffffffu, taken);
        if (lane == 0 && taken) atomicAdd(A.words + kMwTree, (unsigned long long)taken);
        if (!grid_barrier(bar, passed)) return;
        const unsigned long long now = *(volatile unsigned long long*)(A.words + kMwTree);
        if (now == tree) return;  // no component has an outgoing edge
        tree = now;
        // (3) relabel: every node climbs from its label up to kHops hooks (nothing writes them here); a
        // node that stops short of a root leaves the pass's number, and the hooks are then flattened and
        // the nodes, which hold some ancestor of their label, relabelled once more. The next round's
        // labels are the roots that had an edge in this one.
        ++jump_pass;
        bool left = false;
        for (int64_t p0 = t0; p0 < A.n; p0 += nt * kMstTiles) {
            int32_t c[kMstTiles], up[kMstTiles];
#pragma unroll
            for (int q = 0; q < kMstTiles; ++q) c[q] = p0 + q * nt < A.n ? A.comp[p0 + q * nt] : 0;
#pragma unroll
            for (int q = 0; q < kMstTiles; ++q) up[q] = A.parent[c[q]];
            for (int h = 0; h < kHops; ++h) {
                bool moved = false;
#pragma unroll
                for (int q = 0; q < kMstTiles; ++q)
                    if (up[q] != c[q]) {
                        c[q] = up[q];
                        up[q] = A.parent[c[q]];
                        moved = true;
                    }
                if (!moved) break;
            }
#pragma unroll
            for (int q = 0; q < kMstTiles; ++q)
                if (p0 + q * nt < A.n) {
                    A.comp[p0 + q * nt] = c[q];
                    left |= up[q] != c[q];
                }
        }
        for (int64_t i0 = t0 - lane; i0 < nlab; i0 += nt) {
            const int64_t i = i0 + lane;
            const int32_t r = i < nlab ? (round == 0 ? (int32_t)i : list[i]) : -1;
            const bool stays = r >= 0 && A.parent[r] == r && A.best[r] != 0ull;
            const unsigned b = __ballot_sync(0xffffffffu, stays);
            if (!b) continue;
            unsigned long long at = 0;
            if (lane == __ffs(b) - 1) at = atomicAdd(A.words + kMwLabels0 + ((round + 1) & 1), (unsigned long long)__popc(b));
            at = __shfl_sync(0xffffffffu, at, __ffs(b) - 1);
            if (stays) {
                A.labels[(round + 1) & 1][at + __popc(b & ((1u << lane) - 1u))] = r;
                A.best[r] = 0ull;
            }
        }
        mst_left(A.words, left, jump_pass);
        if (!grid_barrier(bar, passed)) return;
        if (*(volatile unsigned long long*)(A.words + kMwJump) < jump_pass) continue;
        for (;;) {
            ++jump_pass;
            left = false;
            for (int64_t i = t0; i < nlab; i += nt) left |= jump_node(A.parent, round == 0 ? i : (int64_t)list[i]);
            mst_left(A.words, left, jump_pass);
            if (!grid_barrier(bar, passed)) return;
            if (*(volatile unsigned long long*)(A.words + kMwJump) < jump_pass) break;
        }
        for (int64_t p = t0; p < A.n; p += nt) A.comp[p] = A.parent[A.comp[p]];
        if (!grid_barrier(bar, passed)) return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(reinterpret_cast<int*>(A.words + kMwErr), 1);
}

// One jumping pass over a forest of all nodes (roots point to themselves); flag set while some node
// does not point at a root yet.
__global__ void k_jump_inplace(int32_t n, int32_t* parent, int* __restrict__ flag) {
    for (int64_t r = (int64_t)blockIdx.x * kBlock + threadIdx.x; r < n; r += (int64_t)gridDim.x * kBlock)
        if (jump_node(parent, r)) *flag = 1;
}

__global__ void k_count_u8(int64_t m, const uint8_t* __restrict__ mask,
                           unsigned long long* __restrict__ cnt) {
    unsigned long long c = 0;
    for (int64_t e = (int64_t)blockIdx.x * kBlock + threadIdx.x; e < m;
         e += (int64_t)gridDim.x * kBlock)
        c += mask[e] != 0;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(cnt, c);
}

}  // namespace

// Flatten a forest given by parent pointers (roots point to themselves) so that every entry
// points at its root: in-place jumping launches until no node moves (one launch when no path is
// longer than kHops; the reach multiplies by about kHops per launch otherwise).
sfg_status sfg_pointer_jump(sfg_ctx* ctx, int32_t n, int32_t* parent) {
    if (n <= 0) return SFG_OK;
    Scratch s(ctx);
    int* flag;
    SFG_TRY(s.get(&flag, 1));
    int* h = nullptr;
    SFG_TRY(sfg_host_word(ctx, 1, &h));
    const int grid = sfg_grid(ctx, (const void*)k_jump_inplace, kBlock, 0, n);
    for (int it = 0; it < 64; ++it) {
        SFG_CUDA(ctx, cudaMemsetAsync(flag, 0, sizeof(int), ctx->stream));
        sfg_tic(ctx, "jump");
        k_jump_inplace<<<grid, kBlock, 0, ctx->stream>>>(n, parent, flag); ++ctx->launches;
        sfg_toc(ctx);
        SFG_LAUNCH_CHECK(ctx, "k_jump_inplace");
        SFG_CUDA(ctx, cudaMemcpyAsync(h, flag, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
        SFG_TRY(sfg_wait(ctx));
        if (!*h) return SFG_OK;
    }
    return sfg_fail(ctx, SFG_ETIMEOUT, "pointer jumping did not converge");
}

sfg_status sfg_count_mask(sfg_ctx* ctx, const uint8_t* mask, int64_t m, int64_t* count_host) {
    Scratch s(ctx);
    unsigned long long* cnt;
    SFG_TRY(s.get(&cnt, 1));
    SFG_CUDA(ctx, cudaMemsetAsync(cnt, 0, 8, ctx->stream));
    if (m > 0) {
        k_count_u8<<<sfg_grid(ctx, (const void*)k_count_u8, kBlock, 0, m), kBlock, 0, ctx->stream>>>(
            m, mask, cnt); ++ctx->launches;
        SFG_LAUNCH_CHECK(ctx, "k_count_u8");
    }
    return sfg_read_i64(ctx, (const int64_t*)cnt, count_host);
}

sfg_status sfg_mst_impl(sfg_ctx* ctx, const sfg_graph* g, const uint8_t* allow, uint8_t* mask,
                        int64_t* n_tree, int32_t* comp_out, const int32_t* key_id,
                        const int32_t* key_inv) {
    const int32_t n = g->n;
    const int64_t m = g->m;
    if (m > 0) SFG_CUDA(ctx, cudaMemsetAsync(mask, 0, m, ctx->stream));
    if (m == 0) {
        if (n_tree) *n_tree = 0;
        if (comp_out && n > 0) {
            k_mst_init<<<sfg_grid(ctx, (const void*)k_mst_init, kBlock, 0, n), kBlock, 0, ctx->stream>>>(
                n, comp_out);
            ++ctx->launches;
            SFG_LAUNCH_CHECK(ctx, "k_mst_init");
        }
        return SFG_OK;
    }
    SFG_TRY(sfg_heavy_prepare(ctx, g));
    const int64_t items = (int64_t)n + (g->hv_n > 0 ? g->hv_nseg : 0);
    Scratch s(ctx);
    MstArgs a{};
    SFG_TRY(s.get(&a.comp, n));
    SFG_TRY(s.get(&a.parent, n));
    SFG_TRY(s.get(&a.best, n));
    SFG_TRY(s.get(&a.ckey, items));
    SFG_TRY(s.get(&a.cnbr, items));
    SFG_TRY(s.get(&a.order, n));
    SFG_TRY(s.get(&a.labels[0], n));
    SFG_TRY(s.get(&a.labels[1], n));
    SFG_TRY(s.get(&a.words, kMwCount));
    int* hw32 = nullptr;
    SFG_TRY(sfg_host_word(ctx, kSfgHostBuild, &hw32));
    unsigned long long* hw = reinterpret_cast<unsigned long long*>(hw32);
    SFG_CUDA(ctx, cudaMemsetAsync(a.words, 0, sizeof(unsigned long long) * kMwCount, ctx->stream));
    a.n = n;
    a.nseg = items - n;
    a.row_ptr = g->row_ptr;
    a.seg = g->hv_seg;
    a.colval = g->colval;
    a.eid = g->eid;
    a.eu = g->eu;
    a.ev = g->ev;
    a.allow = allow;
    a.key_id = key_id;
    a.key_inv = key_inv;
    a.mask = mask;
    a.wait = sfg_grid_wait(ctx, "k_mst");
    void* args[] = {(void*)&a};
    const int grid = sfg_coop_grid(ctx, (const void*)k_mst, kBlock, items);
    sfg_tic(ctx, "mst");
    const cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_mst, dim3(grid), dim3(kBlock), args, 0,
                                                      ctx->stream);
    sfg_toc(ctx);
    if (e != cudaSuccess) return sfg_cuda_fail(ctx, e, "k_mst");
    ++ctx->launches;
    if (comp_out)
        SFG_CUDA(ctx, cudaMemcpyAsync(comp_out, a.comp, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice,
                                      ctx->stream));
    SFG_CUDA(ctx, cudaMemcpyAsync(hw, a.words, sizeof(unsigned long long) * kMwCount, cudaMemcpyDeviceToHost,
                                  ctx->stream));
    SFG_TRY(sfg_wait(ctx));
    if (hw[kMwErr]) return sfg_fail(ctx, SFG_ETIMEOUT, "spanning forest did not converge in 64 rounds");
    if (n_tree) *n_tree = (int64_t)hw[kMwTree];
    return SFG_OK;
}

extern "C" sfg_status sfg_spanning_tree(sfg_ctx* ctx, const sfg_graph* g, const uint8_t* allow,
                                        uint8_t* mask_out, int64_t* n_tree_host) {
    if (!ctx) return SFG_EINVAL;
    SFG_DEVICE(ctx);
    if (!g) return sfg_fail(ctx, SFG_EINVAL, "graph is NULL");
    if (g->m > 0) {
        SFG_TRY(sfg_check_dev(ctx, mask_out, "mask_out"));
        if (allow) SFG_TRY(sfg_check_dev(ctx, allow, "allow"));
    }
    return sfg_mst_impl(ctx, g, allow, mask_out, n_tree_host);
}
