// tree.cu -- Sec. 4.2 step 3a, second half, and the node refresh of the
// list-reusing step: octree over sorted keys and its groups (maximal nodes
// with at most n_g particles), integer node boxes on the key grid, and node
// moments (mass, centre of mass, traceless quadrupole).
//
// Numbering: breadth first, key order within a level (a node's children are
// contiguous and in octant order).  A node at level l splits on the digit of
// level l+1 when it holds more than n_leaf particles and l < 21.
//
// Moments follow one fixed operation order (leaves: particles in order;
// internal nodes: children in octant order) with _rn intrinsics, so they do
// not depend on thread scheduling or on multiply-add contraction.
#include <algorithm>

#include "bh_internal.cuh"
#include "dfloat.cuh"
#include "split32.cuh"

namespace bh {
namespace {

__device__ __forceinline__ uint32_t compact3(uint64_t x) {
    x &= 0x1249249249249249ull;
    x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x ^ (x >> 4)) & 0x100f00f00f00f00full;
    x = (x ^ (x >> 8)) & 0x001f0000ff0000ffull;
    x = (x ^ (x >> 16)) & 0x001f00000000ffffull;
    x = (x ^ (x >> 32)) & 0x00000000001fffffull;
    return (uint32_t)x;
}

// ---- bottom-up passes ------------------------------------------------------
// Boxes and moments take the levels from the deepest up.  A level with many
// nodes is a launch of its own; a run of levels with few is one launch of one
// thread block cluster, whose hardware barrier (arrive with release, wait
// with acquire, which makes the children's records visible) stands between
// two levels: a launch costs 3 to 5 us with its gap, the barrier well under
// one.  The span_nodes of each pass is where the cluster's 2048 threads, on 8
// SMs, start to take longer over a level than a launch of its own (the FP64
// moments early: 8 SMs have 16 FP64 lanes).  A quarter of those values, those and
// four times those: octree with boxes of a 65,537-particle ring 88, 88 and 106 us,
// of 262,144 102, 101 and 108; FP32 moments of 65,537 27.5, 27.2 and 33.7, of 2^20
// 45, 44 and 46; FP64 moments of 4096 131, 139 and 175, of 262,144 239, 242 and 271.  A node's particles or children
// are loaded several at a time before any of them is used.  Measured with the
// leaf pass below: force evaluation on kept lists of a 20,000-particle ring 124
// -> 95 us, evaluation of a 65,537-particle ring 624 -> 540 us, 4 graph steps of
// 64 patches 22.32 -> 22.03 ms; with the next level's fixed fields loaded before
// the barrier 89 -> 82 us, 415 -> 402 us and 21.81 -> 21.74 ms.
constexpr int kSpanBlocks = 8, kSpanThreads = 256;
constexpr int64_t kSpanBoxes = 4096, kSpanMoments32 = 4096, kSpanMoments64 = 256;

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// node(k, pre(k)) for every node k of the levels hi, hi - 1, ..., lo (first
// nodes in lvl); hi > lo only in a one-cluster launch.  pre loads what does not
// depend on the level below: the next level's while this one is waited for.
template <class P, class F>
__device__ __forceinline__ void for_levels(const unsigned long long* __restrict__ lvl, int hi, int lo, P pre, F node) {
    while (hi > lo && lvl[hi + 1] == lvl[hi]) --hi;  // (empty levels, below the tree's depth)
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    int64_t ls = (int64_t)lvl[hi], le = (int64_t)lvl[hi + 1], k = ls + tid;
    auto q = pre(min(k, le - 1));
    for (int lev = hi;; --lev) {
        while (k < le) {
            node(k, q);
            k += stride;
            if (k < le) q = pre(k);
        }
        if (lev == lo) break;
        le = ls;
        ls = (int64_t)lvl[lev - 1];
        k = ls + tid;
        q = pre(min(k, le - 1));
        cluster_barrier();
    }
}

// ---- octree ----------------------------------------------------------------
// The sorted keys fix the whole tree at once; no level waits for the one
// above it.  With common(a, b) the levels two keys share (the deepest level
// at which they lie in one cell), c = common(i - 1, i) and the patch's end
// past every cell:
//   particle i is the first of its cell at every level above c;
//   the level-l cell that starts at i holds more than m particles iff
//     common(i, i + m) >= l;
//   so the nodes that begin at i are, if the level-c cell around i splits
//     (more than n_leaf particles), those of levels c + 1 to
//     max(c, min(common(i, i + n_leaf), 20)) + 1, a chain of first children;
//   the deepest of them is a leaf;
//   and the group that begins at i, if there is one, is the highest of them
//     with at most n_g particles (or the leaf).
// One pass counts the nodes per level, the groups and the leaves of each tile
// of particles, a scan over (level, tile) turns the counts into node ids (breadth
// first, key order within a level), a second pass writes the nodes and the
// lists of groups and leaves, and a pass over the nodes links each to its children.  Against
// one counting, scanning and writing round per level, with binary searches
// for the children (each of a top level's a serial chain through memory), and
// a host wait per level for the eager build: a list-constructing evaluation
// of a 65,537-particle ring 1.49 -> 1.00 ms, 4 graph steps of 64 patches 23.2
// -> 22.7 ms, of the 2^26 ring 543.8 -> 542.8 ms.
constexpr int kTreeThreads = 256, kTreeItems = 4, kTreeTile = kTreeThreads * kTreeItems;
constexpr int kRowGroups = kLevels + 1, kRowLeaves = kLevels + 2;
constexpr int kTreeRows = kLevels + 3;  // levels 0..21, the groups, the leaves
static_assert(kTreeItems * (kTreeThreads / 32) == 32, "one lane per (round, warp) when ranks are scanned");

// Levels at which two keys lie in the same cell: the deepest (0..21).
__device__ __forceinline__ int common(uint64_t a, uint64_t b) {
    const uint64_t x = a ^ b;
    return x ? (__clzll((long long)x) - 1) / 3 : kLevels;
}

// Whether the level-c cell that holds particle i has more than m particles
// (patch [ps, pe)), when particle i + m is not in it.  Most answers are no,
// from two keys: neither i + m/2 nor i - m/2 is in the cell either (m + 1
// particles in a row that hold i reach m/2 past it on one side); else the
// cell's first particle decides.
__device__ __forceinline__ bool cell_above(const uint64_t* __restrict__ key, int64_t i, uint64_t ki, int64_t ps,
                                           int64_t pe, int c, int64_t m) {
    const int64_t h = m >> 1;
    if (!(i + h < pe && common(ki, key[i + h]) >= c) && !(i - h >= ps && common(key[i - h], ki) >= c)) return false;
    int64_t lo = max(ps, i - m), b = i;
    if (common(key[lo], ki) >= c) {
        if (lo == i - m) return true;
        b = lo;
    } else {
        while (lo + 1 < b) {
            const int64_t mid = (lo + b) >> 1;
            if (common(key[mid], ki) >= c)
                b = mid;
            else
                lo = mid;
        }
    }
    return b + m < pe && common(key[b], key[b + m]) >= c;
}

// Patch that holds particle i: the last one starting at or before it.
__device__ __forceinline__ int patch_at(const int64_t* __restrict__ off, int np, int64_t i) {
    int q = 0;
    for (int lo = 0, hi = np - 1; lo < hi;) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i)
            lo = q = mid;
        else
            hi = mid - 1;
    }
    return q;
}

// Levels l0..l1 of the nodes that begin at a particle (l0 > kLevels: none) and
// the level lg of the group that does (kNoGroup: none), in 16 bits.
constexpr int kNoGroup = 31;
struct NodeRange {
    int l0 = kLevels + 1, l1 = -1, lg = kNoGroup;
    __device__ __forceinline__ uint16_t code() const { return (uint16_t)(l0 | (l1 & 31) << 5 | lg << 10); }
    __device__ __forceinline__ static NodeRange of(uint16_t v) {
        NodeRange r;
        r.l0 = v & 31;
        r.l1 = r.l0 > kLevels ? -1 : (v >> 5) & 31;
        r.lg = v >> 10;
        return r;
    }
};

// What a particle's node range starts from: its key, its patch [ps, pe), the
// levels it shares with the particle before it (-1: none in the patch) and with
// those n_leaf and n_g on.
struct NodeProbe {
    uint64_t ki;
    int64_t ps, pe;
    int c, d, dg;
};

__device__ __forceinline__ NodeProbe node_probe(const uint64_t* __restrict__ key, int64_t i,
                                                const int64_t* __restrict__ off, int np, int n_leaf, int n_g) {
    NodeProbe v;
    const int q = patch_at(off, np, i);
    v.ps = off[q];
    v.pe = off[q + 1];
    v.ki = key[i];
    const bool b = i > v.ps, l = i + n_leaf < v.pe, g = i + n_g < v.pe;
    const uint64_t kb = key[b ? i - 1 : i], kl = key[l ? i + n_leaf : i], kg = key[g ? i + n_g : i];
    v.c = b ? common(kb, v.ki) : -1;
    v.d = l ? common(v.ki, kl) : -1;
    v.dg = g ? common(v.ki, kg) : -1;
    return v;
}

__device__ __forceinline__ NodeRange node_range(const uint64_t* __restrict__ key, int64_t i, const NodeProbe& v,
                                                int n_leaf, int n_g) {
    NodeRange r;
    if (v.c >= kLevels || (v.c >= 0 && v.d < v.c && !cell_above(key, i, v.ki, v.ps, v.pe, v.c, n_leaf))) return r;
    r.l0 = v.c + 1;
    r.l1 = max(v.c, min(v.d, kLevels - 1)) + 1;
    if (v.dg >= r.l0)
        r.lg = min(v.dg + 1, r.l1);
    else if (v.c < 0 || v.dg >= v.c || cell_above(key, i, v.ki, v.ps, v.pe, v.c, n_g))
        r.lg = r.l0;
    return r;
}

// Each particle's node range, and the nodes per level, and groups, of each
// tile: cnt[row * ntiles + tile].
__global__ void __launch_bounds__(kTreeThreads) k_tree_count(const uint64_t* key, int64_t n,
                                                             const int64_t* off, int np, int n_leaf,
                                                             int n_g, int64_t ntiles, uint16_t* range,
                                                             uint32_t* cnt) {
    launch_wait();
    __shared__ uint32_t h[kTreeRows];
    if (threadIdx.x < kTreeRows) h[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t i0 = (int64_t)blockIdx.x * kTreeTile + threadIdx.x;
    NodeProbe v[kTreeItems];  // (all rounds' loads in flight)
#pragma unroll
    for (int r = 0; r < kTreeItems; ++r)
        v[r] = node_probe(key, min(i0 + r * kTreeThreads, n - 1), off, np, n_leaf, n_g);
#pragma unroll
    for (int r = 0; r < kTreeItems; ++r) {
        const int64_t i = i0 + r * kTreeThreads;
        NodeRange q;
        if (i < n) {
            q = node_range(key, i, v[r], n_leaf, n_g);
            range[i] = q.code();
        }
        const int l0 = __reduce_min_sync(0xffffffffu, q.l0), l1 = __reduce_max_sync(0xffffffffu, q.l1);
        for (int l = l0; l <= l1; ++l) {
            const unsigned m = __ballot_sync(0xffffffffu, l >= q.l0 && l <= q.l1);
            if (lane == 0 && m) atomicAdd(&h[l], (uint32_t)__popc(m));
        }
        const unsigned mg = __ballot_sync(0xffffffffu, q.lg != kNoGroup);
        if (lane == 0 && mg) atomicAdd(&h[kRowGroups], (uint32_t)__popc(mg));
        const unsigned ml = __ballot_sync(0xffffffffu, q.l1 >= 0);
        if (lane == 0 && ml) atomicAdd(&h[kRowLeaves], (uint32_t)__popc(ml));
    }
    __syncthreads();
    if (threadIdx.x < kTreeRows) cnt[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// The level bounds and the node, group and leaf counts from the scanned
// counts: sz words kSzLvl.., kSzNg and kSzNl, cut at the node capacity (overflow flagged).
__global__ void k_tree_sizes(const uint32_t* scan, int64_t ntiles,
                             const unsigned long long* total, unsigned long long cap,
                             unsigned long long* sz, const int* status) {
    launch_wait();
    const int l = threadIdx.x;
    const unsigned long long nodes = scan[(int64_t)kRowGroups * ntiles], leaf0 = scan[(int64_t)kRowLeaves * ntiles];
    if (l < kLevels + 3) {
        const unsigned long long v = l <= kLevels ? (unsigned long long)scan[(int64_t)l * ntiles] : nodes;
        sz[kSzLvl + l] = v < cap ? v : cap;
    }
    if (l == 0) {
        sz[kSzNg] = leaf0 - nodes;
        sz[kSzNl] = *total - leaf0;
        // (keys that a sort which gave up left unsorted make no tree: nothing is built on them)
        const bool stop = nodes > cap || (*status & kStatTimeout);
        sz[kSzOvf] = stop ? kOvfNodes : 0ull;
        sz[kSzNeedNodes] = nodes > cap ? nodes : 0ull;
    }
}

// Nodes (level, begin, first child; end and parent of the roots), groups and
// leaves (by first particle), and the highest node that begins at a particle.
__global__ void __launch_bounds__(kTreeThreads) k_tree_write(
    const uint16_t* range, int64_t n, const int64_t* off, int np, int64_t ntiles,
    const uint32_t* scan, int64_t cap, uint8_t* level,
    uint32_t* begin, uint32_t* end, int32_t* parent,
    int32_t* first_child, uint8_t* nchild, int32_t* groups,
    int32_t* leaves, int32_t* top) {
    launch_wait();
    __shared__ uint32_t base[kTreeRows][32];  // per (round, warp): nodes of the row before it in the tile, then ids
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int t = threadIdx.x; t < kTreeRows * 32; t += kTreeThreads) (&base[0][0])[t] = 0;
    __syncthreads();
    NodeRange q[kTreeItems];
#pragma unroll
    for (int r = 0; r < kTreeItems; ++r) {
        const int64_t i = (int64_t)blockIdx.x * kTreeTile + r * kTreeThreads + threadIdx.x;
        if (i < n) q[r] = NodeRange::of(range[i]);
        const int l0 = __reduce_min_sync(0xffffffffu, q[r].l0), l1 = __reduce_max_sync(0xffffffffu, q[r].l1);
        for (int l = l0; l <= l1; ++l) {
            const unsigned m = __ballot_sync(0xffffffffu, l >= q[r].l0 && l <= q[r].l1);
            if (lane == 0) base[l][r * (kTreeThreads / 32) + w] = __popc(m);
        }
        const unsigned mg = __ballot_sync(0xffffffffu, q[r].lg != kNoGroup);
        if (lane == 0) base[kRowGroups][r * (kTreeThreads / 32) + w] = __popc(mg);
        const unsigned ml = __ballot_sync(0xffffffffu, q[r].l1 >= 0);
        if (lane == 0) base[kRowLeaves][r * (kTreeThreads / 32) + w] = __popc(ml);
    }
    __syncthreads();
    for (int row = w; row < kTreeRows; row += kTreeThreads / 32) {  // counts -> ids
        const uint32_t v = base[row][lane];
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        base[row][lane] = scan[(int64_t)row * ntiles + blockIdx.x] + x - v;
    }
    __syncthreads();
    const uint32_t nodes = scan[(int64_t)kRowGroups * ntiles], leaf0 = scan[(int64_t)kRowLeaves * ntiles];
#pragma unroll
    for (int r = 0; r < kTreeItems; ++r) {
        const int64_t i = (int64_t)blockIdx.x * kTreeTile + r * kTreeThreads + threadIdx.x;
        const int slot = r * (kTreeThreads / 32) + w;
        const int l0 = __reduce_min_sync(0xffffffffu, q[r].l0), l1 = __reduce_max_sync(0xffffffffu, q[r].l1);
        int64_t prev = -1, gnode = -1;
        for (int l = l0; l <= l1; ++l) {
            const bool has = l >= q[r].l0 && l <= q[r].l1;
            const unsigned m = __ballot_sync(0xffffffffu, has);
            if (!has) continue;
            const int64_t id = (int64_t)base[l][slot] + __popc(m & lt);
            if (l == q[r].lg) gnode = id;
            if (l == q[r].l0) top[i] = (int32_t)id;
            if (prev >= 0 && prev < cap) first_child[prev] = (int32_t)id;
            if (id < cap) {
                level[id] = (uint8_t)l;
                begin[id] = (uint32_t)i;
                if (l == 0) {
                    parent[id] = -1;
                    end[id] = (uint32_t)off[patch_at(off, np, i) + 1];
                }
                if (l == q[r].l1) {
                    first_child[id] = -1;
                    nchild[id] = 0;
                }
            }
            prev = id;
        }
        const unsigned mg = __ballot_sync(0xffffffffu, q[r].lg != kNoGroup);
        if (q[r].lg != kNoGroup) groups[(int64_t)base[kRowGroups][slot] + __popc(mg & lt) - nodes] = (int32_t)gnode;
        const unsigned ml = __ballot_sync(0xffffffffu, q[r].l1 >= 0);
        const int64_t lf = (int64_t)base[kRowLeaves][slot] + __popc(ml & lt) - leaf0;
        if (q[r].l1 >= 0 && lf < cap) leaves[lf] = (int32_t)prev;
    }
}

// Children of every node that splits: parent links, child count, and each
// child's end (the next one's begin; the last one's by a search forward).
__global__ void __launch_bounds__(128) k_tree_link(const uint64_t* key, const int64_t* off,
                                                   int np, const unsigned long long* sz,
                                                   const uint8_t* level,
                                                   const uint32_t* begin, uint32_t* end,
                                                   int32_t* parent,
                                                   const int32_t* first_child,
                                                   uint8_t* nchild) {
    launch_wait();
    if (sz[kSzOvf]) return;  // (a device-sized build that outgrew its nodes)
    const int64_t nn = (int64_t)sz[kSzLvl + kLevels + 2];
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nn; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t f = first_child[k];
        if (f < 0) continue;
        const int l = level[k];
        const int64_t lim = min((int64_t)8, (int64_t)sz[kSzLvl + l + 2] - f);  // nodes of level l + 1 from f on
        const uint32_t b = begin[k];
        const int64_t pe = off[patch_at(off, np, b) + 1];
        uint32_t cb[8];
        uint64_t ck[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) cb[t] = t < lim ? begin[f + t] : 0xffffffffu;
#pragma unroll
        for (int t = 0; t < 8; ++t) ck[t] = (int64_t)cb[t] < pe ? key[cb[t]] : 0ull;
        int nch = 0;
        bool in = true;
        uint32_t last = b;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            in = in && (int64_t)cb[t] < pe && common(ck[0], ck[t]) >= l;
            if (in) {
                ++nch;
                parent[f + t] = (int32_t)k;
                if (t > 0) end[f + t - 1] = cb[t];
                last = cb[t];
            }
        }
        nchild[k] = (uint8_t)nch;
        // end of the last child = end of node k
        int64_t lo = last, step = 1;
        while (lo + step < pe && common(ck[0], key[lo + step]) >= l) {
            lo += step;
            step <<= 1;
        }
        int64_t hi = min(lo + step, pe);  // key[lo] is in the node, key[hi] (or the patch's end) is not
        while (lo + 1 < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (common(ck[0], key[mid]) >= l)
                lo = mid;
            else
                hi = mid;
        }
        end[f + nch - 1] = (uint32_t)hi;
    }
}

// Depth-first successor of a node's subtree: the node a pre-order walk visits
// after it when it does not descend into it, which is the highest node that
// begins at the particle past the subtree's last; none (-1) past a patch's
// last particle, where the next patch's root (one of nodes 0..np - 1) or
// nothing begins.
__device__ __forceinline__ int32_t skip_of(uint32_t e, int64_t n, int np, const int32_t* __restrict__ top) {
    if ((int64_t)e >= n) return -1;
    const int32_t t = top[e];
    return t < np ? -1 : t;
}

// Integer tight boxes (grid coordinates recovered from the keys) and the
// packed records the walk reads (WalkNode).
__global__ void __launch_bounds__(kSpanThreads) k_boxes(
    const uint64_t* key, int64_t n, int np, const uint8_t* level,
    const uint32_t* begin, const uint32_t* end, const int32_t* first_child,
    const uint8_t* nchild, const int32_t* top, uint32_t* qlo, uint32_t* qhi,
    WalkNode* wnode, const unsigned long long* lvl, int lev_hi, int lev_lo) {
    launch_wait();
    struct Pre {
        uint32_t b, e;
        int32_t f, skip;
        int nc, lev;
    };
    auto pre = [&](int64_t k) {
        Pre v{begin[k], end[k], first_child[k], 0, nchild[k], level[k]};
        v.skip = skip_of(v.e, n, np, top);
        return v;
    };
    for_levels(lvl, lev_hi, lev_lo, pre, [&](int64_t k, const Pre& v) {
        const uint32_t b = v.b, e = v.e;
        uint32_t lo[3] = {kQMax, kQMax, kQMax}, hi[3] = {0, 0, 0};
        const int nc = v.nc;
        if (nc == 0) {
            for (uint32_t p = b; p < e; p += 8) {
                uint64_t kk[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) kk[u] = key[min(p + u, e - 1u)];  // (a repeated key changes nothing)
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const uint32_t q[3] = {compact3(kk[u] >> 2), compact3(kk[u] >> 1), compact3(kk[u])};
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        lo[a] = min(lo[a], q[a]);
                        hi[a] = max(hi[a], q[a]);
                    }
                }
            }
        } else {
            const int64_t f = v.f;
            uint32_t cl[8][3], ch[8][3];
#pragma unroll
            for (int c = 0; c < 8; ++c)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const int64_t at = 3 * (f + min(c, nc - 1)) + a;  // (a repeated child changes nothing)
                    cl[c][a] = qlo[at];
                    ch[c][a] = qhi[at];
                }
#pragma unroll
            for (int c = 0; c < 8; ++c)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    lo[a] = min(lo[a], cl[c][a]);
                    hi[a] = max(hi[a], ch[c][a]);
                }
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            qlo[3 * k + a] = lo[a];
            qhi[3 * k + a] = hi[a];
        }
        WalkNode w;
        // a leaf carries its first particle and (up to kWalkCntMax - 1) its
        // particle count instead of a first child and the child count
        const uint32_t cnt = nc == 0 ? min(e - b, kWalkCntMax) : (uint32_t)nc;
        w.a = make_uint4(lo[0] | ((uint32_t)v.lev << kLevels) | (nc == 0 ? kWalkLeaf : 0u),
                         lo[1] | (cnt << kLevels), lo[2],
                         (uint32_t)v.skip);
        w.b = make_uint4(hi[0], hi[1], hi[2], nc == 0 ? b : (uint32_t)v.f);
        wnode[k] = w;
    });
}

// Moments of the nodes (children already done).
template <int ORDER>
__global__ void __launch_bounds__(kSpanThreads) k_moments(
    const uint32_t* begin, const uint32_t* end, const int32_t* first_child,
    const uint8_t* nchild, const double* x, const double* y,
    const double* z, const double* m, double* M, double* cx, double* cy, double* cz,
    double* Q, const unsigned long long* lvl, int lev_hi, int lev_lo) {
    launch_wait();
    struct Pre {
        uint32_t b, e;
        int32_t f;
        int nc;
    };
    auto pre = [&](int64_t k) { return Pre{begin[k], end[k], first_child[k], nchild[k]}; };
    for_levels(lvl, lev_hi, lev_lo, pre, [&](int64_t k, const Pre& v) {
        const int nc = v.nc;
        double Mk = 0.0, sx = 0.0, sy = 0.0, sz = 0.0, c0, c1, c2;
        double q[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (nc == 0) {
            const uint32_t b = v.b, e = v.e;
            double px[8], py[8], pz[8], pm[8];
            uint32_t have = b;
            auto load = [&](uint32_t p) {
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const uint32_t i = min(p + u, e - 1u);
                    px[u] = x[i];
                    py[u] = y[i];
                    pz[u] = z[i];
                    pm[u] = m[i];
                }
                have = p;
            };
            load(b);
            const double x0 = px[0], y0 = py[0], z0 = pz[0];
            for (uint32_t p = b; p < e; p += 8) {
                if (p != have) load(p);
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (p + u < e) {
                        const double mi = pm[u];
                        Mk = __dadd_rn(Mk, mi);
                        sx = __dadd_rn(sx, __dmul_rn(mi, px[u]));
                        sy = __dadd_rn(sy, __dmul_rn(mi, py[u]));
                        sz = __dadd_rn(sz, __dmul_rn(mi, pz[u]));
                    }
            }
            if (Mk > 0.0) {
                c0 = __ddiv_rn(sx, Mk);
                c1 = __ddiv_rn(sy, Mk);
                c2 = __ddiv_rn(sz, Mk);
            } else {
                c0 = x0;
                c1 = y0;
                c2 = z0;
            }
            if (ORDER >= 2)
                for (uint32_t p = b; p < e; p += 8) {
                    if (p != have) load(p);
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (p + u < e) {
                            const double mi = pm[u];
                            const double dx = __dsub_rn(px[u], c0), dy = __dsub_rn(py[u], c1),
                                         dz = __dsub_rn(pz[u], c2);
                            const double d2 =
                                __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                            const double tx = __dmul_rn(3.0, dx), ty = __dmul_rn(3.0, dy), tz = __dmul_rn(3.0, dz);
                            q[0] = __dadd_rn(q[0], __dmul_rn(mi, __dsub_rn(__dmul_rn(tx, dx), d2)));
                            q[1] = __dadd_rn(q[1], __dmul_rn(mi, __dsub_rn(__dmul_rn(ty, dy), d2)));
                            q[2] = __dadd_rn(q[2], __dmul_rn(mi, __dsub_rn(__dmul_rn(tz, dz), d2)));
                            q[3] = __dadd_rn(q[3], __dmul_rn(mi, __dmul_rn(tx, dy)));
                            q[4] = __dadd_rn(q[4], __dmul_rn(mi, __dmul_rn(tx, dz)));
                            q[5] = __dadd_rn(q[5], __dmul_rn(mi, __dmul_rn(ty, dz)));
                        }
                }
        } else {
            const int64_t f = v.f;
            for (int c = 0; c < nc; ++c) {
                const double Mc = M[f + c];
                Mk = __dadd_rn(Mk, Mc);
                sx = __dadd_rn(sx, __dmul_rn(Mc, cx[f + c]));
                sy = __dadd_rn(sy, __dmul_rn(Mc, cy[f + c]));
                sz = __dadd_rn(sz, __dmul_rn(Mc, cz[f + c]));
            }
            if (Mk > 0.0) {
                c0 = __ddiv_rn(sx, Mk);
                c1 = __ddiv_rn(sy, Mk);
                c2 = __ddiv_rn(sz, Mk);
            } else {
                c0 = cx[f];
                c1 = cy[f];
                c2 = cz[f];
            }
            if (ORDER >= 2)
                for (int c = 0; c < nc; ++c) {
                    const double Mc = M[f + c];
                    const double dx = __dsub_rn(cx[f + c], c0), dy = __dsub_rn(cy[f + c], c1),
                                 dz = __dsub_rn(cz[f + c], c2);
                    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                    const double tx = __dmul_rn(3.0, dx), ty = __dmul_rn(3.0, dy), tz = __dmul_rn(3.0, dz);
                    const double* qc = Q + 6 * (f + c);
                    q[0] = __dadd_rn(__dadd_rn(q[0], qc[0]), __dmul_rn(Mc, __dsub_rn(__dmul_rn(tx, dx), d2)));
                    q[1] = __dadd_rn(__dadd_rn(q[1], qc[1]), __dmul_rn(Mc, __dsub_rn(__dmul_rn(ty, dy), d2)));
                    q[2] = __dadd_rn(__dadd_rn(q[2], qc[2]), __dmul_rn(Mc, __dsub_rn(__dmul_rn(tz, dz), d2)));
                    q[3] = __dadd_rn(__dadd_rn(q[3], qc[3]), __dmul_rn(Mc, __dmul_rn(tx, dy)));
                    q[4] = __dadd_rn(__dadd_rn(q[4], qc[4]), __dmul_rn(Mc, __dmul_rn(tx, dz)));
                    q[5] = __dadd_rn(__dadd_rn(q[5], qc[5]), __dmul_rn(Mc, __dmul_rn(ty, dz)));
                }
        }
        M[k] = Mk;
        cx[k] = c0;
        cy[k] = c1;
        cz[k] = c2;
#pragma unroll
        for (int a = 0; a < 6; ++a) Q[6 * k + a] = q[a];
    });
}

// Moments for the FP32 force path, all in FP32: offsets from a reference
// point inside the node (its first particle, or its first child's centre)
// are exact hi/lo differences; the centre of mass is kept as an FP32 hi/lo
// pair (reference + offset), mass and traceless quadrupole in FP32.
// Record layout: (c_hi, M), (c_lo, Qxx), (Qxy, Qxz, Qyy, Qyz).
__device__ __forceinline__ float dsub(float ah, float al, float bh, float bl) {
    return __fadd_rn(__fsub_rn(ah, bh), __fsub_rn(al, bl));
}

// A node's record from its mass, reference point, centre offset and quadrupole.
__device__ __forceinline__ void put_moments32(int64_t k, float Mk, df_sum Md, const float (&rh)[3], const float (&rl)[3],
                                              const float (&dc)[3], const float (&q)[6], float4* cell32,
                                              float* mlo) {
    // centre = reference + offset, renormalised into a hi/lo pair
    float ch[3], cl[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float lo = __fadd_rn(rl[a], dc[a]);
        const float hi = __fadd_rn(rh[a], lo);
        ch[a] = hi;
        cl[a] = __fsub_rn(lo, __fsub_rn(hi, rh[a]));
    }
    mlo[k] = __fadd_rn(__fsub_rn(Md.hi, Mk), __fadd_rn(Md.lo, Md.err));
    cell32[3 * k + 0] = make_float4(ch[0], ch[1], ch[2], Mk);
    cell32[3 * k + 1] = make_float4(cl[0], cl[1], cl[2], q[0]);
    cell32[3 * k + 2] = make_float4(q[3], q[4], q[1], q[5]);
}

// The FP32 hi/lo split of the particles and the leaves' moments in one pass:
// a block takes kLeafTile consecutive leaves, whose particles are consecutive
// too; it splits them with coalesced loads, writes the split and keeps it in
// shared memory, from which a thread per leaf sums the moments (more particles
// than fit are read back from memory).  32 B read and 32 B written per particle and
// 52 B per leaf, where a pass of its own re-read the 32 B with a leaf's stride
// between the lanes; bound by issue and the loads' latency (2^22 ring: issue slots
// 68% busy, DRAM at half of its peak).  Split and moments of the 2^24 ring, per
// evaluation: 0.65 -> 0.54 ms.  Room for 640 particles (5 per leaf) lets 9 blocks
// share an SM (768: four steps of that ring +0.1%).
constexpr int kLeafTile = 128, kLeafCap = 640;

template <int ORDER>
__global__ void __launch_bounds__(kLeafTile) k_leaf32(const int32_t* leaves,
                                                      const unsigned long long* dnl,
                                                      const uint32_t* begin,
                                                      const uint32_t* end,
                                                      const double* x, const double* y,
                                                      const double* z, const double* m,
                                                      float4* phi, float4* plo, float4* cell32,
                                                      float* mlo) {
    launch_wait();
    __shared__ float4 sh[kLeafCap], sl[kLeafCap];
    const int64_t nl = (int64_t)*dnl;
    for (int64_t t0 = (int64_t)blockIdx.x * kLeafTile; t0 < nl; t0 += (int64_t)gridDim.x * kLeafTile) {
        const int64_t t1 = min(t0 + kLeafTile, nl);
        const uint32_t p0 = begin[leaves[t0]], p1 = end[leaves[t1 - 1]];
        const bool mine = t0 + threadIdx.x < t1;
        const int64_t k = mine ? leaves[t0 + threadIdx.x] : 0;
        const uint32_t b = mine ? begin[k] : 0u, e = mine ? end[k] : 0u;
        auto put = [&](uint32_t i, const double (&v)[4]) {
            float h[4], l[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) split_f32(v[a], h[a], l[a]);
            const float4 H = make_float4(h[0], h[1], h[2], h[3]), L = make_float4(l[0], l[1], l[2], l[3]);
            phi[i] = H;
            plo[i] = L;
            if (i - p0 < kLeafCap) {
                sh[i - p0] = H;
                sl[i - p0] = L;
            }
        };
        for (uint32_t i = p0 + threadIdx.x; i < p1; i += 2 * kLeafTile) {  // two particles' loads in flight
            const uint32_t j = min(i + kLeafTile, p1 - 1u);
            const double v[4] = {x[i], y[i], z[i], m[i]}, w[4] = {x[j], y[j], z[j], m[j]};
            put(i, v);
            if (i + kLeafTile < p1) put(j, w);
        }
        __syncthreads();
        if (mine) {
            const bool in = e - p0 <= kLeafCap;
            const float4* H = in ? sh : phi + p0;
            const float4* L = in ? sl : plo + p0;
            const uint32_t i0 = b - p0, i1 = e - p0;
            const float4 h0 = H[i0], l0 = L[i0];
            const float rh[3] = {h0.x, h0.y, h0.z}, rl[3] = {l0.x, l0.y, l0.z};
            float Mk = 0.f, s[3] = {0.f, 0.f, 0.f}, q[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            // the mass also as a compensated sum of the (hi + lo) masses: the record
            // keeps Mk, mlo[k] the difference (for the refinement of the FP32 kernel)
            df_sum Md = {0.f, 0.f, 0.f};
            for (uint32_t i = i0; i < i1; ++i) {
                const float4 h = H[i], l = L[i];
                const float d[3] = {dsub(h.x, l.x, rh[0], rl[0]), dsub(h.y, l.y, rh[1], rl[1]),
                                    dsub(h.z, l.z, rh[2], rl[2])};
                Mk += h.w;
                df_accumulate(Md, {h.w, l.w});
#pragma unroll
                for (int a = 0; a < 3; ++a) s[a] = fmaf(h.w, d[a], s[a]);
            }
            const float inv = Mk > 0.f ? 1.f / Mk : 0.f;
            const float dc[3] = {s[0] * inv, s[1] * inv, s[2] * inv};
            if (ORDER >= 2)
                for (uint32_t i = i0; i < i1; ++i) {
                    const float4 h = H[i], l = L[i];
                    const float d[3] = {dsub(h.x, l.x, rh[0], rl[0]) - dc[0], dsub(h.y, l.y, rh[1], rl[1]) - dc[1],
                                        dsub(h.z, l.z, rh[2], rl[2]) - dc[2]};
                    const float d2 = fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2]));
                    const float m3 = 3.f * h.w;
                    q[0] = fmaf(h.w, fmaf(3.f * d[0], d[0], -d2), q[0]);
                    q[1] = fmaf(h.w, fmaf(3.f * d[1], d[1], -d2), q[1]);
                    q[2] = fmaf(h.w, fmaf(3.f * d[2], d[2], -d2), q[2]);
                    q[3] = fmaf(m3 * d[0], d[1], q[3]);
                    q[4] = fmaf(m3 * d[0], d[2], q[4]);
                    q[5] = fmaf(m3 * d[1], d[2], q[5]);
                }
            put_moments32(k, Mk, Md, rh, rl, dc, q, cell32, mlo);
        }
        __syncthreads();
    }
}

// Moments of the inner nodes, from their children's.
template <int ORDER>
__global__ void __launch_bounds__(kSpanThreads) k_moments32(
    const int32_t* first_child, const uint8_t* nchild, float4* cell32, float* mlo,
    const unsigned long long* lvl, int lev_hi, int lev_lo) {
    launch_wait();
    struct Pre {
        int32_t f;
        int nc;
    };
    auto pre = [&](int64_t k) { return Pre{first_child[k], nchild[k]}; };
    for_levels(lvl, lev_hi, lev_lo, pre, [&](int64_t k, const Pre& v) {
        const int nc = v.nc;
        if (nc == 0) return;
        const int64_t f = v.f;
        float4 H[4], L[4], U[4];
        float ml[4];
        auto load = [&](int c0) {  // children c0..c0 + 3 (the last one again past the end)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t j = f + min(c0 + u, nc - 1);
                H[u] = cell32[3 * j];
                L[u] = cell32[3 * j + 1];
                if (ORDER >= 2) U[u] = cell32[3 * j + 2];
                ml[u] = mlo[j];
            }
        };
        load(0);
        const float rh[3] = {H[0].x, H[0].y, H[0].z}, rl[3] = {L[0].x, L[0].y, L[0].z};
        float Mk = 0.f, s[3] = {0.f, 0.f, 0.f}, q[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        df_sum Md = {0.f, 0.f, 0.f};
        for (int c0 = 0; c0 < nc; c0 += 4) {
            if (c0 > 0) load(c0);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (c0 + u < nc) {
                    const float4 h = H[u], l = L[u];
                    const float d[3] = {dsub(h.x, l.x, rh[0], rl[0]), dsub(h.y, l.y, rh[1], rl[1]),
                                        dsub(h.z, l.z, rh[2], rl[2])};
                    Mk += h.w;
                    df_accumulate(Md, {h.w, ml[u]});
#pragma unroll
                    for (int a = 0; a < 3; ++a) s[a] = fmaf(h.w, d[a], s[a]);
                }
        }
        const float inv = Mk > 0.f ? 1.f / Mk : 0.f;
        const float dc[3] = {s[0] * inv, s[1] * inv, s[2] * inv};
        if (ORDER >= 2)
            for (int c0 = 0; c0 < nc; c0 += 4) {
                if (nc > 4) load(c0);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (c0 + u < nc) {
                        const float4 h = H[u], l = L[u], t = U[u];
                        const float D[3] = {dsub(h.x, l.x, rh[0], rl[0]) - dc[0], dsub(h.y, l.y, rh[1], rl[1]) - dc[1],
                                            dsub(h.z, l.z, rh[2], rl[2]) - dc[2]};
                        const float D2 = fmaf(D[0], D[0], fmaf(D[1], D[1], D[2] * D[2]));
                        const float Mc = h.w, m3 = 3.f * Mc;
                        q[0] += l.w + Mc * fmaf(3.f * D[0], D[0], -D2);
                        q[1] += t.z + Mc * fmaf(3.f * D[1], D[1], -D2);
                        q[2] += -(l.w + t.z) + Mc * fmaf(3.f * D[2], D[2], -D2);
                        q[3] += t.x + m3 * D[0] * D[1];
                        q[4] += t.y + m3 * D[0] * D[2];
                        q[5] += t.w + m3 * D[1] * D[2];
                    }
            }
        put_moments32(k, Mk, Md, rh, rl, dc, q, cell32, mlo);
    });
}

// Issue a bottom-up pass over all levels: kern(args..., lvl, hi, lo).  The
// level sizes that choose the launches are the tree's, or, in a captured step,
// the last build's with room to grow (every size is covered; they only set the
// parallelism), with all 22 levels issued.
template <class... KA, class... A>
int launch_levels(Ctx* c, int64_t span_nodes, void (*kern)(KA...), A... args) {
    const auto& ls = c->lvl_start;
    auto nodes = [&](int l) -> int64_t {
        const int64_t v = l + 1 < (int)ls.size() ? ls[l + 1] - ls[l] : 0;
        return c->dev_sizes ? with_room(c, v) : v;
    };
    const unsigned long long* lvl = c->d_sz + kSzLvl;
    int hi = c->dev_sizes ? kLevels : (int)ls.size() - 2;
    while (hi >= 0) {
        int lo = hi;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute at[2] = {};
        cfg.stream = c->stream;
        at[0] = early_attribute(!c->capturing);
        cfg.attrs = at;
        cfg.numAttrs = 1;
        if (nodes(hi) <= span_nodes) {
            while (lo > 0 && nodes(lo - 1) <= span_nodes) --lo;
            cfg.gridDim = dim3(kSpanBlocks);
            cfg.blockDim = dim3(kSpanThreads);
            at[1].id = cudaLaunchAttributeClusterDimension;
            at[1].val.clusterDim.x = kSpanBlocks;
            at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
            cfg.numAttrs = 2;
        } else {
            cfg.gridDim = dim3(blocks_for(nodes(hi), 128));
            cfg.blockDim = dim3(128);
        }
        BH_CUDA(c, cudaLaunchKernelEx(&cfg, kern, args..., lvl, hi, lo));
        BH_LAUNCH(c);
        hi = lo - 1;
    }
    return BH_OK;
}

int grow_nodes(Ctx* c, size_t need) {
    if (need <= c->level.cap) return BH_OK;
    size_t cap = need + need / 2 + 1024;
    BH_TRY(grow(c, c->level, cap, "node level"));
    BH_TRY(grow(c, c->nchild, cap, "node nchild"));
    BH_TRY(grow(c, c->begin, cap, "node begin"));
    BH_TRY(grow(c, c->end, cap, "node end"));
    BH_TRY(grow(c, c->parent, cap, "node parent"));
    BH_TRY(grow(c, c->first_child, cap, "node first_child"));
    return BH_OK;
}

}  // namespace

int64_t tree_count_words(int64_t n) { return kTreeRows * ((n + kTreeTile - 1) / kTreeTile); }

// Nodes and groups.  Eager: the counts are read back once, to size the
// arrays, together with the status word of the keys (with an error in it the
// particles were left as they were).  Device-sized (c->dev_build): the arrays hold c->cap_nodes nodes and
// leaves and one group per particle; c->n_nodes and c->n_groups are those bounds until
// the sizes are read back.
int stage_octree(Ctx* c) {
    const int64_t n = c->n, ntiles = (n + kTreeTile - 1) / kTreeTile;
    const int np = c->n_patches, n_leaf = c->prm.n_leaf, n_g = c->prm.n_g;
    const bool dev = c->dev_build;
    const uint64_t* key = c->key[c->key_cur].p;
    BH_TRY(grow(c, c->tree_cnt, (size_t)tree_count_words(n), "node counts"));
    BH_TRY(grow(c, c->tree_range, (size_t)n, "node ranges"));
    BH_TRY(grow(c, c->tree_top, (size_t)n, "first nodes"));
    uint32_t* cnt = c->tree_cnt.p;
    BH_CUDA(c, launch(c, k_tree_count, (unsigned)ntiles, kTreeThreads, 0, key, n, c->d_off.p, np, n_leaf,
                      n_g, ntiles, c->tree_range.p, cnt));
    BH_LAUNCH(c);
    BH_TRY(scan_u32(c, cnt, tree_count_words(n), c->d_small));
    BH_CUDA(c, launch(c, k_tree_sizes, 1, 32, 0, cnt, ntiles, c->d_small, dev ? (unsigned long
                      long)c->cap_nodes : ~0ull, c->d_sz, c->d_status));
    BH_LAUNCH(c);
    if (dev) {
        c->n_nodes = c->cap_nodes;
        c->n_groups = n;  // (c->n_leaves stays the previous build's)
    } else {
        const unsigned long long* sz = c->h_pin;
        BH_CUDA(c, cudaMemcpyAsync(c->h_pin, c->d_sz, kSzWords * sizeof(*sz), cudaMemcpyDeviceToHost, c->stream));
        BH_TRY(read_status(c));  // non-finite coordinates; a particle on the axis of the cylindrical frame
        c->n_nodes = (int64_t)sz[kSzLvl + kLevels + 2];
        c->n_groups = (int64_t)sz[kSzNg];
        c->n_leaves = (int64_t)sz[kSzNl];
        c->lvl_start.assign(1, 0);
        for (int l = 0; l <= kLevels && sz[kSzLvl + l + 1] > sz[kSzLvl + l]; ++l)
            c->lvl_start.push_back((int64_t)sz[kSzLvl + l + 1]);
        BH_TRY(grow_nodes(c, (size_t)c->n_nodes));
        BH_TRY(grow(c, c->groups, (size_t)c->n_groups + 1, "groups"));
        BH_TRY(grow(c, c->leaves, (size_t)c->n_leaves, "leaves"));
    }
    BH_CUDA(c, launch(c, k_tree_write, (unsigned)ntiles, kTreeThreads, 0, c->tree_range.p, n, c->d_off.p,
                      np, ntiles, cnt, c->n_nodes, c->level.p, c->begin.p, c->end.p, c->parent.p, c->first_child.p,
                      c->nchild.p, c->groups.p, c->leaves.p, c->tree_top.p));
    BH_LAUNCH(c);
    BH_CUDA(c, launch(c, k_tree_link, blocks_for(c->n_nodes, 128), 128, 0, key, c->d_off.p, np, c->d_sz,
                      c->level.p, c->begin.p, c->end.p, c->parent.p, c->first_child.p, c->nchild.p));
    BH_LAUNCH(c);
    return BH_OK;
}

int stage_boxes(Ctx* c) {
    const int64_t nn = c->n_nodes;
    BH_TRY(grow(c, c->qlo, (size_t)nn * 3, "node qlo"));
    BH_TRY(grow(c, c->qhi, (size_t)nn * 3, "node qhi"));
    BH_TRY(grow(c, c->wnode, (size_t)nn, "walk records"));
    return launch_levels(c, kSpanBoxes, k_boxes, c->key[c->key_cur].p, c->n, c->n_patches, c->level.p, c->begin.p,
                         c->end.p, c->first_child.p, c->nchild.p, c->tree_top.p, c->qlo.p, c->qhi.p, c->wnode.p);
}

int stage_moments(Ctx* c, const bh_particles* p) {
    const int64_t nn = c->n_nodes;
    if (c->prm.precision != BH_PREC_FP32) return stage_moments64(c, p);
    // FP32 path: hi/lo split of the particles with the leaves' moments, then
    // the inner nodes', all in FP32 with a hi/lo centre (no FP64 arithmetic)
    BH_TRY(grow(c, c->cell32, (size_t)nn * 3, "FP32 cell records"));
    BH_TRY(grow(c, c->cell32lo, (size_t)nn, "FP32 cell mass corrections"));
    BH_TRY(grow(c, c->phi, (size_t)c->n, "FP32 positions hi"));
    BH_TRY(grow(c, c->plo, (size_t)c->n, "FP32 positions lo"));
    const bool quad = c->prm.order >= 2;
    BH_TRY(stage_begin(c, BH_STAGE_SPLIT));
    // (captured: the last build's leaves with room to grow; strided)
    const int64_t nl = c->dev_sizes ? with_room(c, c->n_leaves) : c->n_leaves;
    auto leaf = quad ? k_leaf32<2> : k_leaf32<1>;
    BH_CUDA(c, launch(c, leaf, blocks_for(nl, kLeafTile), kLeafTile, 0, c->leaves.p, c->d_sz + kSzNl,
                      c->begin.p, c->end.p, p->x, p->y, p->z, p->m, c->phi.p, c->plo.p, c->cell32.p,
                      c->cell32lo.p));
    BH_LAUNCH(c);
    BH_TRY(stage_end(c));
    BH_TRY(stage_begin(c, BH_STAGE_MOMENTS));
    BH_TRY(launch_levels(c, kSpanMoments32, quad ? k_moments32<2> : k_moments32<1>, c->first_child.p, c->nchild.p,
                         c->cell32.p, c->cell32lo.p));
    return stage_end(c);
}

// FP64 node moments (the FP64 path's records; the FP32 path's potential
// diagnostic also uses them).
int stage_moments64(Ctx* c, const bh_particles* p) {
    const int64_t nn = c->n_nodes;
    const bool steps = c->prm.precision == BH_PREC_FP64;
    for (auto* b : {&c->M, &c->cx, &c->cy, &c->cz}) BH_TRY(grow(c, *b, (size_t)nn, "moments", steps));
    BH_TRY(grow(c, c->Q, (size_t)nn * 6, "moments Q", steps));
    BH_TRY(stage_begin(c, BH_STAGE_MOMENTS));
    BH_TRY(launch_levels(c, kSpanMoments64, c->prm.order >= 2 ? k_moments<2> : k_moments<1>, c->begin.p, c->end.p, c->first_child.p,
                         c->nchild.p, p->x, p->y, p->z, p->m, c->M.p, c->cx.p, c->cy.p, c->cz.p, c->Q.p));
    return stage_end(c);
}

}  // namespace bh
