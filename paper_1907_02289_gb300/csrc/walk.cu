// walk.cu -- Sec. 4.2 step 3d, first half: one tree traversal per group
// builds the group's interaction list (Barnes' group walk): opened leaves
// become particle entries, accepted nodes become cell entries.  The walk is
// depth first in octant order, so both lists come out ordered by first
// particle; it needs no stack, since every node carries the successor of its
// subtree.  A count pass sizes the lists and a fill pass writes them (16-byte
// stores); from the second build on, one pass both counts and writes each
// group's lists into a slot sized from the previous build, and a copy packs
// the slots (a group that outgrows its slot sends the build back to count
// and fill).  The particle entries are then expanded into the particle
// indices the force kernel reads.
//
// Opening test (integer boxes on the key grid, exact): per axis the gap in
// whole cells is delta = max(0, clo - ghi - 1, glo - chi - 1), d2 = sum of
// delta^2.  A node of level l (side 2^(21-l) cells) is opened iff
// fl(theta^2 * d2) < 4^(21-l), or d2 <= (r_coll * S)^2.  Both comparisons
// are monotone in the integer d2, so the host turns them into integer
// thresholds once per build: open iff d2 < D[l] or d2 <= RCQ.  With several
// patches a group walks the tree of its own patch (root = patch index), and
// RCQ is per patch (each patch has its own key grid).
//
// For the FP32 kernel the expansion puts a group's list particles in two
// runs: "near" leaves first, then "far" leaves, far meaning beyond contact
// reach with a margin (so no pair in them can touch) and a gap of at least an
// eighth of the group's largest side.  The kernel forms far separations from
// single FP32 coordinates relative to the group origin (the arithmetic of
// Sec. 4.7), whose error relative to the separation s is then at most about
// 2 u (1 + E / s) (E the group's extent from its centre, at most sqrt(3)
// times its side; u = 2^-24), i.e. 2 u (1 + 8 sqrt(3)) ~ 30 u, and skips the
// contact test for them.
#include <algorithm>
#include <cmath>
#include <vector>

#include "bh_internal.cuh"

namespace bh {
namespace {

struct WalkParams {
    long long D[kLevels + 1];
    const long long* rcq;  // per patch
    const long long* rfar;    // per patch: d2 above this cannot hold a contact pair (margin included)
    const long long* period;  // per patch period of grid axis 0 (cylindrical frame), 0 = none
    const int64_t* off;    // patch particle offsets (np + 1)
    int np;
};

// Patch holding particle index gb: the last patch starting at or before it.
__device__ __forceinline__ int patch_of(const WalkParams& wp, uint32_t gb) {
    int root = 0;
    for (int lo = 0, hi = wp.np - 1; lo < hi;) {
        const int mid = (lo + hi + 1) >> 1;
        if (wp.off[mid] <= (int64_t)gb)
            lo = root = mid;
        else
            hi = mid - 1;
    }
    return root;
}

// Squared gap in whole cells between node box R and the group box [glo, ghi]
// (axis 0 periodic with the given period in cells when period > 0).
__device__ __forceinline__ long long box_gap2(const WalkNode& R, const int (&glo)[3], const int (&ghi)[3],
                                              int period) {
    const int lo0 = (int)(R.a.x & kQMax);
    const int t1 = lo0 - ghi[0] - 1, t2 = glo[0] - (int)R.b.x - 1;
    int d0 = max(0, max(t1, t2));
    if (period > 0 && d0 > 0)  // periodic phi axis: the shorter way round
        d0 = min(d0, max(0, t1 > 0 ? glo[0] + period - (int)R.b.x - 1 : lo0 + period - ghi[0] - 1));
    const int lo1 = (int)(R.a.y & kQMax);
    const int d1 = max(0, max(lo1 - ghi[1] - 1, glo[1] - (int)R.b.y - 1));
    const int d2 = max(0, max((int)R.a.z - ghi[2] - 1, glo[2] - (int)R.b.z - 1));
    return (long long)d0 * d0 + (long long)d1 * d1 + (long long)d2 * d2;
}

// Per-thread list writer: entries are gathered in registers and written as
// aligned 16-byte stores; the partial quads at the two ends of the thread's
// run [base, base + count) are written entry by entry, so no store touches
// another thread's run.  dst must be 16-byte aligned.
struct ListOut {
    int32_t* dst;
    int64_t base, pos, cap;  // entries at or past cap are counted, not written
    int32_t v0, v1, v2, v3;
    __device__ __forceinline__ int32_t at(int s) const { return s == 0 ? v0 : s == 1 ? v1 : s == 2 ? v2 : v3; }
    __device__ __forceinline__ void put_range(int64_t a, int64_t b) const {
        for (int64_t q = a; q < b; ++q) dst[q] = at((int)(q & 3));
    }
    __device__ __forceinline__ void put(int32_t v) {
        if (pos >= cap) {
            ++pos;
            return;
        }
        const int s = (int)(pos & 3);
        v0 = s == 0 ? v : v0;
        v1 = s == 1 ? v : v1;
        v2 = s == 2 ? v : v2;
        v3 = s == 3 ? v : v3;
        if (s == 3) {
            if (pos - 3 >= base)
                *reinterpret_cast<int4*>(dst + (pos - 3)) = make_int4(v0, v1, v2, v3);
            else
                put_range(base, pos + 1);
        }
        ++pos;
    }
    __device__ __forceinline__ void flush() const { put_range(max(base, min(pos, cap) & ~(int64_t)3), min(pos, cap)); }
};

// The walk is stackless: a node that is not descended into is followed by
// its subtree's successor (skip), an opened inner node by its first child,
// which visits the nodes in the same depth-first octant order as a stack.
// Modes: count (list sizes and interaction counts); fill (the lists, at the
// scanned offsets); stash (count, and write each group's lists into a slot
// of capP / capC entries at k * cap, flagging a group that does not fit).
// Count and stash also record the longest lists, which size the next
// build's slots.
constexpr int kWalkCount = 0, kWalkFill = 1, kWalkStash = 2;

struct WalkArgs {
    int64_t ng;
    const unsigned long long* dng;  // device group count (device-sized builds; NULL: ng)
    int64_t slots;                  // groups with a list slot (< 0: every one)
    const int32_t* groups;
    const WalkNode* wn;
    const uint32_t *begin, *end;
    int64_t *np_io, *nc_io, *nj_io;
    int32_t *P, *C;
    unsigned long long* inter;
    int64_t nn;
    int* status;
    int64_t capP, capC;
    unsigned long long *longest, *overflow;
};

// One group's counts: list leaves and cells, list particles (other than its
// own), its particles, and its own particles found in list leaves.
struct WalkCount {
    int64_t np = 0, nc = 0, nj = 0, ni = 0, nown = 0;
};

// A group's box, patch thresholds and list outputs.
struct WalkGroup {
    int glo[3], ghi[3];
    uint32_t gb, ge;
    int root, period;
    long long rcq;
    int32_t *P, *C;          // where its entries go (indexed by baseP.., baseC..)
    int64_t baseP, baseC, capP, capC;
};

// Whether group k is walked in this mode (fill of a device-sized build: only
// the groups whose lists did not fit a slot).
template <int MODE>
__device__ __forceinline__ bool walk_wanted(const WalkArgs& A, int64_t k) {
    if (MODE != kWalkFill || A.slots < 0) return true;
    return !(k < A.slots && A.np_io[k + 1] - A.np_io[k] <= A.capP && A.nc_io[k + 1] - A.nc_io[k] <= A.capC);
}

template <int MODE>
__device__ __forceinline__ WalkGroup walk_group(const WalkArgs& A, const WalkParams& wp, int64_t k) {
    const int32_t g = A.groups[k];
    const WalkNode G = A.wn[g];
    WalkGroup W;
    W.gb = A.begin[g];
    W.ge = A.end[g];
    W.glo[0] = (int)(G.a.x & kQMax); W.glo[1] = (int)(G.a.y & kQMax); W.glo[2] = (int)G.a.z;
    W.ghi[0] = (int)G.b.x; W.ghi[1] = (int)G.b.y; W.ghi[2] = (int)G.b.z;
    W.root = patch_of(wp, W.gb);
    W.rcq = wp.rcq[W.root];
    W.period = (int)wp.period[W.root];
    W.P = A.P;
    W.C = A.C;
    W.baseP = W.baseC = 0;
    W.capP = W.capC = INT64_MAX;
    if (MODE == kWalkFill) {
        W.baseP = A.np_io[k];
        W.baseC = A.nc_io[k];
    } else if (MODE == kWalkStash && (A.slots < 0 || k < A.slots)) {
        W.P = A.P + k * A.capP;
        W.C = A.C + k * A.capC;
        W.capP = A.capP;
        W.capC = A.capC;
    } else if (MODE == kWalkStash) {  // no slot: counted only, filled later
        W.capP = W.capC = 0;
    }
    return W;
}

// The walk of one group by one thread.
template <int MODE>
__device__ __forceinline__ WalkCount walk_serial(const WalkArgs& A, const WalkParams& wp, const WalkGroup& W) {
    constexpr bool WRITE = MODE != kWalkCount;
    WalkCount n;
    n.ni = (int64_t)(W.ge - W.gb);
    ListOut po{W.P, W.baseP, W.baseP, W.capP, 0, 0, 0, 0}, co{W.C, W.baseC, W.baseC, W.capC, 0, 0, 0, 0};
    int node = W.root;
    for (int64_t visits = 0;; ++visits) {
        const WalkNode R = A.wn[node];
        const int after = (int)R.a.w;
        const int lev = (int)((R.a.x >> kLevels) & 31u);
        const bool leaf = (R.a.x & kWalkLeaf) != 0;
        const long long d2 = box_gap2(R, W.glo, W.ghi, W.period);
        const bool open = d2 < wp.D[lev] || d2 <= W.rcq;
        int next = after;
        if (open) {
            if (leaf) {
                if (WRITE) po.put(node);
                ++n.np;
                const uint32_t lb = R.b.w;
                uint32_t lc = R.a.y >> kLevels;
                if (lc == kWalkCntMax) lc = A.end[node] - lb;
                if (lb >= W.gb && lb < W.ge)
                    n.nown += (int64_t)lc;  // the group's own particles
                else
                    n.nj += (int64_t)lc;
            } else {
                next = (int)R.b.w;
            }
        } else {
            if (WRITE) co.put(node);
            ++n.nc;
        }
        if (next < 0) break;
        if (next >= A.nn || visits >= A.nn) {  // never taken for a valid tree
            atomicOr(A.status, kStatBounds);
            break;
        }
        node = next;
    }
    if (WRITE) {
        po.flush();
        co.flush();
    }
    return n;
}

// Count outputs of group k (count and stash modes).
template <int MODE>
__device__ __forceinline__ void walk_counts(const WalkArgs& A, int64_t k, const WalkGroup& W, const WalkCount& n) {
    if (MODE == kWalkStash && (n.np > W.capP || n.nc > W.capC)) atomicOr(A.overflow, 1ull);
    if (MODE != kWalkFill) {
        A.np_io[k] = n.np;
        A.nc_io[k] = n.nc;
        A.nj_io[k] = n.nj;
    }
}

// A thread per group: with many groups neighbouring threads follow nearly the
// same path and the SMs are full.
template <int MODE>
__global__ void __launch_bounds__(128) k_walk(const WalkArgs A, const WalkParams wp) {
    launch_wait();
    const int64_t ng = A.dng ? min(A.ng, (int64_t)*A.dng) : A.ng;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < ng; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = base + threadIdx.x;
        WalkCount n;
        if (k < ng && walk_wanted<MODE>(A, k)) {
            const WalkGroup W = walk_group<MODE>(A, wp, k);
            n = walk_serial<MODE>(A, wp, W);
            walk_counts<MODE>(A, k, W, n);
        }
        if (MODE != kWalkFill) {
            // interaction counts: n_i * (list particles) and n_i * (list cells);
            // longest particle and cell lists
            unsigned long long ipp = (unsigned long long)(n.ni * (n.nj + n.nown)),
                               ipc = (unsigned long long)(n.ni * n.nc);
            unsigned long long lp = (unsigned long long)n.np, lc = (unsigned long long)n.nc;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                ipp += __shfl_xor_sync(0xffffffffu, ipp, o);
                ipc += __shfl_xor_sync(0xffffffffu, ipc, o);
                lp = max(lp, __shfl_xor_sync(0xffffffffu, lp, o));
                lc = max(lc, __shfl_xor_sync(0xffffffffu, lc, o));
            }
            if ((threadIdx.x & 31) == 0) {
                atomicAdd(&A.inter[0], ipp);
                atomicAdd(&A.inter[1], ipc);
                atomicMax(&A.longest[0], lp);
                atomicMax(&A.longest[1], lc);
            }
        }
    }
}

// A warp per group, for trees with few groups, where k_walk is a chain of
// dependent loads on an idle GPU (0.55 us per visited node whatever their
// number).  The warp holds the group's entries in shared memory in depth-first
// order, starting with the root, and takes the tree level by level: 32
// untested entries at a time are tested, then every opened inner node is
// replaced by its children in its place, so the order stays depth first and
// ends as the lists' order.  An entry is a node id with its state in the top
// two bits; an opened node becomes (first child, child count - 1).  Measured,
// the walk by a thread and by a warp per group: 65,537-particle ring (1166
// groups) 151 and 18 us; 100,003-particle cube (4096 groups of 1300 entries) 865
// and 77 us.
//
// Entries that outgrow the buffer are walked in pieces (coop_pieces): the back
// of the buffer holds those whose turn has not come, and a piece from their
// front that fits what is free goes through the same levels in the front of the
// buffer, its settled entries leaving for the lists.
constexpr int kCoopWarps = 4;
constexpr uint32_t kCoopLevel = 2048;  // most entries before a level is taken in pieces
// room beyond: a piece of one opened node adds at most 7 entries per level
constexpr uint32_t kCoopSpare = 7 * kLevels + 13, kCoopCap = kCoopLevel + kCoopSpare;
static_assert(kCoopSpare >= 7 * kLevels + 8, "the last of a chain of opened nodes needs eight places");
constexpr int64_t kCoopGroups = 40000;  // most groups it is chosen for
constexpr uint32_t kEntNew = 0u, kEntCell = 1u << 30, kEntLeaf = 2u << 30, kEntOpen = 3u << 30;
constexpr int kEntBits = 27;  // node id bits beside an opened node's 3 bits of child count

__device__ __forceinline__ uint32_t warp_exclusive(uint32_t v, int lane, uint32_t* total) {
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    *total = __shfl_sync(0xffffffffu, x, 31);
    return x - v;
}

// Places an entry takes once it is opened.
__device__ __forceinline__ uint32_t places(uint32_t v) {
    return v >= kEntOpen ? ((v >> kEntBits) & 7u) + 1u : 1u;
}

// One group's walk by the lanes of a warp (all calls warp-uniform).
template <int MODE>
struct CoopWalk {
    const WalkArgs& A;
    const WalkParams& wp;
    const WalkGroup W;
    uint32_t* E;  // kCoopCap entries
    int lane;
    uint32_t nj = 0, nown = 0;  // of this lane's tests
    int64_t np = 0, nc = 0;     // entries sent to the lists

    // Test the untested entries of E[0, len); whether any was opened, and how
    // many more places the opened ones need.
    __device__ __forceinline__ bool test(uint32_t len, uint32_t* more) {
        uint32_t grow = 0;  // (an opened node with one child is replaced without growth)
        bool opened = false;
        for (uint32_t t = lane; t < len; t += 32) {
            const uint32_t v = E[t];
            if (v >> 30) continue;
            const WalkNode R = A.wn[v];
            const long long d2 = box_gap2(R, W.glo, W.ghi, W.period);
            uint32_t r = kEntCell | v;
            if (d2 < wp.D[(R.a.x >> kLevels) & 31u] || d2 <= W.rcq) {
                const uint32_t c = R.a.y >> kLevels;  // leaf: particles; inner: children
                if (R.a.x & kWalkLeaf) {
                    r = kEntLeaf | v;
                    const uint32_t lb = R.b.w, cnt = c == kWalkCntMax ? A.end[v] - lb : c;
                    if (lb >= W.gb && lb < W.ge)
                        nown += cnt;
                    else
                        nj += cnt;
                } else {
                    r = kEntOpen | (c - 1u) << kEntBits | R.b.w;
                    grow += c - 1u;
                    opened = true;
                }
            }
            E[t] = r;
        }
        const bool any = __any_sync(0xffffffffu, opened);
        *more = __reduce_add_sync(0xffffffffu, grow);
        __syncwarp();
        return any;
    }

    // Opened entries of E[0, len) -> their children, untested, in their places;
    // from the back: an entry never moves to a lower place.
    __device__ __forceinline__ void expand(uint32_t len, uint32_t more) {
        uint32_t out = len + more;
        for (int t0 = (int)((len - 1) & ~31u); t0 >= 0; t0 -= 32) {
            const uint32_t t = (uint32_t)t0 + lane;
            const uint32_t v = t < len ? E[t] : 0u;
            const uint32_t c = t < len ? places(v) : 0u;
            uint32_t tot;
            const uint32_t x = warp_exclusive(c, lane, &tot);
            out -= tot;
            __syncwarp();
            if (t < len && v >= kEntOpen) {
                const uint32_t f = v & ((1u << kEntBits) - 1u);
                for (uint32_t u = 0; u < c; ++u) E[out + x + u] = kEntNew | (f + u);
            } else if (t < len) {
                E[out + x] = v;
            }
            __syncwarp();
        }
    }

    // The lanes' settled entries v (those that have one) -> the lists.
    __device__ __forceinline__ void put(uint32_t v, bool has) {
        const bool isP = has && (v >> 30) == (kEntLeaf >> 30), isC = has && !isP;
        const unsigned mP = __ballot_sync(0xffffffffu, isP), mC = __ballot_sync(0xffffffffu, isC);
        if (MODE != kWalkCount) {
            const unsigned lt = (1u << lane) - 1u;
            const int64_t p = np + __popc(mP & lt), c = nc + __popc(mC & lt);
            if (isP && p < W.capP) W.P[W.baseP + p] = (int32_t)(v & 0x3fffffffu);
            if (isC && c < W.capC) W.C[W.baseC + c] = (int32_t)(v & 0x3fffffffu);
        }
        np += __popc(mP);
        nc += __popc(mC);
    }

    __device__ __forceinline__ void put_all(uint32_t len) {
        for (uint32_t t0 = 0; t0 < len; t0 += 32) put(t0 + lane < len ? E[t0 + lane] : 0u, t0 + lane < len);
    }
};

// The rest of a walk whose tested entries E[0, len) cannot all be opened in the
// buffer.  E[at, kCoopCap) are the entries whose turn has not come, in order.
// Those up to the first opened one go to the lists; then a piece from the
// front of the rest, opened, moves to E[0, ..): as many entries as a quarter of
// the free room holds (their children's children need room too; a half or a
// sixth measures the same), at least one.  It is taken level by level until it
// is settled, or goes back when it does not fit either, by then at least a
// level further.  Pieces of more than one entry leave kCoopSpare places free,
// and those of one, a chain down the levels, add at most 7 entries per level,
// so there is always room for the next one.
// Measured, the list build of a 1,000,003-particle cube (32,768 groups) with such
// groups walked by one lane, with k_walk, and with this: 6.4, 1.6 and 1.0 ms at
// theta 0.5 (2150 entries a group), 13.7, 2.7 and 1.5 ms at theta 0.4 (3500); of a
// 100,003-particle cube at theta 0.4 (4096 groups of 2350) 1.45, 1.69 and 0.22 ms.
// Inlined, or the walk's state goes through memory: 3.5 instead of 1.5 ms.
template <int MODE>
__device__ __forceinline__ void coop_pieces(CoopWalk<MODE>& C, uint32_t len) {
    uint32_t* E = C.E;
    const int lane = C.lane;
    uint32_t at = kCoopCap;
    auto go_back = [&](uint32_t cnt) {  // E[0, cnt) -> in front of E[at, ..), from the back
        for (int t0 = (int)((cnt - 1) & ~31u); t0 >= 0; t0 -= 32) {
            const uint32_t t = (uint32_t)t0 + lane;
            const uint32_t v = t < cnt ? E[t] : 0u;
            __syncwarp();
            if (t < cnt) E[at - cnt + t] = v;
            __syncwarp();
        }
        at -= cnt;
    };
    go_back(len);
    for (int64_t rounds = 0;; ++rounds) {
        for (;;) {  // settled entries up to the first opened one
            const uint32_t cnt = min(32u, kCoopCap - at);
            const uint32_t v = (uint32_t)lane < cnt ? E[at + lane] : 0u;
            const unsigned m = __ballot_sync(0xffffffffu, v >= kEntOpen);
            const uint32_t k = m ? (uint32_t)(__ffs(m) - 1) : cnt;
            C.put(v, (uint32_t)lane < k);
            at += k;
            if (m || at == kCoopCap) break;
        }
        if (at == kCoopCap) return;
        const uint32_t room = at > kCoopSpare ? (at - kCoopSpare) / 4u : 0u;
        uint32_t n = 0, need = 0;  // the piece's entries, and their places once opened
        for (;;) {
            const uint32_t cnt = min(32u, kCoopCap - at);
            const uint32_t v = (uint32_t)lane < cnt ? E[at + lane] : 0u;
            const uint32_t c = (uint32_t)lane < cnt ? places(v) : 0u;
            uint32_t tot;
            const uint32_t x = warp_exclusive(c, lane, &tot) + c;
            const bool in = (uint32_t)lane < cnt && (need + x <= room || (n == 0 && lane == 0));
            const uint32_t k = (uint32_t)__popc(__ballot_sync(0xffffffffu, in));
            if (in) E[n + lane] = v;  // (n + lane < at + lane: read by now)
            if (k > 0) need += __shfl_sync(0xffffffffu, x, (int)k - 1);
            __syncwarp();
            n += k;
            at += k;
            if (k < 32u) break;
        }
        if (need > at || rounds > C.A.nn) {  // never taken for a valid tree
            if (lane == 0) atomicOr(C.A.status, kStatBounds);
            return;
        }
        for (uint32_t more = need - n;;) {
            C.expand(n, more);
            n += more;
            if (!C.test(n, &more)) {
                C.put_all(n);
                break;
            }
            if (n + more + kCoopSpare > at) {
                go_back(n);
                break;
            }
        }
    }
}

template <int MODE>
__global__ void __launch_bounds__(32 * kCoopWarps) k_walk_coop(const __grid_constant__ WalkArgs A,
                                                             const __grid_constant__ WalkParams wp) {
    launch_wait();
    __shared__ uint32_t buf[kCoopWarps][kCoopCap];
    const int lane = threadIdx.x & 31;
    uint32_t* E = buf[threadIdx.x >> 5];
    const int64_t ng = A.dng ? min(A.ng, (int64_t)*A.dng) : A.ng;
    unsigned long long ipp = 0, ipc = 0, lp = 0, lc = 0;
    for (int64_t k = (int64_t)blockIdx.x * kCoopWarps + (threadIdx.x >> 5); k < ng;
         k += (int64_t)gridDim.x * kCoopWarps) {
        if (!walk_wanted<MODE>(A, k)) continue;
        CoopWalk<MODE> C{A, wp, walk_group<MODE>(A, wp, k), E, lane};
        __syncwarp();
        if (lane == 0) E[0] = kEntNew | (uint32_t)C.W.root;
        __syncwarp();
        // (untested entries are nodes of one level; the last level's are leaves)
        for (uint32_t len = 1, more;; len += more) {
            if (!C.test(len, &more)) {
                C.put_all(len);
                break;
            }
            if (len + more > kCoopLevel) {
                coop_pieces<MODE>(C, len);
                break;
            }
            C.expand(len, more);
        }
        WalkCount n;
        n.np = C.np;
        n.nc = C.nc;
        n.nj = (int64_t)__reduce_add_sync(0xffffffffu, C.nj);
        n.nown = (int64_t)__reduce_add_sync(0xffffffffu, C.nown);
        if (lane == 0) {
            const int64_t ni = (int64_t)(C.W.ge - C.W.gb);
            walk_counts<MODE>(A, k, C.W, n);
            ipp += (unsigned long long)(ni * (n.nj + n.nown));
            ipc += (unsigned long long)(ni * n.nc);
            lp = max(lp, (unsigned long long)n.np);
            lc = max(lc, (unsigned long long)n.nc);
        }
    }
    if (MODE != kWalkFill && lane == 0) {
        atomicAdd(&A.inter[0], ipp);
        atomicAdd(&A.inter[1], ipc);
        atomicMax(&A.longest[0], lp);
        atomicMax(&A.longest[1], lc);
    }
}

// One warp per group: particle entries -> particle indices, leaving out the
// group's own particles (the force kernels evaluate those in a separate phase
// that excludes i = j).  SPLIT: near leaves first, far leaves after them
// (each run in list order); jm[k] = index of the first far particle, and
// the far interactions n_i x (far particles) are summed into *n_far.
template <bool SPLIT>
__global__ void k_expand(int64_t ng, const unsigned long long* dng, const int32_t* groups,
                         const int64_t* pp_off, const int32_t* P, const uint32_t* begin,
                         const uint32_t* end, const WalkNode* wn, WalkParams wp,
                         const int64_t* jj_off, uint32_t* JJ, int64_t* jm,
                         unsigned long long* n_far) {
    launch_wait();
    if (dng) ng = min(ng, (int64_t)*dng);
    const int lane = threadIdx.x & 31;
    const int64_t wstride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < ng; k += wstride) {
        const int32_t g = groups[k];
        const uint32_t gb = begin[g], ge = end[g];
        const int64_t e0 = pp_off[k], e1 = pp_off[k + 1];
        int glo[3] = {0, 0, 0}, ghi[3] = {0, 0, 0};
        long long rfar = 0, ext2 = 0;
        int period = 0;
        if (SPLIT) {
            const WalkNode G = wn[g];
            glo[0] = (int)(G.a.x & kQMax); glo[1] = (int)(G.a.y & kQMax); glo[2] = (int)G.a.z;
            ghi[0] = (int)G.b.x; ghi[1] = (int)G.b.y; ghi[2] = (int)G.b.z;
            const long long ext = max(ghi[0] - glo[0], max(ghi[1] - glo[1], ghi[2] - glo[2])) + 1;
            ext2 = ext * ext;
            const int root = patch_of(wp, gb);
            rfar = wp.rfar[root];
            period = (int)wp.period[root];
        }
        // leaf entry e -> (first particle, count; 0 for the group's own
        // leaves) from its walk record, and whether it is far
        auto entry = [&](int64_t e, uint32_t& b, uint32_t& cnt, bool& far) {
            b = 0;
            cnt = 0;
            far = false;
            if (e < e1) {
                const int32_t leaf = P[e];
                const WalkNode R = wn[leaf];
                b = R.b.w;
                cnt = R.a.y >> kLevels;
                if (cnt == kWalkCntMax) cnt = end[leaf] - b;
                if (b >= gb && b < ge) cnt = 0;
                if (SPLIT && cnt > 0) {
                    const long long d2 = box_gap2(R, glo, ghi, period);
                    far = d2 > rfar && 64 * d2 >= ext2;
                }
            }
        };
        int64_t jn = jj_off[k], jf = jn;
        if (SPLIT) {  // far run starts after every near particle
            uint32_t near = 0;
            for (int64_t e = e0 + lane; e < e1; e += 32) {
                uint32_t b, cnt;
                bool far;
                entry(e, b, cnt, far);
                near += far ? 0u : cnt;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) near += __shfl_xor_sync(0xffffffffu, near, o);
            jf = jn + near;
            if (lane == 0) {
                jm[k] = jf;
                const unsigned long long ni = ge - gb;
                atomicAdd(n_far, ni * (unsigned long long)(jj_off[k + 1] - jf));
            }
        }
        for (int64_t e = e0; e < e1; e += 32) {
            uint32_t b, cnt;
            bool far;
            entry(e + lane, b, cnt, far);
            const uint32_t cn = far ? 0u : cnt, cf = far ? cnt : 0u;
            uint32_t xn = cn, xf = cf;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t yn = __shfl_up_sync(0xffffffffu, xn, o);
                const uint32_t yf = __shfl_up_sync(0xffffffffu, xf, o);
                if (lane >= o) {
                    xn += yn;
                    xf += yf;
                }
            }
            const uint32_t tn = __shfl_sync(0xffffffffu, xn, 31), tf = __shfl_sync(0xffffffffu, xf, 31);
            const int64_t pos = far ? jf + (xf - cf) : jn + (xn - cn);
            for (uint32_t t = 0; t < cnt; ++t) JJ[pos + t] = b + t;
            jn += tn;
            jf += tf;
        }
    }
}

// One warp per group: the group's stashed lists (slots of capP / capC
// entries) to their places in the packed lists.  slots >= 0 (device-sized
// build): only the groups below slots whose lists fit their slot.
__global__ void k_unstash(int64_t ng, const unsigned long long* dng, int64_t slots,
                          const int64_t* pp_off, const int64_t* pc_off,
                          const int32_t* sP, const int32_t* sC, int64_t capP,
                          int64_t capC, int32_t* P, int32_t* C) {
    launch_wait();
    if (dng) ng = min(ng, (int64_t)*dng);
    const int lane = threadIdx.x & 31;
    const int64_t wstride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < ng; k += wstride) {
        const int64_t p0 = pp_off[k], np = pp_off[k + 1] - p0, c0 = pc_off[k], nc = pc_off[k + 1] - c0;
        if (slots >= 0 && !(k < slots && np <= capP && nc <= capC)) continue;
        // four loads in flight per lane
        auto copy = [&](int32_t* dst, const int32_t* src, int64_t cnt) {
            for (int64_t t0 = 0; t0 < cnt; t0 += 128) {
                int32_t v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t t = t0 + 32 * u + lane;
                    v[u] = t < cnt ? src[t] : 0;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t t = t0 + 32 * u + lane;
                    if (t < cnt) dst[t] = v[u];
                }
            }
        };
        copy(P + p0, sP + k * capP, np);
        copy(C + c0, sC + k * capC, nc);
    }
}

// Walk thresholds per patch from its key grid (S = 2^21 / L).  Contact
// reach in grid units: Cartesian r_coll S; cylindrical (phi, r, z): two
// particles within r_coll have |dr|, |dz| <= r_coll and a phi difference of
// at most ~r_coll / r_min, so (r_coll / r_min + 4e-6) S bounds their grid
// distance (4e-6 covers twice the FP32 tree coordinates' error), and the phi
// axis wraps after floor(2 pi S) cells.  rcq = floor(reach^2); the far threshold
// of the split expansion widens the reach by 1e-5 of itself plus two cells,
// so that no rounding of a coordinate into its cell can put a touching pair
// into a far leaf.  Round-to-nearest operations throughout (no contraction).
__global__ void k_walk_thresholds(const double* box, int np, double r_coll, int cyl,
                                  long long* rcq, long long* rfar,
                                  long long* period) {
    launch_wait();
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= np) return;
    const double S = __ddiv_rn(2097152.0, box[8 * q + 3]);
    double a;
    long long per = 0;
    if (cyl) {
        a = __ddiv_rn(r_coll, box[8 * q + 1]);
        a = __dadd_rn(a, 4e-6);
        a = __dmul_rn(a, S);
        per = (long long)floor(__dmul_rn(6.283185307179586, S));
    } else {
        a = __dmul_rn(r_coll, S);
    }
    const double r2 = __dmul_rn(a, a);
    rcq[q] = (r2 >= 9.0e18) ? (long long)9.0e18 : (long long)floor(r2);
    const double w = r_coll > 0.0 ? __dadd_rn(__dmul_rn(a, 1.0 + 1e-5), 2.0) : 0.0;
    const double w2 = __dmul_rn(w, w);
    rfar[q] = (w2 >= 9.0e18) ? (long long)9.0e18 : (long long)floor(w2);
    period[q] = per;
}

// Device-sized build: the list totals against the buffers' room.
__global__ void k_list_room(const unsigned long long* tot, long long roomP, long long roomC,
                            long long roomJ, unsigned long long* sz) {
    launch_wait();
    if (threadIdx.x != 0) return;
    if ((long long)tot[0] > roomP || (long long)tot[1] > roomC || (long long)tot[2] > roomJ) sz[kSzOvf] |= kOvfLists;
}

WalkParams walk_params(const Ctx* c) {
    WalkParams w;
    const double th2 = c->prm.theta * c->prm.theta;
    const long long big = (long long)1 << 53;
    for (int l = 0; l <= kLevels; ++l) {
        const double s = std::ldexp(1.0, kLevels - l);
        const double s2 = s * s;
        if (th2 == 0.0) {
            w.D[l] = big;
            continue;
        }
        const double est = std::floor(s2 / th2);
        if (!(est < (double)big)) {
            w.D[l] = big;
            continue;
        }
        long long d = (long long)est;
        while (d > 0 && th2 * (double)(d - 1) >= s2) --d;
        while (!(th2 * (double)d >= s2)) ++d;
        w.D[l] = d;
    }
    w.rcq = c->d_rcq.p;
    w.rfar = c->d_rfar.p;
    w.period = c->d_period.p;
    w.off = c->d_off.p;
    w.np = c->n_patches;
    return w;
}

}  // namespace

namespace {

// Walk thresholds of every patch, on the device from the root boxes.
int walk_thresholds(Ctx* c) {
    const int np = c->n_patches;
    BH_TRY(grow(c, c->d_rcq, (size_t)np, "walk contact thresholds"));
    BH_TRY(grow(c, c->d_rfar, (size_t)np, "far thresholds"));
    BH_TRY(grow(c, c->d_period, (size_t)np, "walk periods"));
    BH_CUDA(c, launch(c, k_walk_thresholds, blocks_for(np, 64), 64, 0, c->d_box, np, c->prm.r_coll,
                      c->prm.key_frame == 1, c->d_rcq.p, c->d_rfar.p, c->d_period.p));
    BH_LAUNCH(c);
    return BH_OK;
}

WalkArgs walk_args(const Ctx* c, const unsigned long long* dng, int64_t slots) {
    WalkArgs A = {};
    A.ng = c->n_groups;
    A.dng = dng;
    A.slots = slots;
    A.groups = c->groups.p;
    A.wn = c->wnode.p;
    A.begin = c->begin.p;
    A.end = c->end.p;
    A.np_io = c->cnt_p.p;
    A.nc_io = c->cnt_c.p;
    A.nj_io = c->cnt_j.p;
    A.inter = c->d_small + 8;
    A.nn = c->n_nodes;
    A.status = c->d_status;
    A.overflow = c->d_small + 11;
    A.longest = c->d_small + 12;  // two words
    return A;
}

// The walk of about `groups` groups (device-sized: more are strided over).
template <int MODE>
int launch_walk(Ctx* c, const WalkArgs& A, const WalkParams& wp, int64_t groups) {
    if (groups <= kCoopGroups && A.nn <= (int64_t)1 << kEntBits)
        BH_CUDA(c, launch(c, k_walk_coop<MODE>, blocks_for(groups, kCoopWarps), 32 * kCoopWarps, 0, A, wp));
    else
        BH_CUDA(c, launch(c, k_walk<MODE>, blocks_for(groups, 128), 128, 0, A, wp));
    BH_LAUNCH(c);
    return BH_OK;
}

// Particle entries -> particle indices (near run, then far run for the FP32
// kernel) and the FP32 kernel's group order.
int expand_lists(Ctx* c, const WalkParams& wp, const unsigned long long* dng, unsigned grid) {
    const int64_t ng = c->n_groups;
    const bool split = c->prm.precision == BH_PREC_FP32;
    unsigned long long* n_far = c->d_small + 10;  // (cleared before the walk)
    if (split) BH_TRY(grow(c, c->cnt_jm, (size_t)ng + 1, "list split points"));
    auto expand = split ? k_expand<true> : k_expand<false>;
    BH_CUDA(c, launch(c, expand, grid, 256, 0, ng, dng, c->groups.p, c->cnt_p.p, c->P.p, c->begin.p,
                      c->end.p, c->wnode.p, wp, c->cnt_j.p, c->JJ.p, split ? c->cnt_jm.p : nullptr, n_far));
    BH_LAUNCH(c);
    return BH_OK;
}

}  // namespace

int stage_lists(Ctx* c) {
    const int64_t ng = c->n_groups;
    BH_TRY(grow(c, c->cnt_p, (size_t)ng + 1, "list offsets P"));
    BH_TRY(grow(c, c->cnt_c, (size_t)ng + 1, "list offsets C"));
    BH_TRY(grow(c, c->cnt_j, (size_t)ng + 1, "list offsets J"));
    BH_TRY(walk_thresholds(c));
    const WalkParams wp = walk_params(c);
    unsigned long long* inter = c->d_small + 8;
    // One walk when the previous build gave slot sizes and the slots take
    // at most 4x the previous lists' storage; else (and after an overflow)
    // a count walk and a fill walk.
    const int64_t capP = c->walk_cap_p, capC = c->walk_cap_c;
    // (a list capacity bounds the entries held, so it rules out the slots)
    bool stash = capP > 0 && capC > 0 && c->prm.list_capacity == 0 &&
                 (double)ng * (double)(capP + capC) <= 4.0 * (double)(c->n_pp + c->n_pc) + 1.0e6;
    if (stash) {
        BH_TRY(grow(c, c->stash_p, (size_t)(ng * capP), "stashed particle lists"));
        BH_TRY(grow(c, c->stash_c, (size_t)(ng * capC), "stashed cell lists"));
    }
    BH_CUDA(c, cudaMemsetAsync(inter, 0, 6 * sizeof(unsigned long long), c->stream));  // words 8..13
    WalkArgs A = walk_args(c, nullptr, -1);
    if (stash) {
        A.P = c->stash_p.p;
        A.C = c->stash_c.p;
        A.capP = capP;
        A.capC = capC;
        BH_TRY(launch_walk<kWalkStash>(c, A, wp, ng));
    } else {
        BH_TRY(launch_walk<kWalkCount>(c, A, wp, ng));
    }
    int64_t* const arr[3] = {c->cnt_p.p, c->cnt_c.p, c->cnt_j.p};
    BH_TRY(scan3_i64(c, arr, ng, c->d_small, nullptr));
    const unsigned long long* h = c->h_pin;
    BH_CUDA(c, cudaMemcpyAsync(c->h_pin, c->d_small, 16 * sizeof(*h), cudaMemcpyDeviceToHost, c->stream));
    BH_CUDA(c, cudaStreamSynchronize(c->stream));
    c->n_pp = (int64_t)h[0];
    c->n_pc = (int64_t)h[1];
    c->n_jj = (int64_t)h[2];
    c->n_int_pp = (int64_t)h[8];
    c->n_int_pc = (int64_t)h[9];
    c->list_overflowed = false;
    if (c->prm.list_capacity > 0 && c->n_pp + c->n_pc + c->n_jj > c->prm.list_capacity) {
        c->list_overflowed = true;
        c->need_pp = c->n_pp;
        c->need_pc = c->n_pc;
        c->need_jj = c->n_jj;
        return fail(c, BH_E_LIST_OVERFLOW,
                    "the lists need %lld entries (%lld leaf, %lld cell, %lld list-particle), list_capacity is %lld",
                    (long long)(c->n_pp + c->n_pc + c->n_jj), (long long)c->n_pp, (long long)c->n_pc,
                    (long long)c->n_jj, (long long)c->prm.list_capacity);
    }
    BH_TRY(grow(c, c->P, (size_t)c->n_pp + 1, "particle lists"));
    BH_TRY(grow(c, c->C, (size_t)c->n_pc + 1, "cell lists"));
    BH_TRY(grow(c, c->JJ, (size_t)c->n_jj + 1, "list particle indices"));
    if (stash && h[11] == 0) {
        BH_CUDA(c, launch(c, k_unstash, blocks_for(ng * 32, 256), 256, 0, ng, nullptr, -1, c->cnt_p.p,
                          c->cnt_c.p, c->stash_p.p, c->stash_c.p, capP, capC, c->P.p, c->C.p));
        BH_LAUNCH(c);
        ++c->n_one_walk_builds;
    } else {
        A.P = c->P.p;
        A.C = c->C.p;
        A.capP = A.capC = 0;
        BH_TRY(launch_walk<kWalkFill>(c, A, wp, ng));
    }
    // slots of the next build: the longest lists of this one plus a quarter,
    // in whole 16-byte units
    c->walk_cap_p = (int64_t)(((h[12] + h[12] / 4 + 4) + 3) & ~3ull);
    c->walk_cap_c = (int64_t)(((h[13] + h[13] / 4 + 4) + 3) & ~3ull);
    BH_TRY(expand_lists(c, wp, nullptr, blocks_for(ng * 32, 256)));
    c->n_int_pp_far = 0;
    const bool f32 = c->prm.precision == BH_PREC_FP32;
    if (f32) BH_TRY(build_order32(c));
    BH_CUDA(c, cudaEventRecord(c->build_event, c->stream));
    c->far_pending = f32;  // its count is read when asked for
    if (f32) {
        const int rc = reserve_force32(c);  // (while the lists are written; the evaluation reports a lack of memory)
        if (rc != BH_E_NOMEM) BH_TRY(rc);
    }
    return BH_OK;
}

// Device-sized list build, first part: the walk of every group (counting,
// and writing each group's lists into its slot when it has one that fits:
// c->dev_slots slots of walk_cap_p / walk_cap_c entries), the list offsets,
// and the room check of the totals against the P, C and JJ buffers as they
// are (kOvfLists).  Group count on the device; c->n_groups is its bound.
int stage_lists_dev_walk(Ctx* c) {
    const int64_t ng = c->n_groups;
    const unsigned long long* dng = c->d_sz + kSzNg;
    BH_TRY(grow(c, c->cnt_p, (size_t)ng + 1, "list offsets P"));
    BH_TRY(grow(c, c->cnt_c, (size_t)ng + 1, "list offsets C"));
    BH_TRY(grow(c, c->cnt_j, (size_t)ng + 1, "list offsets J"));
    BH_TRY(walk_thresholds(c));
    const WalkParams wp = walk_params(c);
    unsigned long long* inter = c->d_small + 8;
    const int64_t slots = c->dev_slots, capP = c->walk_cap_p, capC = c->walk_cap_c;
    BH_TRY(grow(c, c->stash_p, (size_t)std::max<int64_t>(1, slots * capP), "stashed particle lists"));
    BH_TRY(grow(c, c->stash_c, (size_t)std::max<int64_t>(1, slots * capC), "stashed cell lists"));
    BH_CUDA(c, cudaMemsetAsync(inter, 0, 6 * sizeof(unsigned long long), c->stream));  // words 8..13
    WalkArgs A = walk_args(c, dng, slots);
    A.P = c->stash_p.p;
    A.C = c->stash_c.p;
    A.capP = capP;
    A.capC = capC;
    BH_TRY(launch_walk<kWalkStash>(c, A, wp, std::max<int64_t>(slots, 1)));
    int64_t* const arr[3] = {c->cnt_p.p, c->cnt_c.p, c->cnt_j.p};
    BH_TRY(scan3_i64(c, arr, ng, c->d_small, dng));
    BH_CUDA(c, launch(c, k_list_room, 1, 32, 0, c->d_small, (long long)c->P.cap - 1, (long long)c->C.cap -
                      1, (long long)c->JJ.cap - 1, c->d_sz));
    BH_LAUNCH(c);
    return BH_OK;
}

// Second part (issued to run only when the lists fit): the groups' lists
// from their slots or, for the groups without a fitting slot, from a second
// walk; the expansion into particle indices; the FP32 kernel's group order.
int stage_lists_dev_fill(Ctx* c) {
    const int64_t ng = c->n_groups;
    const unsigned long long* dng = c->d_sz + kSzNg;
    const WalkParams wp = walk_params(c);
    const int64_t slots = c->dev_slots, capP = c->walk_cap_p, capC = c->walk_cap_c;
    const unsigned grid = blocks_for(std::max<int64_t>(slots, 1) * 32, 256);  // a warp per expected group
    BH_CUDA(c, launch(c, k_unstash, grid, 256, 0, ng, dng, slots, c->cnt_p.p, c->cnt_c.p, c->stash_p.p,
                      c->stash_c.p, capP, capC, c->P.p, c->C.p));
    BH_LAUNCH(c);
    WalkArgs A = walk_args(c, dng, slots);
    A.P = c->P.p;
    A.C = c->C.p;
    A.capP = capP;
    A.capC = capC;
    BH_TRY(launch_walk<kWalkFill>(c, A, wp, std::max<int64_t>(slots, 1)));
    BH_TRY(expand_lists(c, wp, dng, grid));
    if (c->prm.precision == BH_PREC_FP32) BH_TRY(build_order32(c));
    return BH_OK;
}

}  // namespace bh
