// sort.cu -- Sec. 4.2 step 3a, first half: root box, Morton keys, the
// stable LSD radix sort of (key, original index) and the gather of every
// particle array into key order.
//
// Keys: q_a = min(floor((x_a - lo_a) * S), 2^21 - 1), S = 2^21 / L, with L the
// largest extent of the root box (1 if 0); key bit 3b+2/3b+1/3b = bit b of
// q_x/q_y/q_z.  The subtraction and product are done with _rn intrinsics so
// that no multiply-add contraction changes a key.
#include <algorithm>

#include "bh_internal.cuh"

namespace bh {
namespace {

constexpr int kBoxThreads = 256;

// Order-preserving map of a finite double's bits to an unsigned integer
// (negative values: all bits flipped; others: the sign bit set), so that the
// box's min/max are integer comparisons (the FP64 ones run at 1/64 of the
// FP32 rate here).  -0 orders below +0; the value selected is exact either way.
__device__ __forceinline__ unsigned long long ord_of(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double val_of(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7fffffffffffffffull) : ~k));
}

__device__ __forceinline__ void warp_minmax(unsigned long long& mn, unsigned long long& mx) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
}

// Per-block min/max of each axis of one patch -> 6 partials per block
// {mn x,y,z, mx x,y,z}.  Without a block map: patch blockIdx.y, its
// gridDim.x blocks, partials at q * gridDim.x + block.  With one (several
// patches of uneven sizes): block b works on patch map[b].x as its map[b].y-th
// of poff[q + 1] - poff[q] blocks (blocks in proportion to the patch sizes),
// partials at b.
__global__ void k_box_partial(const double* x, const double* y,
                              const double* z, const int64_t* off,
                              const uint2* map, const int* poff,
                              unsigned long long* part, int* status) {
    launch_wait();
    __shared__ unsigned long long s[6][kBoxThreads / 32];
    unsigned long long mn[3] = {~0ull, ~0ull, ~0ull}, mx[3] = {0ull, 0ull, 0ull};
    bool bad = false;
    int q, j, nbq;
    int64_t slot;
    if (map) {
        const uint2 e = map[blockIdx.x];
        q = (int)e.x;
        j = (int)e.y;
        nbq = poff[q + 1] - poff[q];
        slot = blockIdx.x;
    } else {
        q = blockIdx.y;
        j = blockIdx.x;
        nbq = gridDim.x;
        slot = (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
    }
    const int64_t e = off[q + 1];
    auto take = [&](const double (&v)[3]) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const unsigned long long b = (unsigned long long)__double_as_longlong(v[a]);
            bad |= ((b >> 52) & 0x7ffu) == 0x7ffu;  // infinity or NaN
            const unsigned long long k = ord_of(v[a]);
            mn[a] = min(mn[a], k);
            mx[a] = max(mx[a], k);
        }
    };
    const int64_t step = (int64_t)nbq * blockDim.x;
    int64_t i = off[q] + (int64_t)j * blockDim.x + threadIdx.x;
    for (; i + 3 * step < e; i += 4 * step) {  // twelve loads in flight
        double v[4][3];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[u][0] = x[i + u * step];
            v[u][1] = y[i + u * step];
            v[u][2] = z[i + u * step];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) take(v[u]);
    }
    for (; i < e; i += step) {
        const double v[3] = {x[i], y[i], z[i]};
        take(v);
    }
    if (bad) atomicOr(status, kStatNonFinite);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        warp_minmax(mn[a], mx[a]);
        if (lane == 0) {
            s[a][w] = mn[a];
            s[3 + a][w] = mx[a];
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        unsigned long long r = s[threadIdx.x][0];
        for (int k = 1; k < kBoxThreads / 32; ++k)
            r = threadIdx.x < 3 ? min(r, s[threadIdx.x][k]) : max(r, s[threadIdx.x][k]);
        part[6 * slot + threadIdx.x] = r;  // (as the ordered integer; a block with no particle keeps the identity)
    }
}

// box of patch q = blockIdx.x from its partials (nb per patch, or those of
// blocks poff[q] .. poff[q + 1] - 1): {lo_x, lo_y, lo_z, L, S} at box + 8 q.
// Cylindrical frame (cyl): every particle must be off the axis (r > 0), else
// kStatAxis.
__global__ void k_box_final(const unsigned long long* part_all, int nb, const int* poff,
                            double* box_all, int cyl, int* status) {
    launch_wait();
    const unsigned long long* part = part_all + 6 * (poff ? (int64_t)poff[blockIdx.x] : (int64_t)blockIdx.x * nb);
    if (poff) nb = poff[blockIdx.x + 1] - poff[blockIdx.x];
    double* box = box_all + 8 * blockIdx.x;
    __shared__ double r[6];
    {  // a warp per value
        const int a = threadIdx.x >> 5, lane = threadIdx.x & 31;
        unsigned long long mn = ~0ull, mx = 0ull;
        for (int b = lane; b < nb; b += 32) {
            const unsigned long long v = part[6 * b + a];
            mn = min(mn, v);
            mx = max(mx, v);
        }
        warp_minmax(mn, mx);
        if (lane == 0) r[a] = val_of(a < 3 ? mn : mx);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double ext = 0.0;
        for (int a = 0; a < 3; ++a) {
            box[a] = r[a];
            double e = __dsub_rn(r[3 + a], r[a]);
            if (e > ext) ext = e;
        }
        double L = ext > 0.0 ? ext : 1.0;
        box[3] = L;
        box[4] = __ddiv_rn(2097152.0, L);
        if (cyl && !(r[1] > 0.0)) atomicOr(status, kStatAxis);
    }
}

// Sec. 4.3: tree coordinates (phi, r, z) for a ring, phi and r as FP32
// numbers (a tree coordinate only has to place a particle within its key
// cell, 2^-21 of the box; the walk's contact clause has a margin for their
// error).  x, y rounded to FP32; phi from atan of the octant-reduced ratio,
// itself reduced to [0, tan(pi/12)] with
// atan(t) = pi/6 + atan((sqrt(3) t - 1) / (t + sqrt(3))) and summed as the
// Taylor series to u^11 (truncation below 3e-9 rad); r = sqrt(x^2 + y^2).
// Every operation is an IEEE-rounded FP32 +, -, *, / or sqrt in a fixed
// order, so phi is a deterministic function of (x, y), within 1e-6 rad of
// the true angle.
__device__ __forceinline__ float atan01(float t) {
    const float sqrt3 = 1.7320508075688772f, tan15 = 0.2679491924311227f, pi6 = 0.5235987755982988f;
    float base = 0.0f, u = t;
    if (t > tan15) {
        u = __fdiv_rn(__fsub_rn(__fmul_rn(t, sqrt3), 1.0f), __fadd_rn(t, sqrt3));
        base = pi6;
    }
    const float u2 = __fmul_rn(u, u);
    float p = -1.0f / 11.0f;
    p = __fadd_rn(__fmul_rn(p, u2), 1.0f / 9.0f);
    p = __fadd_rn(__fmul_rn(p, u2), -1.0f / 7.0f);
    p = __fadd_rn(__fmul_rn(p, u2), 1.0f / 5.0f);
    p = __fadd_rn(__fmul_rn(p, u2), -1.0f / 3.0f);
    p = __fadd_rn(__fmul_rn(p, u2), 1.0f);
    return __fadd_rn(base, __fmul_rn(u, p));
}

__global__ void k_cyl(const double* x, const double* y, int64_t n,
                      double* phi, double* r) {
    launch_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float X = __double2float_rn(x[i]), Y = __double2float_rn(y[i]);
    const float ax = fabsf(X), ay = fabsf(Y);
    const float mx = ax > ay ? ax : ay, mn = ax > ay ? ay : ax;
    float a = 0.0f;
    if (mx != 0.0f) {
        a = atan01(__fdiv_rn(mn, mx));
        if (ay > ax) a = __fsub_rn(1.5707963267948966f, a);
        if (X < 0.0f) a = __fsub_rn(3.141592653589793f, a);
        if (Y < 0.0f) a = __fsub_rn(6.283185307179586f, a);
    }
    phi[i] = (double)a;
    r[i] = (double)__fsqrt_rn(__fadd_rn(__fmul_rn(X, X), __fmul_rn(Y, Y)));
}

__device__ __forceinline__ uint64_t spread3(uint32_t v) {
    uint64_t x = v & kQMax;
    x = (x | (x << 32)) & 0x001f00000000ffffull;
    x = (x | (x << 16)) & 0x001f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// min(max(floor((v - lo) * S), 0), 2^21 - 1) with one FP64 subtraction, one
// product and one truncating conversion (truncation = floor for t >= 0); the
// clamps read the sign and the exponent of t.
__device__ __forceinline__ uint32_t quantise(double v, double lo, double S) {
    const double t = __dmul_rn(__dsub_rn(v, lo), S);
    const unsigned long long b = (unsigned long long)__double_as_longlong(t);
    if (b >> 63) return 0u;                                         // t < 0 (or -0)
    if (((b >> 52) & 0x7ffu) >= 1023u + kLevels) return kQMax;      // t >= 2^21 (infinities and NaN too)
    return min(__double2uint_rz(t), kQMax);
}

// Keys of every particle on its patch's grid (patch by binary search of the
// offsets).
__global__ void k_keys(const double* x, const double* y,
                       const double* z, int64_t n, const int64_t* off, int np,
                       const double* boxes, uint64_t* key) {
    launch_wait();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int q = 0;
    for (int lo = 0, hi = np - 1; lo < hi;) {  // last patch starting at or before i
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i)
            lo = q = mid;
        else
            hi = mid - 1;
    }
    const double* box = boxes + 8 * q;
    const double S = box[4];
    uint32_t qx = quantise(x[i], box[0], S), qy = quantise(y[i], box[1], S),
             qz = quantise(z[i], box[2], S);
    key[i] = (spread3(qx) << 2) | (spread3(qy) << 1) | spread3(qz);
}

// ---------------------------------------------------------------------------
// Radix sort: 8-bit digits, stable, one launch per digit (passes over bits
// [8p, 8p+8)) after one that counts all eight digits of every key.  A block
// takes the next tile (an atomic ticket, so every earlier tile has been taken
// by a running block), ranks its keys (ballots within a warp, per-warp digit
// counters), publishes its digit counts, reorders the keys by digit in shared
// memory, and finds the counts of all earlier tiles by looking back over the
// published words (a tile's own count, or the running total up to it) before
// the coalesced scatter: each pass reads and writes every key once, where
// counting, scanning and scattering launches read them twice.
// Stability: ranks follow (tile, warp, round, lane) = input order.
//
// Several patches (independent particle sets, each sorted on its own): tiles
// never straddle a patch, and the look-back of a tile ends at its patch's
// first.  tmeta holds per tile {first key, key count | digit-count slot << 13,
// first tile of its patch, tile count of its patch}; NULL means one patch cut
// into uniform tiles.  A patch of one tile needs no counts over the patch.
//
// Look-back words: digit pass + 1 in the top 4 bits (the words are cleared
// once per sort, so those of an earlier pass never match), a flag for a
// running total, and the count; 32 bits below 2^27 keys, else 64.  A look-back
// waits for a running block and ends after a bounded number of polls, with an error
// in the status word; every index it led to is checked against n, and the
// particles are then left as they were.
// (Decoupled look-back and one sweep per digit: Merrill and Garland 2016, Adinets and
// Merrill 2022; the code is this library's own.)
// Measured against counting, scanning and scattering launches (42 launches,
// and a host wait for the digit counts): 3,000,001 keys 469 -> 360 us, the
// evaluation of a 65,537-particle ring 860 -> 675 us.
// ---------------------------------------------------------------------------
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortTile = kSortThreads * kSortItems; // 4608
constexpr int kSlotShift = 13;                       // kSortTile < 2^13
constexpr int kSortHist = 8 * kRadix;                // digit counts per slot

struct TileInfo {
    int64_t start;  // first key of the tile
    int cnt;        // keys in the tile
    int slot;       // digit counts of its patch
    int first, nt;  // first tile and tile count of its patch
};

template <int ITEMS>
__device__ __forceinline__ TileInfo tile_info(const uint32_t* __restrict__ tmeta, int64_t n, int ntiles, int t) {
    TileInfo ti;
    if (tmeta) {
        const uint4 m = reinterpret_cast<const uint4*>(tmeta)[t];
        ti.start = m.x;
        ti.cnt = (int)(m.y & ((1u << kSlotShift) - 1u));
        ti.slot = (int)(m.y >> kSlotShift);
        ti.first = (int)m.z;
        ti.nt = (int)m.w;
    } else {
        constexpr int tile = kSortThreads * ITEMS;
        ti.start = (int64_t)t * tile;
        const int64_t r = n - ti.start;
        ti.cnt = (int)(r < tile ? r : tile);
        ti.slot = 0;
        ti.first = 0;
        ti.nt = ntiles;
    }
    return ti;
}

// Digit counts of every pass, per patch of more than one tile: hist[slot][pass][digit].
template <int ITEMS>
__global__ void __launch_bounds__(256) k_digit_hist(const uint64_t* key, int64_t n, int ntiles,
                                                    const uint32_t* tmeta, uint32_t* hist) {
    launch_wait();
    __shared__ uint32_t h[8][kRadix];
    const int per = (ntiles + gridDim.x - 1) / gridDim.x;
    const int t0 = blockIdx.x * per, t1 = min(t0 + per, ntiles);
    int slot = -1;
    auto flush = [&]() {
        __syncthreads();
        if (slot >= 0)
            for (int i = threadIdx.x; i < kSortHist; i += blockDim.x)
                if ((&h[0][0])[i]) atomicAdd(&hist[(int64_t)slot * kSortHist + i], (&h[0][0])[i]);
        __syncthreads();
        for (int i = threadIdx.x; i < kSortHist; i += blockDim.x) (&h[0][0])[i] = 0;
        __syncthreads();
    };
    for (int t = t0; t < t1; ++t) {
        const TileInfo ti = tile_info<ITEMS>(tmeta, n, ntiles, t);
        if (ti.nt == 1) continue;
        if (ti.slot != slot) {
            flush();
            slot = ti.slot;
        }
#pragma unroll 6
        for (int i = threadIdx.x; i < ti.cnt; i += 256) {
            const uint64_t k = key[ti.start + i];
#pragma unroll
            for (int p = 0; p < 8; ++p) atomicAdd(&h[p][(k >> (8 * p)) & 0xff], 1u);
        }
    }
    if (slot >= 0) flush();
}

template <class W>
struct Look {
    static constexpr int kTag = 8 * sizeof(W) - 4;
    static constexpr W kTotal = (W)1 << (kTag - 1), kCount = kTotal - 1;
    __device__ __forceinline__ static W load(const W* p) {
        W v;
        if constexpr (sizeof(W) == 4)
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        else
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
        return v;
    }
    __device__ __forceinline__ static void store(W* p, W v) {
        if constexpr (sizeof(W) == 4)
            asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
        else
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
    }
};

template <int ITEMS>
struct SweepSmem {
    uint32_t whist[kSortWarps][kRadix];
    uint32_t tstart[kRadix];
    uint32_t goff[kRadix];
    unsigned long long wtot[kRadix / 32];
    int tile;
    union {
        uint64_t skey[kSortThreads * ITEMS];
        uint32_t sidx[kSortThreads * ITEMS];
    };
};

// FIRST: the index of a key is its position (iin is not read).
template <class W, bool FIRST, int ITEMS>
__global__ void __launch_bounds__(kSortThreads, 3) k_sweep(
    const uint64_t* kin, const uint32_t* iin, int64_t n, int pass, int ntiles,
    const uint32_t* tmeta, const uint32_t* hist, W* words, uint32_t* ticket,
    uint64_t* kout, uint32_t* iout, int most_polls, int* status) {
    launch_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SweepSmem<ITEMS>& S = *reinterpret_cast<SweepSmem<ITEMS>*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, shift = 8 * pass;
    if (tid == 0) S.tile = (int)atomicAdd(ticket, 1u);
    for (int i = tid; i < kSortWarps * kRadix; i += kSortThreads) (&S.whist[0][0])[i] = 0;
    __syncthreads();
    const int tile = S.tile;
    const TileInfo ti = tile_info<ITEMS>(tmeta, n, ntiles, tile);
    const int wbase = w * (32 * ITEMS);
    const unsigned lt = (1u << lane) - 1u;
    uint64_t kr[ITEMS];
    uint32_t pr[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int pos = wbase + r * 32 + lane;
        kr[r] = pos < ti.cnt ? kin[ti.start + pos] : ~0ull;
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const bool valid = wbase + r * 32 + lane < ti.cnt;
        const uint32_t d = (uint32_t)(kr[r] >> shift) & 0xffu;
        unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const bool bit = (d >> b) & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? m : ~m;
        }
        const uint32_t old = S.whist[w][d];
        __syncwarp();
        if (valid && (peers & lt) == 0) S.whist[w][d] = old + __popc(peers);
        __syncwarp();
        pr[r] = old + __popc(peers & lt);
    }
    __syncthreads();
    // per digit: exclusive over warps; tile count; exclusive over digits (of
    // the tile, and of the patch)
    W* mine = words + (int64_t)tile * kRadix;
    const W tag = (W)(pass + 1) << Look<W>::kTag;
    uint32_t total = 0, base = 0;
    unsigned long long x = 0, own = 0;
    if (tid < kRadix) {
#pragma unroll
        for (int ww = 0; ww < kSortWarps; ++ww) {
            const uint32_t t = S.whist[ww][tid];
            S.whist[ww][tid] = total;
            total += t;
        }
        if (ti.nt > 1)
            Look<W>::store(&mine[tid], tag | (tile == ti.first ? Look<W>::kTotal : (W)0) | (W)total);
        const uint32_t hc = ti.nt > 1 ? hist[(int64_t)ti.slot * kSortHist + pass * kRadix + tid] : total;
        own = (unsigned long long)hc << 32 | total;
        x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) S.wtot[w] = x;
    }
    __syncthreads();
    if (tid < kRadix) {
        x -= own;
        for (int ww = 0; ww < w; ++ww) x += S.wtot[ww];
        S.tstart[tid] = (uint32_t)x;
        base = (uint32_t)(x >> 32);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
        if (wbase + r * 32 + lane < ti.cnt) {
            const uint32_t d = (uint32_t)(kr[r] >> shift) & 0xffu;
            pr[r] += S.tstart[d] + S.whist[w][d];
            S.skey[pr[r]] = kr[r];
        }
    if (tid < kRadix) {
        W excl = 0;
        if (tile > ti.first) {
            // eight earlier tiles' words at a time, so that their loads overlap:
            // the tiles that start together all look back over each other
            // (3,000,001 keys: one at a time 358 us, eight 349, 32 400)
            constexpr int LB = 8;
            int left = most_polls;
            bool done = left == 0;  // (0: the wait runs out before it begins)
            for (int t = tile - 1; !done;) {
                W v[LB];
#pragma unroll
                for (int u = 0; u < LB; ++u)
                    v[u] = t - u >= ti.first ? Look<W>::load(&words[(int64_t)(t - u) * kRadix + tid]) : (W)0;
                int got = 0;
#pragma unroll
                for (int u = 0; u < LB; ++u)
                    if (got == u && !done && v[u] >> Look<W>::kTag == (W)(pass + 1)) {
                        excl += v[u] & Look<W>::kCount;
                        done = (v[u] & Look<W>::kTotal) != 0;  // (the patch's first tile has it)
                        got = u + 1;
                    }
                t -= got;
                if (got == 0 && --left == 0) done = true;  // (the earlier tile is running: never)
            }
            if (left == 0) atomicOr(status, kStatTimeout);
            Look<W>::store(&mine[tid], tag | Look<W>::kTotal | (excl + (W)total));
        }
        // the patch's first output is its first key's position
        const int64_t p0 = tmeta ? ti.start - (int64_t)(tile - ti.first) * (kSortThreads * ITEMS) : 0;
        S.goff[tid] = (uint32_t)p0 + base + (uint32_t)excl - S.tstart[tid];
    }
    __syncthreads();
    uint32_t g[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int q = r * kSortThreads + tid;
        g[r] = 0xffffffffu;
        if (q < ti.cnt) {
            const uint64_t k = S.skey[q];
            g[r] = S.goff[(uint32_t)(k >> shift) & 0xffu] + (uint32_t)q;
            if ((int64_t)g[r] < n) kout[g[r]] = k;  // (past it only after a look-back that gave up)
        }
    }
    uint32_t ir[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const int pos = wbase + r * 32 + lane;
        ir[r] = FIRST ? (uint32_t)(ti.start + pos) : pos < ti.cnt ? iin[ti.start + pos] : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
        if (wbase + r * 32 + lane < ti.cnt) S.sidx[pr[r]] = ir[r];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
        if ((int64_t)g[r] < n) iout[g[r]] = S.sidx[r * kSortThreads + tid];
}

// Sort (key[0]) into (key[0], idx[0]): eight passes, the first one numbering
// the keys by position.
template <class W, int ITEMS>
cudaError_t sort_passes(cudaStream_t s, bool early, uint64_t* const (&kb)[2], uint32_t* const (&ib)[2], int64_t n,
                        const uint32_t* tmeta, int ntiles, int nslots, int num_sms, uint32_t* scratch, SortLimits lim,
                        int* status) {
    const SortScratch z = sort_scratch(n, ntiles, nslots, lim.wide_from);
    W* words = reinterpret_cast<W*>(scratch);
    uint32_t* hist = scratch + z.words;
    uint32_t* ticket = hist + (int64_t)nslots * kSortHist;
    cudaError_t e = cudaMemsetAsync(scratch, 0, (size_t)z.total * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    if (nslots > 0) {
        const int nb = std::min(ntiles, 4 * num_sms);
        e = launch_on(s, early, k_digit_hist<ITEMS>, nb, 256, 0, kb[0], n, ntiles, tmeta, hist);
        if (e != cudaSuccess) return e;
    }
    const int smem = (int)sizeof(SweepSmem<ITEMS>);
    for (int pass = 0; pass < 8; ++pass) {
        const int a = pass & 1, b = 1 - a;
        auto kern = pass == 0 ? k_sweep<W, true, ITEMS> : k_sweep<W, false, ITEMS>;
        e = launch_on(s, early, kern, ntiles, kSortThreads, smem, kb[a], ib[a], n, pass, ntiles, tmeta, hist, words,
                      ticket + pass, kb[b], ib[b], lim.polls, status);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t sort_any(cudaStream_t s, bool early, uint64_t* const (&kb)[2], uint32_t* const (&ib)[2], int64_t n,
                     const uint32_t* tmeta, int ntiles, int nslots, int num_sms, uint32_t* scratch, SortLimits lim,
                     int* status) {
    auto run = n >= lim.wide_from               ? sort_passes<unsigned long long, kSortItems>
               : !tmeta && small_tiles(n, lim.wide_from) ? sort_passes<uint32_t, kSortSmallItems>
                                                : sort_passes<uint32_t, kSortItems>;
    return run(s, early, kb, ib, n, tmeta, ntiles, nslots, num_sms, scratch, lim, status);
}
constexpr int kSortLaunches = 9;  // kernels of one sort

// All particle arrays (8-byte elements) gathered into key order in one pass:
// the permutation is read once and every array's load is in flight at once;
// into scratch + a n, then copied back to dst[a] (the same arrays).
struct Gather8 {
    const unsigned long long* src[8];
    unsigned long long* dst[8];
    int na;
    const int* stop;  // status word: with one of stop_bits in it the particles stay as they are
    int stop_bits;
};

__global__ void k_gather_all(Gather8 G, unsigned long long* scratch, const uint32_t* perm,
                             int64_t n, int* status) {
    launch_wait();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || (*G.stop & G.stop_bits)) return;
    const uint32_t j = perm[i];
    if (j >= n) {
        atomicOr(status, kStatBounds);
        return;
    }
    unsigned long long v[8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
        if (a < G.na) v[a] = G.src[a][j];
#pragma unroll
    for (int a = 0; a < 8; ++a)
        if (a < G.na) scratch[(int64_t)a * n + i] = v[a];
}

// The gathered arrays back into place (one launch; eight copies of a small
// set's arrays cost their launches).
__global__ void k_copy_back(Gather8 G, const unsigned long long* scratch, int64_t n) {
    launch_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || (*G.stop & G.stop_bits)) return;
    unsigned long long v[8];
#pragma unroll
    for (int a = 0; a < 8; ++a)
        if (a < G.na) v[a] = scratch[(int64_t)a * n + i];
#pragma unroll
    for (int a = 0; a < 8; ++a)
        if (a < G.na) G.dst[a][i] = v[a];
}

}  // namespace

// Root box and keys of each patch (one patch: the whole set).  idx holds
// global particle indices.
int stage_keys(Ctx* c, const bh_particles* p) {
    const int64_t n = c->n;
    const int nbmax = c->num_sms * 4;
    for (int b = 0; b < 2; ++b) {
        BH_TRY(grow(c, c->key[b], (size_t)n, "keys"));
        BH_TRY(grow(c, c->idx[b], (size_t)n, "sort indices"));
    }
    // tree coordinates: (x, y, z), or (phi, r, z) in the cylindrical frame
    const double *cx = p->x, *cy = p->y;
    if (c->prm.key_frame == 1) {
        BH_TRY(grow(c, c->cyl, 2 * (size_t)n, "cylindrical coordinates"));
        BH_CUDA(c, launch(c, k_cyl, blocks_for(n, 256), 256, 0, p->x, p->y, n, c->cyl.p, c->cyl.p + n));
        BH_LAUNCH(c);
        cx = c->cyl.p;
        cy = c->cyl.p + n;
    }
    // all patches at once: blocks for the boxes (in proportion to the patch
    // sizes when there are several), then one pass for the keys
    const int np = c->n_patches;
    if (np > 1) {
        const int nbt = c->n_box_blocks;
        BH_TRY(grow(c, c->box_part, 6 * (size_t)nbt, "box partials"));
        BH_CUDA(c, launch(c, k_box_partial, nbt, kBoxThreads, 0, cx, cy, p->z, c->d_off.p, c->box_map.p,
                          c->box_poff.p, c->box_part.p, c->d_status));
        BH_LAUNCH(c);
        BH_CUDA(c, launch(c, k_box_final, np, 6 * 32, 0, c->box_part.p, 0, c->box_poff.p, c->d_box,
                          c->prm.key_frame == 1, c->d_status));
        BH_LAUNCH(c);
    } else {
        const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(nbmax, blocks_for(n, 4 * kBoxThreads)));
        BH_TRY(grow(c, c->box_part, 6 * (size_t)nb, "box partials"));
        BH_CUDA(c, launch(c, k_box_partial, nb, kBoxThreads, 0, cx, cy, p->z, c->d_off.p, nullptr, nullptr,
                          c->box_part.p, c->d_status));
        BH_LAUNCH(c);
        BH_CUDA(c, launch(c, k_box_final, 1, 6 * 32, 0, c->box_part.p, nb, nullptr, c->d_box,
                          c->prm.key_frame == 1, c->d_status));
        BH_LAUNCH(c);
    }
    BH_CUDA(c, launch(c, k_keys, blocks_for(n, 256), 256, 0, cx, cy, p->z, n, c->d_off.p, np, c->d_box,
                      c->key[0].p));
    BH_LAUNCH(c);
    c->key_cur = 0;
    return BH_OK;
}

// Tiles of the context's sort, and digit-count slots.
static void sort_shape(const Ctx* c, int* ntiles, int* nslots) {
    const bool batch = c->n_patches > 1;
    *ntiles = batch ? (int)c->n_tiles : (int)sort_tiles(c->n, c->sort_limits.wide_from);
    *nslots = batch ? c->n_sort_slots : *ntiles > 1 ? 1 : 0;
}

int reserve_sort(Ctx* c) {
    int ntiles, nslots;
    sort_shape(c, &ntiles, &nslots);
    const SortScratch z = sort_scratch(c->n, ntiles, nslots, c->sort_limits.wide_from);
    return grow(c, c->sort_scratch, (size_t)z.total, "sort scratch");
}

int stage_sort(Ctx* c) {
    const int64_t n = c->n;
    const uint32_t* tmeta = c->n_patches > 1 ? c->tile_meta.p : nullptr;
    int ntiles, nslots;
    sort_shape(c, &ntiles, &nslots);
    BH_TRY(reserve_sort(c));
    if (c->sort_attr_device != c->device) {  // once per device
        BH_CUDA(c, sort_setup_device());
        c->sort_attr_device = c->device;
    }
    uint64_t* const kb[2] = {c->key[0].p, c->key[1].p};
    uint32_t* const ib[2] = {c->idx[0].p, c->idx[1].p};
    BH_CUDA(c, sort_any(c->stream, !c->capturing, kb, ib, n, tmeta, ntiles, nslots, c->num_sms, c->sort_scratch.p,
                        c->sort_limits, c->d_status));
    c->n_launches += kSortLaunches - (nslots > 0 ? 0 : 1);
    c->key_cur = 0;
    return BH_OK;
}

int stage_permute(Ctx* c, bh_particles* p) {
    const int64_t n = c->n;
    BH_TRY(grow(c, c->pscratch, 8 * (size_t)n, "particle scratch"));
    unsigned long long* arrs[8] = {(unsigned long long*)p->x,  (unsigned long long*)p->y,
                                   (unsigned long long*)p->z,  (unsigned long long*)p->vx,
                                   (unsigned long long*)p->vy, (unsigned long long*)p->vz,
                                   (unsigned long long*)p->m,  (unsigned long long*)p->id};
    const uint32_t* perm = c->idx[c->key_cur].p;
    Gather8 G = {};
    // (a captured step goes on with any other error in the word: it is one of before the step)
    G.stop = c->d_status;
    G.stop_bits = c->dev_build ? kStatTimeout : ~0;
    for (int a = 0; a < 8; ++a)
        if (arrs[a]) {
            G.dst[G.na] = arrs[a];
            G.src[G.na++] = arrs[a];
        }
    unsigned long long* scratch = (unsigned long long*)c->pscratch.p;
    BH_CUDA(c, launch(c, k_gather_all, blocks_for(n, 256), 256, 0, G, scratch, perm, n, c->d_status));
    BH_LAUNCH(c);
    BH_CUDA(c, launch(c, k_copy_back, blocks_for(n, 256), 256, 0, G, scratch, n));
    BH_LAUNCH(c);
    return BH_OK;
}

// Sort tiles of the patches: 4 words per tile (see k_sweep); *nslots = patches
// of more than one tile.
int64_t sort_tiles_for(const std::vector<int64_t>& off, std::vector<uint32_t>* meta, int* nslots) {
    int64_t t = 0;
    *nslots = 0;
    for (size_t q = 0; q + 1 < off.size(); ++q) {
        const int64_t np = off[q + 1] - off[q], nt = (np + kSortTile - 1) / kSortTile, t0 = t;
        const uint32_t slot = nt > 1 ? (uint32_t)(*nslots)++ : 0u;
        for (int64_t u = 0; u < nt; ++u, ++t) {
            const int64_t st = off[q] + u * kSortTile, r = off[q + 1] - st;
            meta->push_back((uint32_t)st);
            meta->push_back((uint32_t)(r < kSortTile ? r : kSortTile) | slot << kSlotShift);
            meta->push_back((uint32_t)t0);
            meta->push_back((uint32_t)nt);
        }
    }
    return t;
}

cudaError_t sort_setup_device() {
    // (the small tiles need less than the default limit)
    const int smem = (int)sizeof(SweepSmem<kSortItems>);
    static_assert(sizeof(SweepSmem<kSortSmallItems>) <= 48 * 1024, "default shared-memory limit");
    const void* kerns[4] = {(const void*)k_sweep<uint32_t, true, kSortItems>,
                            (const void*)k_sweep<uint32_t, false, kSortItems>,
                            (const void*)k_sweep<unsigned long long, true, kSortItems>,
                            (const void*)k_sweep<unsigned long long, false, kSortItems>};
    for (const void* k : kerns) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Context-free form of stage_sort for callers that supply every buffer,
// ending in (keys, idx) again; nothing here synchronises.
cudaError_t sort_pairs_with(cudaStream_t s, uint64_t* keys, uint32_t* idx, uint64_t* ktmp, uint32_t* itmp,
                            int64_t n, int num_sms, uint32_t* scratch, int polls, int* status) {
    if (n <= 0) return cudaSuccess;
    const int ntiles = (int)sort_tiles(n, kSortWide);
    uint64_t* const kb[2] = {keys, ktmp};
    uint32_t* const ib[2] = {idx, itmp};
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;  // (a caller may be capturing its stream)
    const cudaError_t e = cudaStreamIsCapturing(s, &st);
    if (e != cudaSuccess) return e;
    return sort_any(s, st == cudaStreamCaptureStatusNone, kb, ib, n, nullptr, ntiles, ntiles > 1 ? 1 : 0, num_sms,
                    scratch, {kSortWide, polls}, status);
}

}  // namespace bh
