// force.cu -- Sec. 4.2 step 3d, second half: the double loop over the
// particles of a group and the entries of its shared interaction list.
//
//   list particles: Eq. (1) read as an acceleration (gravity G m_j r/r^3,
//                   softened by eps, held at its r_coll value inside r_coll,
//                   plus the spring/dashpot contact term inside r_coll);
//   list cells:     centre-of-mass monopole (Sec. 5.1) and, for order 2, the
//                   traceless quadrupole about the centre of mass.
//
// This file: the plain FP64 kernels (absolute coordinates) of the force and
// of the self-gravity potential, the FP32 hi/lo split on its own
// (bh_split_f32), and the dispatcher.  Pairs that may be in
// contact (r^2 <= r_coll^2 up to rounding) are re-evaluated in the oracle's
// exact operation order, so the r <= r_coll decision is the oracle's.
#include <algorithm>
#include <cmath>

#include "force_common.cuh"
#include "split32.cuh"

namespace bh {
namespace {

constexpr int kWarps = 4;

struct __align__(16) D4 {
    double x, y, z, w;
};

struct Smem64 {
    union {
        struct {
            D4 pj[32];
            uint32_t jid[32];
        } p;
        double cl[32][10];  // M, c3, Q6
    };
};

struct Args64 {
    int64_t ng;
    const unsigned long long* dng;    // device group count (device-sized list builds; NULL: ng)
    const unsigned long long* abort;  // nonzero: that build outgrew its buffers, nothing is done
    const int32_t* groups;
    const uint32_t *begin, *end;
    const int64_t* jj_off;
    const uint32_t* JJ;
    const int64_t* pc_off;
    const int32_t* C;
    const double *x, *y, *z, *vx, *vy, *vz, *m;
    const double *M, *cx, *cy, *cz, *Q;
    ForceParams fp;
    bool add_central;
    double *ax, *ay, *az;  // force
    double* phi;           // potential
    uint32_t n;
    int64_t nn;
    int* status;
    const int64_t* off;    // patches: particle offsets (np + 1)
    int np, n_g, slots;    // item slots per group
};

// Items of a group (see item64): log2 of the largest, by the size of the
// particle set alone (a patch's sums are then those of the patch alone):
// smaller items give a small set's SMs more to share, at the price of staging
// the lists more often.  Measured, a force evaluation with 1, 2, 4, 8 and 16
// particles: 16,384-particle cube 694, 715, 788, 915, 1207 us; 20,000-particle
// ring 460, 441, 452, 507, 573 us; 65,537: 1344, 1246, 1227, 1263, 1366 us;
// 2^20: 27.7, 26.0, 25.2, 24.9, 24.9 ms.
__host__ __device__ __forceinline__ int item_lcap(int64_t n) {
    return n >= 80000 ? 3 : n >= 40000 ? 2 : n >= 20000 ? 1 : 0;
}
__host__ __device__ __forceinline__ int whole_items(int n_g, int lcap) { return n_g >> lcap > 1 ? n_g >> lcap : 1; }

// ---- 1 / sqrt(s) -----------------------------------------------------------
// The FP64 pipe (2 lanes per clock and SM: one warp instruction takes it 16
// cycles) bounds these kernels; the integer and FP32 pipes idle beside it.
// So the inverse square root and its powers are taken from a hardware
// estimate y0 (21 significant bits) by the binomial series of
// s^(-k/2) = y0^k (1 - e)^(-k/2), e = 1 - s y0^2 (|e| <= 2^-18 or so):
//   (1 - e)^(-1/2) = 1 + e/2 + 3/8 e^2 + O(e^3),
//   (1 - e)^(-3/2) = 1 + 3/2 e + 15/8 e^2 + O(e^3)
// with y0^2 exact (42 bits, squared as an integer), e exact to one rounding
// (FMA), and the e^2 term, below 2^-36, in FP32: what is left out is below
// 2^-53 of the result.  One FP64 comparison, conversion or product saved is
// worth 30 integer instructions here.
struct RSeed {
    double y0, a, e;  // estimate, its square, 1 - s y0^2
    double q;         // kq e^2
};

// Whether s is far enough from overflow and underflow for the series (its
// powers included); else the callers take the library functions.
__device__ __forceinline__ bool rseed_ok(double s) {
    return (uint32_t)((__double2hiint(s) >> 20) - 423) < 1200u;  // 2^-600 <= s < 2^600
}

__device__ __forceinline__ RSeed rseed(double s, float kq) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(s));
    const uint32_t h = (uint32_t)__double2hiint(y);
    RSeed r;
    r.y0 = __hiloint2double((int)h, 0);
    const uint32_t m = (h & 0xfffffu) | 0x100000u;
    const uint64_t sq = (uint64_t)m * m;  // in [2^40, 2^42)
    const uint32_t p = (uint32_t)(sq >> 41);
    r.a = __longlong_as_double((long long)(((uint64_t)(2u * (h >> 20) - 1024u + p) << 52) + (sq << (12 - p))));
    r.e = fma(-s, r.a, 1.0);
    // kq e^2 in FP32, by integer conversions (the FP64 ones take the FP64 pipe);
    // an e below 2^-126 counts as that
    const uint32_t eh = max((uint32_t)__double2hiint(r.e) & 0x7fffffffu, 897u << 20);
    const float ef = __uint_as_float((eh - (896u << 20)) << 3);
    const uint32_t qb = __float_as_uint(__fmul_rn(__fmul_rn(kq, ef), ef));
    r.q = __hiloint2double((int)((qb >> 3) + (896u << 20)), (int)(qb << 29));
    return r;
}

// m s^(-3/2)
__device__ __forceinline__ double inv_cube(double m, double s) {
    if (!rseed_ok(s)) {
        const double ri = rsqrt(s);
        return m * ri * ri * ri;
    }
    const RSeed r = rseed(s, 1.875f);
    const double f0 = (m * r.y0) * r.a;
    return fma(f0, fma(1.5, r.e, r.q), f0);
}

// s^(-1/2)
__device__ __forceinline__ double inv_sqrt(double s) {
    if (!rseed_ok(s)) return rsqrt(s);
    const RSeed r = rseed(s, 0.375f);
    return fma(r.y0, fma(0.5, r.e, r.q), r.y0);
}

// x / 2 without the FP64 pipe (except for subnormal results).
__device__ __forceinline__ double half_of(double x) {
    const uint32_t h = (uint32_t)__double2hiint(x), e = (h >> 20) & 0x7ffu;
    if (e - 2u < 0x7fdu) return __hiloint2double((int)(h - (1u << 20)), __double2loint(x));
    return 0.5 * x;
}

// ---- the kernels -----------------------------------------------------------
// Sum over the group's own particles and its list particles, then its list
// cells, for one item of a group: 2^k of its particles whose list is split
// over 32 / 2^k lanes each.  A group of n_i particles is cut along the binary
// digits of n_i (62 = 7 x 8 + 4 + 2), so every lane has a particle and the
// FP64 pipe does no work for padding (32-lane chunks left 26% of it idle for
// the 2^20 ring's groups, more than half for groups of 8 to 20).  A warp per
// item; list entries staged 32 at a time in shared memory, the next
// 32 loaded while these are evaluated.  Measured against one warp per group
// in 32-lane chunks with rsqrt(), sqrt() and divisions: force evaluation of a
// 2^17 ring 6.07 -> 2.78 ms (62.8e6 -> 38.8e6 FP64 warp instructions, pipe 53
// -> 71% busy), of the 2^20 ring 39.9 -> 24.2 ms, potential of a 2^18 ring
// 13.5 -> 3.8 ms, force evaluation of a 4096-particle cube 2.3 -> 0.2 ms.
// Against sums in 80 bits the accelerations of that cube went from 9.3e-16 to
// 1.6e-16 (relative 2-norm), of a 20,000-particle ring with quadrupoles and
// contacts from 8.5e-16 to 2.2e-16, the potentials from 6.8e-16 to 0.8e-16 and from
// 4.5e-16 to 0.9e-16: shorter sums, and the series instead of three roundings.
template <bool POT, int ORDER, bool EPS>
__device__ __forceinline__ void item64(const Args64& A, Smem64& S, int64_t k, uint32_t b, uint32_t e, uint32_t i0,
                                       int lsz, int lane) {
    const ForceParams& fp = A.fp;
    const int nsp = 32 >> lsz;
    const int s = lane >> lsz;
    const uint32_t i = i0 + (uint32_t)(lane & ((1 << lsz) - 1));
    const double xi = A.x[i], yi = A.y[i], zi = A.z[i];
    double g0 = 0.0, g1 = 0.0, g2 = 0.0;     // G-free sums (potential: g0)
    double an[3] = {0.0, 0.0, 0.0};          // pairs evaluated exactly, G included
    const long long rc2_hi = __double_as_longlong(fp.rc2_hi), rc2 = __double_as_longlong(fp.rc2);
    const double inv_sc = POT && fp.rc2 + fp.eps2 > 0.0 ? 1.0 / sqrt(fp.rc2 + fp.eps2) : 0.0;
    const double half_sc3 = 0.5 * inv_sc * inv_sc * inv_sc;
    {
        const int64_t j0 = A.jj_off[k], own = (int64_t)(e - b), tot = own + (A.jj_off[k + 1] - j0);
        auto index = [&](int64_t t) -> uint32_t {
            if (t < own) return b + (uint32_t)t;
            if (t >= tot) return b;
            const uint32_t j = A.JJ[j0 + t - own];
            if (j < A.n) return j;
            atomicOr(A.status, kStatBounds);
            return b;
        };
        auto load = [&](uint32_t j) { return D4{A.x[j], A.y[j], A.z[j], A.m[j]}; };
        uint32_t j = index(lane), jn = index(lane + 32);
        D4 d = load(j);
        for (int64_t t0 = 0; t0 < tot; t0 += 32) {
            S.p.pj[lane] = d;
            S.p.jid[lane] = j;
            __syncwarp();
            j = jn;
            d = load(j);
            jn = index(t0 + 64 + lane);
            const int nt = (int)min((int64_t)32, tot - t0);
            for (int q = s; q < nt; q += nsp) {
                const D4 pj = S.p.pj[q];
                const double dx = pj.x - xi, dy = pj.y - yi, dz = pj.z - zi;
                const double r2 = dx * dx + dy * dy + dz * dz;
                const long long rb = __double_as_longlong(r2);  // r2 >= 0: orders as its bits
                if (POT) {
                    if (rb > rc2) {
                        g0 = fma(-pj.w, inv_sqrt(EPS ? r2 + fp.eps2 : r2), g0);
                    } else if (rb != 0 && S.p.jid[q] != i) {
                        g0 -= pj.w * inv_sc + pj.w * (fp.rc2 - r2) * half_sc3;
                    }
                } else {
                    if (rb > rc2_hi) {
                        const double f = inv_cube(pj.w, EPS ? r2 + fp.eps2 : r2);
                        g0 = fma(f, dx, g0);
                        g1 = fma(f, dy, g1);
                        g2 = fma(f, dz, g2);
                    } else {
                        const uint32_t jq = S.p.jid[q];
                        if (jq != i)
                            exact_pair64(fp, xi, yi, zi, A.vx[i], A.vy[i], A.vz[i], A.m[i], pj.x, pj.y, pj.z, A.vx[jq],
                                         A.vy[jq], A.vz[jq], pj.w, an);
                    }
                }
            }
            __syncwarp();
        }
    }
    {
        const int64_t c0 = A.pc_off[k], c1 = A.pc_off[k + 1];
        constexpr int NC = ORDER >= 2 ? 10 : 4;
        auto index = [&](int64_t t) -> int32_t {
            if (t >= c1) return 0;
            const int32_t cc = A.C[t];
            if (cc >= 0 && cc < A.nn) return cc;
            atomicOr(A.status, kStatBounds);
            return 0;
        };
        double v[NC];
        auto load = [&](int32_t cc) {
            v[0] = A.M[cc];
            v[1] = A.cx[cc];
            v[2] = A.cy[cc];
            v[3] = A.cz[cc];
            if (ORDER >= 2) {
                const double2* Q = reinterpret_cast<const double2*>(A.Q) + 3 * (int64_t)cc;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const double2 u = Q[a];
                    v[NC - 6 + 2 * a] = u.x;
                    v[NC - 5 + 2 * a] = u.y;
                }
                if (POT)  // half the diagonal: d.Qd / 2 then takes 9 operations instead of 13
#pragma unroll
                    for (int a = 0; a < 3; ++a) v[NC - 6 + a] = half_of(v[NC - 6 + a]);
            }
        };
        int32_t cn = index(c0 + lane);
        load(cn);
        cn = index(c0 + 32 + lane);
        for (int64_t t0 = c0; t0 < c1; t0 += 32) {
#pragma unroll
            for (int a = 0; a < NC; ++a) S.cl[lane][a] = v[a];
            __syncwarp();
            load(cn);
            cn = index(t0 + 64 + lane);
            const int nt = (int)min((int64_t)32, c1 - t0);
            for (int q = s; q < nt; q += nsp) {
                const double* cl = S.cl[q];
                const double dx = cl[1] - xi, dy = cl[2] - yi, dz = cl[3] - zi;  // d = c - x_i = -R
                const double R2 = EPS ? fma(dx, dx, fma(dy, dy, fma(dz, dz, fp.eps2))) : dx * dx + dy * dy + dz * dz;
                if (ORDER < 2) {
                    if (POT) {
                        g0 = fma(-cl[0], inv_sqrt(R2), g0);
                    } else {
                        const double f = inv_cube(cl[0], R2);
                        g0 = fma(f, dx, g0);
                        g1 = fma(f, dy, g1);
                        g2 = fma(f, dz, g2);
                    }
                    continue;
                }
                const double ri = inv_sqrt(R2), ri2 = ri * ri;
                if (POT) {  // -(M + (d.Qd) / (2 R^4)) / R
                    const double hq = dx * (cl[NC - 6] * dx + cl[NC - 3] * dy + cl[NC - 2] * dz) +
                                      dy * (cl[NC - 5] * dy + cl[NC - 1] * dz) + dz * (cl[NC - 4] * dz);
                    g0 = fma(-ri, fma(hq, ri2 * ri2, cl[0]), g0);
                } else {    // ((M R^2 + 5/2 (d.Qd) / R^2) d - Q d) / R^5
                    const double qx = cl[NC - 6] * dx + cl[NC - 3] * dy + cl[NC - 2] * dz;
                    const double qy = cl[NC - 3] * dx + cl[NC - 5] * dy + cl[NC - 1] * dz;
                    const double qz = cl[NC - 2] * dx + cl[NC - 1] * dy + cl[NC - 4] * dz;
                    const double dqd = dx * qx + dy * qy + dz * qz;
                    const double ri5 = ri2 * ri2 * ri;
                    const double w = fma(2.5, dqd * ri2, cl[0] * R2);
                    g0 = fma(ri5, fma(w, dx, -qx), g0);
                    g1 = fma(ri5, fma(w, dy, -qy), g1);
                    g2 = fma(ri5, fma(w, dz, -qz), g2);
                }
            }
            __syncwarp();
        }
    }
    if (POT) {
        for (int o = 1 << lsz; o < 32; o <<= 1) g0 += __shfl_xor_sync(0xffffffffu, g0, o);
        if (s == 0) A.phi[i] = fp.G * g0;
        return;
    }
    double a[3] = {fma(fp.G, g0, an[0]), fma(fp.G, g1, an[1]), fma(fp.G, g2, an[2])};
    for (int o = 1 << lsz; o < 32; o <<= 1)
#pragma unroll
        for (int c = 0; c < 3; ++c) a[c] += __shfl_xor_sync(0xffffffffu, a[c], o);
    if (s != 0) return;
    if (A.add_central) central64(fp.GMc, xi, yi, zi, a);
    A.ax[i] = a[0];
    A.ay[i] = a[1];
    A.az[i] = a[2];
}

template <bool POT, int ORDER, bool EPS>
__global__ void __launch_bounds__(32 * kWarps) k_sum64(const Args64 A) {
    launch_wait();
    __shared__ Smem64 sm[kWarps];
    if (A.abort && *A.abort) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t ng = A.dng ? min(A.ng, (int64_t)*A.dng) : A.ng;
    // item u = (group, slot): slots below `whole` take the group's items of
    // 2^lcap particles (every whole-th one), the next ones the item of each
    // smaller power of two that the size's binary digits ask for
    for (int64_t u = (int64_t)blockIdx.x * kWarps + w; u < ng * A.slots; u += (int64_t)gridDim.x * kWarps) {
        const int64_t k = u / A.slots;
        const int slot = (int)(u - k * A.slots);
        const int32_t g = A.groups[k];
        const uint32_t b = A.begin[g], e = A.end[g], ni = e - b;
        int q = 0;
        for (int lo = 0, hi = A.np - 1; lo < hi;) {  // its patch: the last one starting at or before b
            const int mid = (lo + hi + 1) >> 1;
            if (A.off[mid] <= (int64_t)b)
                lo = q = mid;
            else
                hi = mid - 1;
        }
        const int lcap = item_lcap(A.off[q + 1] - A.off[q]), whole = whole_items(A.n_g, lcap);
        if (slot < whole) {
            for (uint32_t c = slot; c < ni >> lcap; c += whole) {
                item64<POT, ORDER, EPS>(A, sm[w], k, b, e, b + (c << lcap), lcap, lane);
                __syncwarp();
            }
        } else if (slot - whole < lcap) {
            const int bit = slot - whole;
            if ((ni >> bit) & 1u)
                item64<POT, ORDER, EPS>(A, sm[w], k, b, e, b + ((ni >> (bit + 1)) << (bit + 1)), bit, lane);
            __syncwarp();
        }
    }
}

// W = 1/2 sum m_i phi_i in a fixed order (fixed grid, grid-stride loops,
// block tree, one final pass), so repeated calls give the same bits.
constexpr int kWBlocks = 512, kWThreads = 256;

__global__ void __launch_bounds__(kWThreads) k_wsum_partial(int64_t n, const double* m,
                                                            const double* phi, double* part) {
    launch_wait();
    __shared__ double sh[kWThreads];
    double acc = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kWThreads + threadIdx.x; i < n; i += (int64_t)kWBlocks * kWThreads)
        acc += 0.5 * m[i] * phi[i];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kWThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_wsum_final(const double* part, double* out) {
    launch_wait();
    if (threadIdx.x != 0) return;
    double s = 0.0;
    for (int b = 0; b < kWBlocks; ++b) s += part[b];
    *out = s;
}

// The split alone, for callers and tests of it (bh_split_f32).
__global__ void k_split_values(const double* __restrict__ v, int64_t n, float* __restrict__ hi,
                               float* __restrict__ lo) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float h, l;
    split_f32(v[i], h, l);
    hi[i] = h;
    lo[i] = l;
}

}  // namespace

ForceParams force_params(const Ctx* c) {
    const bh_params& p = c->prm;
    ForceParams fp;
    fp.G = p.G;
    fp.eps2 = p.eps * p.eps;
    fp.rc2 = p.r_coll * p.r_coll;
    fp.rc2_hi = fp.rc2 * (1.0 + 1e-10);
    fp.kappa = p.kappa;
    fp.eta = p.eta;
    fp.r_coll = p.r_coll;
    fp.GMc = p.G * p.M_central;
    fp.eps2f = (float)fp.eps2;
    fp.rc2f = (float)fp.rc2;
    fp.kappaf = (float)p.kappa;
    fp.etaf = (float)p.eta;
    fp.rcollf = (float)p.r_coll;
    fp.Gf = (float)p.G;
    fp.order = p.order;
    return fp;
}

namespace {

Args64 args64(const Ctx* c, const bh_particles* p, const ForceParams& fp) {
    Args64 A = {};
    A.ng = groups_bound(c);
    A.dng = dev_groups(c);
    A.groups = c->groups.p;
    A.begin = c->begin.p;
    A.end = c->end.p;
    A.jj_off = c->cnt_j.p;
    A.JJ = c->JJ.p;
    A.pc_off = c->cnt_c.p;
    A.C = c->C.p;
    A.x = p->x;
    A.y = p->y;
    A.z = p->z;
    A.vx = p->vx;
    A.vy = p->vy;
    A.vz = p->vz;
    A.m = p->m;
    A.M = c->M.p;
    A.cx = c->cx.p;
    A.cy = c->cy.p;
    A.cz = c->cz.p;
    A.Q = c->Q.p;
    A.fp = fp;
    A.n = (uint32_t)c->n;
    A.nn = nodes_bound(c);
    A.status = c->d_status;
    A.off = c->d_off.p;
    A.np = c->n_patches;
    A.n_g = c->prm.n_g;
    return A;
}

template <bool POT>
int launch_sum64(Ctx* c, Args64& A) {
    A.slots = 0;
    for (int q = 0; q < c->n_patches; ++q) {
        const int lc = item_lcap(c->h_off[q + 1] - c->h_off[q]);
        A.slots = std::max(A.slots, whole_items(c->prm.n_g, lc) + lc);
    }
    const int64_t ng = std::min(A.ng, groups_expected(c));  // (the kernel strides over more)
    const int64_t nb = (ng * A.slots + kWarps - 1) / kWarps;
    const unsigned grid = (unsigned)std::min<int64_t>(nb, (int64_t)1 << 30);
    const bool eps = A.fp.eps2 != 0.0;
    auto kern = A.fp.order >= 2 ? (eps ? k_sum64<POT, 2, true> : k_sum64<POT, 2, false>)
                                : (eps ? k_sum64<POT, 1, true> : k_sum64<POT, 1, false>);
    BH_CUDA(c, launch(c, kern, grid, 32 * kWarps, 0, A));
    BH_LAUNCH(c);
    return BH_OK;
}

}  // namespace

int stage_force(Ctx* c, bh_particles* p, bool add_central) {
    const ForceParams fp = force_params(c);
    add_central = add_central && c->prm.M_central != 0.0;
    if (c->prm.precision == BH_PREC_FP64) {
        Args64 A = args64(c, p, fp);
        A.abort = c->abort;
        A.add_central = add_central;
        A.ax = p->ax;
        A.ay = p->ay;
        A.az = p->az;
        BH_TRY(timing_begin(c));
        BH_TRY(stage_begin(c, BH_STAGE_FORCE));
        BH_TRY(launch_sum64<false>(c, A));
        BH_TRY(stage_end(c));
        return timing_end(c);
    }
    // the hi/lo split and the FP32 records were made by stage_moments
    return launch_force32(c, p, fp, add_central);
}

int stage_potential(Ctx* c, const bh_particles* p, double* phi, double* W) {
    BH_TRY(stage_moments64(c, p));  // FP64 moments of the current positions, either precision
    if (!phi) {
        BH_TRY(grow(c, c->pot, (size_t)c->n, "potential", false));
        phi = c->pot.p;
    }
    const ForceParams fp = force_params(c);
    Args64 A = args64(c, p, fp);
    A.phi = phi;
    BH_TRY(launch_sum64<true>(c, A));
    if (W) {
        BH_TRY(grow(c, c->diag, (size_t)kWBlocks + 1, "potential energy sums", false));
        BH_CUDA(c, launch(c, k_wsum_partial, kWBlocks, kWThreads, 0, c->n, p->m, phi, c->diag.p));
        BH_LAUNCH(c);
        BH_CUDA(c, launch(c, k_wsum_final, 1, 32, 0, c->diag.p, c->diag.p + kWBlocks));
        BH_LAUNCH(c);
        BH_CUDA(c, cudaMemcpyAsync(W, c->diag.p + kWBlocks, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        BH_CUDA(c, cudaStreamSynchronize(c->stream));
    }
    return BH_OK;
}

}  // namespace bh

extern "C" int bh_split_f32(const double* v, float* hi, float* lo, int64_t n, void* stream) {
    if (n < 0 || (n > 0 && (!v || !hi || !lo)) || (n > 0 && hi == lo)) return BH_E_INVAL;
    if (n == 0) return BH_OK;
    bh::k_split_values<<<bh::blocks_for(n, 256), 256, 0, (cudaStream_t)stream>>>(v, n, hi, lo);
    return cudaGetLastError() == cudaSuccess ? BH_OK : BH_E_CUDA;
}
