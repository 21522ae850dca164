// bh_internal.cuh -- context layout and helpers shared by the libbh.so
// translation units (not part of the public ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <string>
#include <vector>

#include "../../include/bh.h"

namespace bh {

constexpr int kLevels = 21;                    // key depth: 21 octal digits, 63 bits
constexpr uint32_t kQMax = (1u << kLevels) - 1;

// Device status word bits (set by kernels, read at synchronising calls).
constexpr int kStatNonFinite = 1;
constexpr int kStatListOverflow = 2;
constexpr int kStatTimeout = 4;
constexpr int kStatBounds = 8;  // an internal index check failed (access skipped)
constexpr int kStatRange = 16;  // a contact term outside the fixed-point accumulator's range
constexpr int kStatAxis = 32;   // cylindrical key frame with a particle on the axis (r = 0)

// Sizes of a device-sized list build (a list-constructing step captured as
// one graph: nothing is read back while it runs), in Ctx::d_sz.
constexpr int kSzLvl = 0;                   // kLevels + 3 words: first node of each level, then the node count
constexpr int kSzNg = kLevels + 3;          // group count
constexpr int kSzOvf = kSzNg + 1;           // overflow bits
constexpr int kSzNeedNodes = kSzOvf + 1;    // nodes wanted when the node capacity ran out (a lower bound)
constexpr int kSzNl = kSzNeedNodes + 1;     // leaf count
constexpr int kSzItems = kSzNl + 1;         // work items of the FP32 force kernel
constexpr int kSzWords = 32;
constexpr unsigned long long kOvfNodes = 1, kOvfLists = 2;

// Device buffer that only grows.
template <typename T>
struct DBuf {
    T* p = nullptr;
    size_t cap = 0;
};

// ---- sizes of the radix sort (sort.cu) --------------------------------------
constexpr int kSortThreads = 384;
constexpr int kSortItems = 12;  // keys per lane of a tile
// One small particle set is cut into tiles of 4 keys per lane instead, so that
// more SMs share it and a tile takes less time.  At the line its 391 tiles still
// run at once (3 blocks on each of 152 SMs).  Sorts of random keys with 4 and with
// 12 keys per lane: 65,537 keys 75 and 98 us, 400,000 115 and 130, 600,000 134 and
// 184, 800,000 157 and 193, 1,200,000 204 and 205.
constexpr int kSortSmallItems = 4;
constexpr int64_t kSortSmall = 600000;
constexpr int kRadix = 256;
constexpr int64_t kSortWide = (int64_t)1 << 27;  // keys from which the look-back words have 64 bits
constexpr int kSortPolls = 1 << 22;              // look-back polls before a tile gives up
struct SortLimits {
    int64_t wide_from;
    int polls;
};
constexpr bool small_tiles(int64_t n, int64_t wide_from) { return n < kSortSmall && n < wide_from; }
constexpr int64_t sort_tiles(int64_t n, int64_t wide_from) {  // of one set
    const int64_t tile = kSortThreads * (small_tiles(n, wide_from) ? kSortSmallItems : kSortItems);
    return (n + tile - 1) / tile;
}
// Scratch: look-back words, digit counts and tickets, cleared together at the
// start of a sort.
struct SortScratch {
    int64_t words, total;  // 32-bit words of the look-back part and in all
};
constexpr SortScratch sort_scratch(int64_t n, int64_t ntiles, int64_t nslots, int64_t wide_from) {
    const int64_t words = ntiles * kRadix * (n < wide_from ? 1 : 2);
    return {words, words + nslots * 8 * kRadix + 8};
}
constexpr int64_t sort_scratch_words(int64_t n) {
    return sort_scratch(n, sort_tiles(n, kSortWide), 1, kSortWide).total;
}

struct Ctx;
int fail(Ctx* c, int code, const char* fmt, ...);

// cudaMalloc-backed growth (the contents are not kept); returns BH_OK or
// BH_E_NOMEM (with message).  in_steps: a captured step may hold the buffer, so
// that step is captured again once it has moved.
int grow_raw(Ctx* c, void** p, size_t* cap, size_t bytes_needed, const char* what, bool in_steps);
template <typename T>
int grow(Ctx* c, DBuf<T>& b, size_t n, const char* what, bool in_steps = true) {
    size_t cap_bytes = b.cap * sizeof(T);
    int rc = grow_raw(c, (void**)&b.p, &cap_bytes, n * sizeof(T), what, in_steps);
    b.cap = cap_bytes / sizeof(T);
    return rc;
}

// Per-node packed record read by the walk (one 32-byte load per visit):
// a = (qlo.x | level << 21 | leaf flag, qlo.y | count << 21, qlo.z,
// successor of the subtree or -1), b = (qhi.xyz, first child, or for a leaf
// its first particle); the count is a leaf's particles or an inner node's
// children.  A leaf count of kWalkCntMax means "that many or
// more": the walk then reads the node's end.
struct WalkNode {
    uint4 a, b;
};
constexpr uint32_t kWalkLeaf = 1u << 26;
constexpr uint32_t kWalkCntMax = (1u << 11) - 1;

// Launch tuning of the FP32 force kernel (bh_set_tuning / the autotuner).
struct Tuning {
    int chunk = 96;          // largest i-chunk of a work item: 32, 64 or 96 particles
    int warps = 4;           // warps per block, 1..8
    int sched = BH_SCHED_DYNAMIC;
    int order_by_cost = 1;   // within a size class, largest estimated cost first
    int graph = 0;           // 1: every step of bh_step as a CUDA graph, 2: list-reusing ones only
    int order_window = 0;    // > 0: size-class order within windows of this many groups
    int graph_contact_room = 0;  // > 0: contact candidates a graph step may hold (0: automatic)
    int graph_room = 25;         // percent of room over the last build in a list-constructing graph step
};

struct Ctx {
    bh_params prm;
    Tuning tune;
    cudaStream_t stream = nullptr;
    int device = 0, num_sms = 0;
    std::string err;

    // state
    int64_t n = 0;
    bool have_tree = false, have_lists = false, have_acc = false;
    int64_t k_eval = 0;        // force evaluations done (drives the rebuild schedule)
    int64_t evals_since_build = 0, n_rebuilds = 0;
    int64_t n_launches = 0;    // kernels launched by this context

    // optional CUDA-event timing of the force kernel (one event pair per launch)
    // and of every stage (BH_STAGE_*)
    bool timing = false;
    std::vector<cudaEvent_t> ev_pool;
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev_force;
    struct StageEv {
        int stage;
        cudaEvent_t a, b;
    };
    std::vector<StageEv> ev_stage;       // recorded, not yet read
    std::vector<int> stage_open;         // indices into ev_stage of stages begun, not ended
    double stage_ms[BH_N_STAGES] = {};   // read stage times, summed since the last reset
    int64_t stage_calls[BH_N_STAGES] = {};

    // list capacity (bh_params.list_capacity; 0 = none) and the sizes a build
    // that exceeded it needed
    bool list_overflowed = false;
    int64_t need_pp = 0, need_pc = 0, need_jj = 0;

    // patches: independent particle sets, each with its own root box and
    // tree (a forest whose roots are nodes 0..n_patches-1); 1 for one set
    int n_patches = 1;
    std::vector<int64_t> h_off;         // particle offsets of the patches (n_patches + 1)
    DBuf<int64_t> d_off;                // the same on the device
    DBuf<uint32_t> tile_meta;           // sort tiles per patch (4 words per tile), n_patches > 1
    int64_t n_tiles = 0;
    int n_sort_slots = 0;               // patches of more than one sort tile
    DBuf<uint2> box_map;                // root-box blocks of the patches: (patch, block within it)
    DBuf<int> box_poff;                 // first root-box block of each patch (n_patches + 1)
    int n_box_blocks = 0;
    DBuf<long long> d_rcq;              // per patch walk contact threshold
    DBuf<long long> d_rfar;             // per patch far threshold of the split expansion
    DBuf<long long> d_period;           // per patch phi period in grid cells (cylindrical frame; 0 = none)

    // status and small device scalars
    int* d_status = nullptr;
    double* d_box = nullptr;   // per patch: lo[3], L, S, spare x3 (8 doubles)
    unsigned long long* d_small = nullptr;  // scan totals etc. (64 words)
    unsigned long long* h_pin = nullptr;    // page-locked words for size read-backs (64)
    cudaEvent_t read_event = nullptr;       // what the host waits for: a copied count, the last read of an array

    // keys and sort
    DBuf<uint64_t> key[2];
    DBuf<uint32_t> idx[2];
    int key_cur = 0;           // buffer holding the sorted keys / perm
    DBuf<uint32_t> sort_scratch;  // look-back words, digit counts, tickets
    SortLimits sort_limits{kSortWide, kSortPolls};
    DBuf<double> pscratch;     // permutation scratch (8 arrays x 8 bytes per particle)
    DBuf<double> cyl;          // cylindrical frame: phi[n], r[n]
    DBuf<unsigned long long> box_part;  // root-box partials (6 per block, as ordered integers)
    DBuf<uint8_t> scan_tmp;

    // tree
    int64_t n_nodes = 0;
    std::vector<int64_t> lvl_start;  // node id range of each level (size depth+2)
    DBuf<uint8_t> level, nchild;
    DBuf<uint32_t> begin, end;
    DBuf<int32_t> parent, first_child;
    DBuf<uint32_t> qlo, qhi;         // 3 per node
    DBuf<WalkNode> wnode;
    DBuf<uint16_t> tree_range;       // per particle: levels of the nodes that begin there
    DBuf<int32_t> tree_top;          // per particle at which nodes begin: the highest of them
    DBuf<uint32_t> tree_cnt;         // per (level, particle tile): nodes that begin there, then first ids

    // moments
    DBuf<double> M, cx, cy, cz, Q;   // Q: 6 per node
    DBuf<float4> cell32;             // 3 per node: (c_hi, M), (c_lo, Qxx), (Qxy, Qxz, Qyy, Qyz)
    DBuf<float> cell32lo;            // per node: exact mass - M of the record (FP32)
    DBuf<float4> phi, plo;           // per particle FP32 split: (x_hi, m), (x_lo, 0)
    DBuf<uint2> refine;                 // (particle, list slot) queued for the refinement pass
    DBuf<float> cbnd;                   // particles with contact candidates: FP32 bound,
    DBuf<uint32_t> cslot;               // list slot,
    DBuf<unsigned> cflag;               // and a flag the post-contact check claims
    DBuf<unsigned long long> contacts;  // (i, j) contact candidates for the FP64 pass
    DBuf<double> diag;                   // diagnostic partial sums
    DBuf<double> pot;                    // per-particle potential when the caller passes none
    DBuf<unsigned long long> contact_acc;  // per particle fixed-point contact sums (3 per particle)
    int64_t n_contacts = 0;
    int64_t n_refined = 0;              // particles the refinement pass re-evaluated (last read)
    bool refine_pending = false;        // an evaluation ran since n_refined was read
    bool contact_stats = false;         // the device contact counters hold an FP32 evaluation's counts

    // groups
    int64_t n_groups = 0;
    DBuf<int32_t> groups;            // node ids ordered by begin
    int64_t n_leaves = 0;
    DBuf<int32_t> leaves;            // node ids ordered by begin
    DBuf<int2> order;                // FP32 force kernel's work items (group, i-chunk) in processing order
    DBuf<unsigned long long> order_cnt;  // order buckets: counts/starts and cursors
    DBuf<uint32_t> ord_cnt;              // windowed order: bucket counts, then cursors, per window
    int sort_attr_device = -1;           // device the sort kernel's smem limit was raised on
    int f32_attr_device = -1;            // device the FP32 kernels' smem limit was raised on
    unsigned f32_blocks = 0;             // grid of the last FP32 force launch
    DBuf<unsigned long long> warp_time;  // per warp (start, end) of the last persistent launch
    int64_t warp_time_n = 0;
    bool capturing = false;              // issuing work into a stream capture
    cudaGraphExec_t graph_exec = nullptr;  // the captured list-reusing step
    cudaStream_t cap_stream = nullptr;   // private stream the step is captured on
    // host-buffer stepping: positions, masses and ids are final once the last
    // evaluation's tree/moments stage is enqueued; their copy back is
    // enqueued right there, on a second stream, so that it overlaps the force
    // kernel (the host waits after that kernel to size the contact pass)
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t pos_event = nullptr;
    bool want_pos_event = false, pos_event_recorded = false;
    bool early_now = false;              // the evaluation being run is the call's last
    const bh_particles* early_dst = nullptr;  // host arrays of the early copy
    const bh_particles* early_src = nullptr;  // device arrays it copies from
    bool early_ids = true;               // the early copy includes masses and ids
    int64_t h2d_bytes = 0, d2h_bytes = 0;  // copied by bh_step_host so far
    // sizes of the step being issued are read on the device, within bounds that
    // outlive the current lists (captured steps of either kind)
    bool dev_sizes = false;
    int64_t buf_gen = 0;                 // buffers that a captured step may hold (re)allocated so far
    bool graph_ok = false;               // graph_exec matches the current arrays and settings,
    int64_t graph_gen = 0;               // the buffers,
    int64_t graph_size[2] = {};          // and about the sizes: groups and nodes it was captured with
    bh_particles graph_p{};              // particle arrays the graph was captured with
    int64_t graph_launches = 0;          // kernels in the graph

    // device-sized list builds: a list-constructing step of bh_step issued as
    // one graph (graph tuning on), its buffers sized from the previous build
    unsigned long long* d_sz = nullptr;  // kSzWords device words (level bounds, group count, overflow)
    bool dev_build = false;              // issuing a device-sized build (no size read-backs)
    const unsigned long long* abort = nullptr;  // while issuing the forces and kick of such a step: its
                                                // overflow bits (nonzero: those kernels do nothing)
    int64_t cap_nodes = 0;               // node capacity of the build being issued
    int64_t dev_slots = 0;               // groups with a list slot in it
    cudaGraphExec_t rgraph_exec = nullptr;  // the captured list-constructing step
    bool rgraph_ok = false;              // rgraph_exec matches the arrays and capacities
    int64_t rgraph_gen = 0;
    bh_particles rgraph_p{};
    int64_t rgraph_launches = 0;
    int64_t rgraph_cap[5] = {};          // nodes, slots, P, C, JJ it was captured with
    int64_t rgraph_walk_cap[2] = {};     // and list slot sizes
    cudaStream_t body_stream[2] = {nullptr, nullptr};  // its conditional bodies are captured on these
    // force-kernel timing inside step graphs: event-record nodes around the
    // kernel, given fresh events before each launch while timing is on
    struct GraphTiming {
        cudaGraph_t g = nullptr;             // the graph the executable was instantiated from
        cudaGraphNode_t node[2] = {nullptr, nullptr};
        bool have = false;
    };
    GraphTiming gt_reuse, gt_rebuild, gt_tmp;
    GraphTiming* gt_cur = nullptr;           // the graph being captured
    cudaEvent_t gt_idle[2] = {nullptr, nullptr};  // recorded by those nodes while timing is off
    int64_t n_graph_builds = 0;          // list builds that ran inside a graph
    int64_t n_graph_build_redos = 0;     // of those, builds redone eagerly after a capacity ran out
    int64_t n_graph_captures = 0;        // step graphs captured

    // lists
    int64_t n_pp = 0, n_pc = 0, n_jj = 0;
    int64_t n_int_pp = 0, n_int_pc = 0;
    int64_t n_int_pp_far = 0;            // FP32 path: pp interactions with far list particles
    bool far_pending = false;            // a list build ran since n_int_pp_far was read (word 10 of d_small)
    cudaEvent_t build_event = nullptr;   // end of the last eager tree or list build
    DBuf<int64_t> cnt_p, cnt_c, cnt_j;   // per group counts, then offsets (ng + 1)
    DBuf<int64_t> cnt_jm;                // FP32 path: per group index of the first far list particle
    DBuf<int32_t> stash_p, stash_c;      // per group list slots of the one-walk build
    int64_t walk_cap_p = 0, walk_cap_c = 0;  // their sizes (0: count and fill walks)
    int64_t n_one_walk_builds = 0;       // list builds whose lists came from one walk
    DBuf<int32_t> P, C;
    DBuf<uint32_t> JJ;

    // host-buffer stepping
    DBuf<double> hbuf;                   // 10 arrays of n doubles
    DBuf<int64_t> hid;
};

// ---- CUDA error plumbing -------------------------------------------------
#define BH_CUDA(c, call)                                                              \
    do {                                                                              \
        cudaError_t e_ = (call);                                                      \
        if (e_ != cudaSuccess)                                                        \
            return ::bh::fail((c), BH_E_CUDA, "%s failed: %s (%s:%d)", #call,          \
                              cudaGetErrorString(e_), __FILE__, __LINE__);            \
    } while (0)
#define BH_TRY(expr)                 \
    do {                             \
        int r_ = (expr);             \
        if (r_ != BH_OK) return r_;  \
    } while (0)
#define BH_LAUNCH(c)                                                                  \
    do {                                                                              \
        cudaError_t e_ = cudaGetLastError();                                          \
        if (e_ != cudaSuccess)                                                        \
            return ::bh::fail((c), BH_E_CUDA, "kernel launch failed: %s (%s:%d)",      \
                              cudaGetErrorString(e_), __FILE__, __LINE__);            \
        (c)->n_launches++;                                                            \
    } while (0)

// Kernel launches with programmatic dependent launch: a kernel may be set up
// while the one before it in the stream still runs, and waits, before it reads
// or writes anything, until that one has completed (and, in turn, all before
// it).  Every kernel launched this way begins with launch_wait(), and takes no
// __restrict__ pointer: that would promise that nothing else writes the memory
// while the kernel lives, which now begins before its inputs are written, and
// with the promise a load may be moved above the wait.  An eager
// evaluation is some 50 short dependent launches: of a 65,537-particle ring 495
// -> 423 us, of the 4096 cube 452 -> 390 us.  Not in captured steps (early =
// false), whose graph launches got slower with it: 4 steps of a
// 300,007-particle ring 1450 -> 1480 us.
__device__ __forceinline__ void launch_wait() {
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}

inline cudaLaunchAttribute early_attribute(bool early) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = early ? 1 : 0;
    return at;
}

template <class... KA, class... A>
cudaError_t launch_on(cudaStream_t s, bool early, void (*kern)(KA...), dim3 grid, dim3 block, size_t smem, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = early_attribute(early);
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <class... KA, class... A>
cudaError_t launch(Ctx* c, void (*kern)(KA...), dim3 grid, dim3 block, size_t smem, A... args) {
    return launch_on(c->stream, !c->capturing, kern, grid, block, smem, args...);
}

inline unsigned blocks_for(int64_t n, int threads) {
    int64_t b = (n + threads - 1) / threads;
    return (unsigned)(b < 1 ? 1 : b);
}

// ---- stage entry points (one translation unit each) ------------------------
// scan.cu: exclusive prefix sums in place, n >= 1; the total goes to *d_total
// (device).  scan3_i64: three arrays of n (+ 1) elements, totals to
// d_total[0..2] and to each array's element n; with dn, the element count is
// read on the device (*dn, at most n).
int scan_u32(Ctx* c, uint32_t* v, int64_t n, unsigned long long* d_total);
int scan3_i64(Ctx* c, int64_t* const (&v)[3], int64_t n, unsigned long long* d_total, const unsigned long long* dn);

// sort.cu
int stage_keys(Ctx* c, const bh_particles* p);     // root box + keys (+ status on NaN)
int stage_sort(Ctx* c);                            // stable LSD radix sort of (key, idx)
int reserve_sort(Ctx* c);                          // its scratch (before a captured step)
int stage_permute(Ctx* c, bh_particles* p);        // gather particle arrays into key order
int setup_patches(Ctx* c, int n_patches, const int64_t* off);  // bh_api.cu
int64_t sort_tiles_for(const std::vector<int64_t>& off, std::vector<uint32_t>* meta, int* nslots);  // sort.cu
// context-free sort over caller buffers (sort.cu); scratch >= sort_scratch_words(n) words
cudaError_t sort_setup_device();
cudaError_t sort_pairs_with(cudaStream_t s, uint64_t* keys, uint32_t* idx, uint64_t* ktmp, uint32_t* itmp,
                            int64_t n, int num_sms, uint32_t* scratch, int polls, int* status);

// tree.cu
int stage_octree(Ctx* c);                          // nodes and groups; sets n_nodes, n_groups
int64_t tree_count_words(int64_t n);               // words of tree_cnt for n particles
int stage_boxes(Ctx* c);                           // integer boxes + walk records
int stage_moments(Ctx* c, const bh_particles* p);  // M, c, Q (+ FP32 cell records)
int stage_moments64(Ctx* c, const bh_particles* p);  // FP64 M, c, Q whatever the precision

// walk.cu
int stage_lists(Ctx* c);                           // walk (count, fill) + particle expansion
int stage_lists_dev_walk(Ctx* c);                  // device-sized: walk, offsets, room check
int stage_lists_dev_fill(Ctx* c);                  // device-sized: lists, expansion, group order

// force.cu
int build_order32(Ctx* c);                         // FP32 kernel's work items (per list build)
bool same_items32(const Ctx* c, const bh_tuning& a, const bh_tuning& b);  // the same items with either's chunk and window
int reserve_force32(Ctx* c);                       // its buffers
int stage_force(Ctx* c, bh_particles* p, bool add_central);
int stage_potential(Ctx* c, const bh_particles* p, double* phi, double* W);  // self-gravity potential (FP64)

// bh_api.cu: wait for the stream and report the device status word
int read_status(Ctx* c);

// Bounds of the step being issued: the sizes themselves, or, with sizes read on
// the device, the buffers' capacities (bounds of indices) and the sizes with
// graph_room to grow (for grids; every size is covered).
inline int64_t with_room(const Ctx* c, int64_t v) { return v + v * c->tune.graph_room / 100 + 64; }
inline const unsigned long long* dev_groups(const Ctx* c) { return c->dev_sizes ? c->d_sz + kSzNg : nullptr; }
inline int64_t groups_bound(const Ctx* c) {
    if (!c->dev_sizes || c->dev_build) return c->n_groups;
    size_t b = c->groups.cap;
    for (size_t v : {c->cnt_p.cap, c->cnt_c.cap, c->cnt_j.cap}) b = v < b ? v : b;
    if (c->prm.precision == BH_PREC_FP32 && c->cnt_jm.cap < b) b = c->cnt_jm.cap;
    return (int64_t)b - 1;
}
inline int64_t groups_expected(const Ctx* c) {
    return c->dev_build ? (c->dev_slots > 1 ? c->dev_slots : 1) : c->dev_sizes ? with_room(c, c->n_groups) : c->n_groups;
}
inline int64_t nodes_bound(const Ctx* c) {
    if (!c->dev_sizes || c->dev_build) return c->n_nodes;
    return (int64_t)(c->prm.precision == BH_PREC_FP32 ? c->cell32lo.cap : c->M.cap);
}

// bh_api.cu: force-kernel and stage timing (no-ops unless enabled, or while
// capturing a graph); stage_end closes the innermost stage begun
int timing_begin(Ctx* c);
int timing_end(Ctx* c);
int stage_begin(Ctx* c, int stage);
int stage_end(Ctx* c);

// update.cu
int stage_kick(Ctx* c, bh_particles* p, double h);
int stage_kick_drift(Ctx* c, bh_particles* p, double h, double dt, bool twice = false);
int stage_diagnostics(Ctx* c, const bh_particles* p, double* host_out);  // 11 sums to the host

}  // namespace bh
