// bc_internal.cuh -- device-side types, exact integer helpers and the launch
// functions shared by the translation units of libbcgpu.so.
//
// State layout (row-major n rows of ld entries, structure of arrays; Section 5 stores the
// triple (d, sigma, flag) per pair in one row-major array -- here each field is its own
// array so a pass reads only the fields it needs):
//   D   [n*ld]  distance type DT (int32 or int64), INF = DT max
//   S   [n*ld]  uint64 path counts sigma_st
//   Dl  [n*ld]  dependencies delta_s.(t) as float-float pairs (ff.cuh), 0 on the diagonal
// ld is n rounded up to a multiple of kRowAlign entries, so every row starts on a 32-byte
// boundary and the vector loads of the passes serve every n; the entries past n hold
// INF / 0 / 0 (no path) and no pass changes them.  With rows packed at n entries an odd n
// had to take one column per thread: 16 edge and vertex updates of BA n = 5003 took
// 10.4 ms that way and take 5.7 ms so (the column test was 297 us and the rank-1 pass
// 113 us of an update's 490 us).
//   BC  [n]    fp64 pair (hi, lo): compensated running sums of the G_D scores
// E* superset ("E*+") -- every arc that lies on some shortest path, plus arcs that
// may no longer do so (Section 6: any superset of E* gives the right DAGs) -- is a
// CSR with per-vertex slack: arcs of vertex a sit in slots [off[a], off[a]+len[a]),
// followed by empty slots.  A segment that fills up moves to the free region past the
// laid-out ones (off[a] changes, its old slots are emptied).  A slot holds tail, head and
// weight in 8 bytes (Arc), so one load brings what a pass over the slots needs.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "ff.cuh"

namespace bcg {

enum : int32_t { ERRF_OVERFLOW = 1, ERRF_DIST = 2, ERRF_TIMEOUT = 4, ERRF_ARG_DEVICE = 8 };

// Per-handle device counters: [0] rows re-accumulated [1] no-op updates [2] most rows of
// one update [3] updates [4] pairs lowered [5] pairs with new tied paths [6] rows scanned
// [7] rows re-accumulated in full [8] rows corrected pair by pair [9] (row, target) pairs
// of those corrections [10] pairs corrected by DAG walks [11] vertices those walks found
// [12] E* arcs they examined.
constexpr int kStats = 13;

// Saturation marker for a distance sum that does not fit: INT64_MAX.  For DT =
// int64 this equals INF, so callers test for it before comparing.
constexpr int64_t SAT = INT64_MAX;

template <typename DT> struct Inf;
template <> struct Inf<int32_t> { static constexpr int64_t v = INT32_MAX; };
template <> struct Inf<int64_t> { static constexpr int64_t v = INT64_MAX; };

// a + b for finite non-negative a, b; SAT when the sum is not a finite DT value.
template <typename DT>
__device__ __forceinline__ int64_t dsum(int64_t a, int64_t b) {
    if constexpr (sizeof(DT) == 4) {
        int64_t s = a + b;
        return s >= Inf<int32_t>::v ? SAT : s;
    } else {
        return (b > INT64_MAX - 1 - a) ? SAT : a + b;
    }
}

__device__ __forceinline__ void set_err(int32_t* err, int32_t f) { atomicOr(err, f); }

// Block-uniform read of the sticky error word: other CTAs of the same launch may set it
// at any time, so kernels that use barriers take one decision for the whole CTA.
// Every thread of the block must call it.
__device__ __forceinline__ bool block_err(const int32_t* err) {
    __shared__ int32_t s_err;
    __syncthreads();
    if (threadIdx.x == 0) s_err = *reinterpret_cast<const volatile int32_t*>(err);
    __syncthreads();
    return s_err != 0;
}

// 64 x 64 -> 64 product of path counts; flags overflow when the high word is used.
__device__ __forceinline__ uint64_t mul_chk(uint64_t a, uint64_t b, int32_t* err) {
    if (__umul64hi(a, b) != 0ull) set_err(err, ERRF_OVERFLOW);
    return a * b;
}

__device__ __forceinline__ uint64_t add_chk(uint64_t a, uint64_t b, int32_t* err) {
    uint64_t s = a + b;
    if (s < a) set_err(err, ERRF_OVERFLOW);
    return s;
}

// Entries of a row of the state (and of the column vectors the passes read beside it).
constexpr int kRowAlign = 8;
__host__ __device__ inline int32_t row_pitch(int32_t n) { return (n + kRowAlign - 1) & ~(kRowAlign - 1); }

// One slot of the superset: the arc's tail and head (15 bits each; the head in bits 2..16,
// so that masking gives four times it) and its weight, held as 2^31 - 1 where it does not
// fit 31 bits (an int64 graph keeps the weights in full beside the slots, e_w64) and as
// -2^31 in an empty slot.
struct __align__(8) Arc {
    uint32_t ids;
    int32_t w;
    __host__ __device__ int dst() const { return (int)((ids >> 2) & 0x7FFFu); }
    __host__ __device__ int src() const { return (int)(ids >> 17); }
    __host__ __device__ bool empty() const { return w < 0; }
};
constexpr int kMaxVertices = 32768;
inline __host__ __device__ Arc make_arc(int32_t a, int32_t b, int64_t w) {
    return Arc{((uint32_t)a << 17) | ((uint32_t)b << 2), w < INT32_MAX ? (int32_t)w : INT32_MAX};
}
inline __host__ __device__ Arc empty_arc() { return Arc{0u, INT32_MIN}; }
// Slots a warp of the accumulation takes at a time; the slot array is a whole number of
// groups.
constexpr int kGroupSlots = 256;

constexpr int kPairCap = 128;   // changed targets of a row corrected pair by pair (k_pair.cu)

// The edges of one update as the DAG walks of the pair corrections need them: the
// updated vertex v, the other endpoints x_j and the weight of {v, x_j} before the
// update (-1: the edge is new).  Updates with more edges use the column test.
constexpr int kWalkMaxEdges = 32;
struct WalkUpd {
    int32_t v;
    int32_t k;
    int32_t x[kWalkMaxEdges];
    int64_t wold[kWalkMaxEdges];
};
constexpr int kPairPlanBytes = 40;   // of the column test's plan per target (the walks' dense tables lie there too)

// One edge of a vertex update, as staged on the device (matches bc_vedge).
struct VEdge {
    int32_t x;
    int32_t dir;
    int64_t w;
};

// One write into the E*+ CSR (slot < 0: only the length of vertex a changes).
struct EOp {
    int32_t slot;
    int32_t a;
    int32_t b;
    int32_t len_a;
    int64_t w;
};
constexpr int kMaxEOps = 64;
struct EOps {
    int32_t count;
    int32_t pad;
    EOp op[kMaxEOps];
};
// Move of the E* segment of vertex a (len arcs) from slot from to slot to, in the free
// region past the laid-out segments.
struct EMove {
    int32_t a;
    int32_t from;
    int32_t to;
    int32_t len;
};
constexpr int kMaxEMoves = 32;
struct EMoves {
    int32_t count;
    int32_t pad;
    EMove mv[kMaxEMoves];
};

// Where the arrays of an accumulation CTA live (dev_accum_source): byte offsets into its
// shared memory or, for the ones marked, into its part of the work space (acc_layout).
struct AccLayout {
    int32_t row, cnt, level, far, sink, big, mask, base, pool, cell;
    uint8_t mask_ws, pool_ws, cell_ws;
    int32_t pcap;        // heads the pool holds
    int32_t smem;        // bytes of shared memory
    int32_t ws;          // bytes of work space
    uint8_t all_smem;    // no array but far is in the work space
};
inline __host__ __device__ int64_t group_slots(int64_t slots) {
    return (slots + kGroupSlots - 1) / kGroupSlots * kGroupSlots;
}
AccLayout acc_layout(int n, int64_t e_cap, bool is_static);
// Most shared memory of an accumulation CTA (of the 227 KB a CTA may have), and what its
// kernels are allowed: the allowance belongs to the kernel, which every handle and every
// batch launches with a layout of its own, so none of them sets less.
constexpr int32_t kAccSmemMax = 224 * 1024;
inline bool acc_all_smem(const AccLayout& l) { return l.all_smem != 0; }

// Device state of one handle (plain pointers; owned by the host-side bc_graph).
struct Dev {
    int32_t n;
    int32_t ld;          // entries of a state row (row_pitch(n))
    int32_t dbytes;      // 4 or 8
    int32_t directed;
    int32_t nsm;
    void* D;
    uint64_t* S;
    ff* Dl;
    double* bc_hi;
    double* bc_lo;
    // full graph (G or G_D), used by the static computation
    Arc* g_arc;          // [g_arcs] by tail
    int64_t* g_w64;      // [g_arcs] weights in full (int64 distances; else NULL)
    int32_t* g_off;      // [n + 1] first arc of each tail
    int64_t g_arcs;
    unsigned long long* g_count;   // [3] number of arcs in g_arc, and of two lists of the search
    // E*+ CSR with slack
    int32_t* e_off;
    int32_t* e_len;
    Arc* e_arc;          // [e_cap]
    int64_t* e_w64;      // [e_cap] weights in full (int64 distances; else NULL)
    int64_t e_cap;       // a multiple of kGroupSlots
    int64_t e_used;      // slots laid out or moved to so far; the rest is the free region
    // error word, counters
    int32_t* err;
    int64_t* stats;      // [0] rows re-accumulated [1] no-op updates [2] max rows [3] updates
                         // [4] pairs lowered [5] pairs with new ties [6] rows scanned
    // scratch
    uint32_t* changed;   // [n] 1: the row changed in the current update
    int32_t* rows;       // [n] rows of the IN phase, or of a fused edge pass's first direction
    int32_t* rows2;      // [n] rows of the OUT phase, or of the second direction
    int32_t* acc_rows;   // [n] rows that changed (each list in the order of its atomics: no result
                         // depends on it)
    int32_t* counts;     // [0] rows [1] acc_rows [2] rows2 [3] full rows [4] pair pieces handed out
                         // [5] rows corrected pair by pair [6] CTAs of k_update_end done [8..10] rows
                         // in the walks' lists (light rows and the two below) [11..13] rows taken
                         // from them; all zero between updates
    void* fD;            // [n] per-row distance to v after the phase (DT)
    uint64_t* fS;        // [n] per-row path count to v after the phase
    uint64_t* fM;        // [n] per-row multiplier of a tie
    void* cD;            // [ld] per-column distances from v (DT); INF past n
    uint64_t* cS;        // [ld] per-column path counts from v
    uint64_t* cM;        // [ld] per-column multiplier of a tie
    void* cD2;           // [ld] second column vector (fused undirected edge pass): distances (DT)
    uint64_t* cS2;       // [ld] its path counts
    ff* partial;         // [nrb * ld] column partial sums
    int32_t nrb_max;     // row blocks of the BC reduction
    AccLayout acc_lay[2];   // of the accumulation kernel: updates, static computation
    int32_t acc_threads[2]; // its threads per CTA
    int32_t acc_grid[2];    // its CTAs
    int32_t acc_grid_wide[2];  // its CTAs of kAccThreadsWide threads
    int32_t acc_wide;       // 1: wide CTAs for partial waves of sources
    int32_t acc_narrow_only;  // 1: never the wide CTAs (kept across launch-shape updates)
    int32_t* ws;         // accumulation work space, acc_ctas * ws_stride ints
    int32_t acc_ctas;    // most CTAs of any accumulation launch
    int64_t ws_stride;
    // pair-dependency corrections (undirected graphs): the pairs changed by this update,
    // their values before it, and the changed targets of each row
    int32_t pair_on;
    int32_t tcap;        // targets recorded per row (kPairCap); more -> full re-accumulation
    uint32_t* chg;       // [n * chg_words] bit (s,t): pair changed in this update
    int32_t chg_words;   // (n + 31) / 32
    void* oldD;          // [n*ld] d(s,t) before the update, valid where the bit is set (DT)
    uint64_t* oldS;      // [n*ld] sigma_st before the update, likewise
    int32_t* tcnt;       // [n] changed targets of the row
    int32_t* tlist;      // [n * tcap]
    void* plan;          // [n * tcap] per-target scalars of the pair corrections (k_pair.cu)
    int64_t* pair_w;     // [n + 1] prefix of the pair corrections' work item weights
    int32_t* full_rows;  // [n] rows re-accumulated in full (counts[3])
    int32_t* pair_rows;  // [n] rows corrected pair by pair, most targets first (counts[5])
    int32_t pair_walk;   // 1: pair corrections by DAG walks (k_walk.cu), scratch below
    int64_t walk_cap;    // most entries of a walk's table in shared memory
    int32_t* walk_rows;  // [2n] rows with more targets, rows that outgrew their table
    int64_t* bcfix;      // [3n + 1] BC change of the changed rows in this update, per column
                         // fixed-point words (units of 2^-24, 2^-71 and, behind those of all
                         // columns, 2^-112), then whether any of the last is used; zero between
                         // updates
    cudaStream_t st;
    // a third stream for the rows walked by a CTA each (undirected graphs): forked from st
    // before the light rows, joined back after them
    cudaStream_t st3;
    cudaEvent_t ev3_join;
};

constexpr int kRowsPerBlock = 64;   // rows per partial sum of the BC reduction
// Threads of an accumulation CTA (one source at a time) for the few rows over the target
// cap of an update on graphs of at least kAccWideMinN vertices (one source's levels
// spread over more threads); otherwise 256, 512 or 1024 by its shared memory
// (accum_config).  The batched path picks 128, 256 or 512 by autotuning.
constexpr int kAccThreadsWide = 1024;
constexpr int kAccWideMinN = 4096;

// Accumulation launch shape for n and the current E* capacity (sets the acc_ fields and
// ws_stride of d); the work space must then hold acc_ctas * ws_stride ints.
void accum_config(Dev& d);

// Recording of changed pairs by the passes that write D and sigma (pair corrections).
struct PairRec {
    uint32_t* chg;
    int32_t chg_words;
    void* oldD;
    uint64_t* oldS;
    int32_t* tcnt;       // NULL: nothing is recorded
    int32_t* tlist;
    int32_t tcap;
    int32_t first;       // no pair has changed yet in this update (the IN phase; row v)
    int32_t ld;          // entries of a state row
};

// The recording buffers of a handle with pair corrections.
__host__ __device__ inline PairRec make_pair_rec(const Dev& d) {
    PairRec r;
    r.chg = d.chg;
    r.chg_words = d.chg_words;
    r.oldD = d.oldD;
    r.oldS = d.oldS;
    r.tcnt = d.tcnt;
    r.tlist = d.tlist;
    r.tcap = d.tcap;
    r.first = 0;
    r.ld = d.ld;
    return r;
}

// Columns per thread of the pair-correction column test: two 16-byte loads of a row of
// int32 distances, one of int64 ones.
__host__ __device__ constexpr int pair_vn(int dbytes) { return dbytes == 4 ? 8 : 2; }

// The first change of pair (s,t) in an update sets its bit, saves its old distance and
// path count, and lists t as a changed target of row s (targets beyond the capacity
// are only counted).  Later changes of the same pair (the OUT phase after the IN
// phase) keep the saved values.  Each pair is written by one thread per pass, and a
// bit set by an earlier pass is visible, so a plain read of the word decides; the bit
// is then set without waiting for the old word.
template <typename DT>
__device__ __forceinline__ void record_change(const PairRec& r, int s, int t, int64_t d_old,
                                              uint64_t sig_old) {
    const uint32_t bit = 1u << (t & 31);
    uint32_t* w = r.chg + (size_t)s * r.chg_words + (t >> 5);
    if (!r.first && (*w & bit)) return;
    atomicOr(w, bit);
    const size_t i = (size_t)s * r.ld + t;
    static_cast<DT*>(r.oldD)[i] = (DT)d_old;
    r.oldS[i] = sig_old;
    const int pos = atomicAdd(r.tcnt + s, 1);
    if (pos < r.tcap) r.tlist[(size_t)s * r.tcap + pos] = t;
}

// ---- programmatic dependent launch ----
// The kernels of an update run one after another on the handle's stream.  They are
// launched with programmatic stream serialization allowed, so the launch of the next
// kernel is processed while this one runs, and each one starts with pdl_enter(): a wait
// for the previous kernel's completion and memory before touching any data.  No kernel
// triggers its dependents early: the next kernel's CTAs are placed only as this grid's
// CTAs exit (an early trigger let every later kernel's CTAs occupy SMs while waiting,
// which slowed the running kernel).  Launched the ordinary way, or after a non-kernel
// operation, the wait has no effect.
__device__ __forceinline__ void pdl_enter() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                            Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// ---- launches (k_update.cu) ----
cudaError_t scan_setup();
void launch_estar_write(const Dev& d, const EOps& ops);
void launch_estar_move(const Dev& d, const EMoves& moves);
void launch_alg4_in(const Dev& d, int32_t v, const VEdge* e, int32_t k, int full, const EOps& ops);
void launch_out_prep(const Dev& d, int32_t v, const VEdge* e, int32_t k, int full);
void launch_scan_in(const Dev& d, int32_t v);
void launch_scan_out(const Dev& d, int32_t v);
void launch_write_row(const Dev& d, int32_t v);
void launch_edge_prep(const Dev& d, int32_t u, int32_t v, int64_t w, const EOps& ops);
void launch_edge_scan(const Dev& d);
void launch_estar_keep(const Dev& d, uint8_t* keep);
PairRec pair_rec(const Dev& d);
void launch_pair_plan(const Dev& d);
void launch_pairdep(const Dev& d);
cudaError_t pair_setup();   // kernel attributes (the weights pass's dynamic shared memory)
// The pair corrections by walks: rows to their classes (k_pair_plan's place), then the walks.
void launch_walk_class(const Dev& d);
void launch_walks(const Dev& d, const WalkUpd& upd, cudaEvent_t ready);   // ready: when the classes are (NULL: one stream)
cudaError_t walk_setup();   // kernel attributes
void launch_update_end(const Dev& d);

// ---- launches (k_accum.cu) ----
void launch_accum(const Dev& d, int is_static);
void launch_accum_rows(const Dev& d, const int32_t* rows, const int32_t* count);
void launch_bc_static(const Dev& d);

// ---- launches (k_static.cu) ----
void launch_sssp(const Dev& d, int64_t w_max, bool all_arcs);
void launch_estar_flags(const Dev& d, uint8_t* flags);

}  // namespace bcg
