// k_walk.cu -- pair corrections of a row at a time, by walks of the shortest-path DAG.
//
// The rows of an update with at most kPairCap changed targets are corrected by
//     delta'_s(x) = delta_s(x) + sum over changed pairs (s,t) of [delta'_st(x) - delta_st(x)]
// (k_pair.cu).  For one state and the set T of the row's changed targets,
//     delta_T(x) = sum over t in T of sigma_sx * sigma_xt / sigma_st
// is the dependency of s on x restricted to the targets in T, and it obeys Eq. 4 with
// the 1 replaced by "y is in T":
//     delta_T(x) = sum over arcs (x,y) of DAG(s) of sigma_sx / sigma_sy * ([y in T] + delta_T(y)).
// It is zero outside the ancestors of T, so a walk backwards from T over the arcs with
// d(s,x) + w(x,y) = d(s,y) (Eq. 1) finds every vertex with a correction, and the
// recurrence over the arcs found gives all the sums, without a term per target and
// without reading row t.  In G_D of an undirected graph the arcs into y are y's own arcs
// reversed (same weight), read from the E* superset; before the update E*+ held every
// arc of the old E* (arcs are only added between re-layouts, and a re-layout keeps the
// arcs of the state it reads), and the arcs of the update itself carry their old weight
// from `upd` (or did not exist).  The old row is the new one except at T, where the
// saved values hold.
//
// A pair (s,y) with y not in T keeps its whole set of shortest paths, so every ancestor of
// y is outside T and has the same DAG arcs in both states: past T the two recurrences
// differ only in the values that they carry, and, being linear, run as one on the
// difference.  So a target has two entries in the row's table (old, carrying minus its
// sum, and new), any other vertex one, and each is expanded once.
//
// A warp takes a light row with a table of 128 entries, a CTA a row with more targets and
// a larger table, both hash tables in shared memory; rows that outgrow theirs are taken
// by a last launch, whose CTAs fall back to dense arrays in device memory.  Sums are
// fixed-point integers of two words, in units of 2^-119, added by atomics, so a row's result
// depends neither on the order of its arcs nor on the class it ran in.
//
// Bound by latency and by the instructions of short, uneven loops (ncu, light rows at
// n = 8192: 42 % of the issue slots, 17 % of the memory rate): per level of a walk the
// segment, an arc, its tail's distance; hence many rows in flight (a warp and 5.5 KB each)
// and several arcs of a lane in flight.  It replaced a walk per pair and state that listed
// the vertices found, and a second pass that evaluated sigma_sx * sigma_xt / sigma_st for
// each from rows s and t (Barabasi-Albert, 8 edges a vertex, weights 1..100): at n = 8192,
// 31,500 pairs an update, 267 us an update against 391, with 64-bit distances 348 against
// 443; 16 updates at n = 16384 8.6 ms against 11.4.  Of that: one walk for both states
// 560 -> 446 us an update at n = 16384 (a quarter fewer arcs, half the entries); two warps
// a CTA with 64 registers instead of 48 and more warps, 478 -> 436.
//
// Every undirected graph walks by default, alone and in a batch.  Per update alone, column
// test / walks: n = 512 153 / 79 us, 1024 168 / 89, 2048 159 / 104, 4096 246 / 157, 8192
// 547 / 271; 64-bit distances, n = 1500: 116 / 97.  A batch of 96 graphs of 32..512 vertices,
// 8 rounds: the column test's kernels 3.4 ms, the walks' 1.0.
#include <algorithm>

#include "bc_batch.cuh"
#include "bc_device.cuh"

namespace bcg {

namespace {

constexpr int kNone = -1;                 // the end of a list of DAG arcs
constexpr int kManyArcs = 96;               // vertices with as many are walked one by one
constexpr int kLightTargets = 16;         // rows with more changed targets: a CTA each

// The state of a graph as the walks read and write it.
template <typename DT>
struct WalkGraph {
    int n, ld, tcap;
    int cap;               // most entries of a shared-memory table to use
    const DT* D;
    const uint64_t* S;
    const DT* oD;          // values before the update, valid at the changed pairs
    const uint64_t* oS;
    const int32_t* tcnt;
    const int32_t* tlist;
    const int32_t* e_off;
    const int32_t* e_len;
    const Arc* e_arc;
    const int64_t* e_w64;
    ff* Dl;
    int64_t* bcfix;
    int64_t* stats;        // [8] rows and [9] pairs corrected [10] pairs walked [11] vertices found [12] arcs examined
    unsigned char* dense;  // dense_tables(n) tables
};
template <typename DT>
__host__ __device__ __forceinline__ WalkGraph<DT> walk_graph(const Dev& d) {
    WalkGraph<DT> a;
    a.n = d.n;
    a.ld = d.ld;
    a.tcap = d.tcap;
    a.cap = d.walk_cap < (1 << 20) ? (int)d.walk_cap : 1 << 20;
    a.D = (const DT*)d.D;
    a.S = d.S;
    a.oD = (const DT*)d.oldD;
    a.oS = d.oldS;
    a.tcnt = d.tcnt;
    a.tlist = d.tlist;
    a.e_off = d.e_off;
    a.e_len = d.e_len;
    a.e_arc = d.e_arc;
    a.e_w64 = d.e_w64;
    a.Dl = d.Dl;
    a.bcfix = d.bcfix;
    a.stats = d.stats;
    a.dense = reinterpret_cast<unsigned char*>(d.plan);
    return a;
}

// An update's edges in a batch (alone: WalkUpd).
struct BatchWalkUpd {
    int32_t v, k;
    const VEdge* ent;
    const int64_t* old_w;
    __device__ __forceinline__ int32_t x(int u) const { return ent[u].x; }
    __device__ __forceinline__ int64_t wold(int u) const { return old_w[u]; }
};
struct OneWalkUpd {
    int32_t v, k;
    const WalkUpd& upd;
    __device__ __forceinline__ int32_t x(int u) const { return upd.x[u]; }
    __device__ __forceinline__ int64_t wold(int u) const { return upd.wold[u]; }
};

template <typename DT>
struct WalkArgs {
    WalkGraph<DT> g;
    const int32_t* rows;   // rows that changed
    const int32_t* count;
    int32_t* full_rows;    // rows with more targets than tcap
    int32_t* full_count;
    int32_t* list[3];      // light rows, CTA rows, rows that outgrew their table
    int32_t* ctl;          // [0..2] rows in the lists [3..5] rows taken past each warp's or CTA's first
    const int32_t* err;
    WalkUpd upd;
};

// Each listed row to its class; the rows over the cap to those re-accumulated in full.
template <typename DT>
__global__ void __launch_bounds__(256) k_walk_class(const __grid_constant__ WalkArgs<DT> a) {
    pdl_enter();
    if (*a.err) return;
    const int cnt = *a.count;
    int rows = 0, tgts = 0;
    for (int i0 = blockIdx.x * blockDim.x; i0 < cnt; i0 += gridDim.x * blockDim.x) {   // warp-uniform
        const int i = i0 + threadIdx.x;
        const int s = i < cnt ? a.rows[i] : 0;
        const int T = i < cnt ? a.g.tcnt[s] : 0;
        append_row(T > a.g.tcap, s, a.full_rows, a.full_count);
        append_row(T > 0 && T <= min(kLightTargets, a.g.tcap), s, a.list[0], a.ctl + 0);
        append_row(T > kLightTargets && T <= a.g.tcap, s, a.list[1], a.ctl + 1);
        if (T <= a.g.tcap) {
            rows += T > 0;
            tgts += T;
        }
    }
    rows = __reduce_add_sync(FULL, rows);
    tgts = __reduce_add_sync(FULL, tgts);
    if ((threadIdx.x & 31) == 0 && rows) {
        atomicAdd(reinterpret_cast<unsigned long long*>(a.g.stats + 8), (unsigned long long)rows);
        atomicAdd(reinterpret_cast<unsigned long long*>(a.g.stats + 9), (unsigned long long)tgts);
        atomicAdd(reinterpret_cast<unsigned long long*>(a.g.stats + 10), (unsigned long long)tgts);
    }
}

// The same over a batch: the graphs whose update of round r walks.
__device__ __forceinline__ BatchWalkUpd batch_upd(const BatchArgs& b, int r, int g) {
    const BatchUpd& u = b.upd[(int64_t)r * b.G + g];
    return BatchWalkUpd{u.v, u.k, b.entries + u.first, b.wold + u.first};
}
__device__ __forceinline__ void append_pair(bool want, int2 gs, int2* list, int32_t* count) {
    const unsigned m = __ballot_sync(FULL, want);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    int p = 0;
    if (lane == 0) p = atomicAdd(count, __popc(m));
    p = __shfl_sync(FULL, p, 0) + __popc(m & ((1u << lane) - 1u));
    if (want) list[p] = gs;
}
__global__ void __launch_bounds__(256) kb_walk_class(BatchArgs b, int r) {
    const int64_t total = b.plan_pr[b.G];
    for (int64_t j0 = (int64_t)blockIdx.x * blockDim.x; j0 < total; j0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = j0 + threadIdx.x;
        int g = -1, s = 0, T = 0, cap = 0;
        if (j < total) {
            g = graph_of(b.plan_pr, b.G, j);
            const Dev& d = b.devs[g];
            if (batch_walks_graph(b, r, g)) {
                s = d.acc_rows[j - b.plan_pr[g]];
                T = d.tcnt[s];
                cap = d.tcap;
                if (T > cap) d.full_rows[atomicAdd(d.counts + 3, 1)] = s;
            }
        }
        const int2 gs = make_int2(g, s);
        append_pair(T > 0 && T <= min(kLightTargets, cap), gs, b.wlist, b.wctl + 0);
        append_pair(T > kLightTargets && T <= cap, gs, b.wlist + b.wrows, b.wctl + 1);
        // the counters of a graph, once per warp
        const unsigned peers = __match_any_sync(FULL, g);
        const int rows = __popc(__ballot_sync(FULL, T > 0 && T <= cap) & peers);
        const int tgts = __reduce_add_sync(peers, T <= cap ? T : 0);
        if (rows && (int)(threadIdx.x & 31) == __ffs(peers) - 1) {
            unsigned long long* st = reinterpret_cast<unsigned long long*>(b.devs[g].stats);
            atomicAdd(st + 8, (unsigned long long)rows);
            atomicAdd(st + 9, (unsigned long long)tgts);
            atomicAdd(st + 10, (unsigned long long)tgts);
        }
    }
}

// Counters of the group (warp or CTA) that has a row.
struct WalkShared {
    int seen;    // entries made, less the targets' without a path
    int bare;    // those
    int nodes;   // DAG arcs found
    int ready;   // entries whose children are done
    int over;    // the table is too small for the row
    int row;     // the next row
};

// A row's table.  An entry's key is 2 * vertex + 1, a target's old entry's 2 * vertex; -1
// where free.  IX numbers entries and DAG arcs ("nodes").
template <typename DT, typename IX>
struct WalkTable {
    uint64_t* sig;              // sigma_sx
    unsigned long long* acc;    // the difference's share of x so far, at a target with a path plus 1
                                // (old: all of it negative), in units of 2^-55,
    unsigned long long* low;    // and what is below that, in units of 2^-119
    DT* d;                      // d(s,x)
    int32_t* key;
    int32_t* head;              // DAG arcs into x: first node
    uint32_t* cnt;              // DAG children of x not done yet, in 16-bit halves (a vertex has fewer
                                // than n, and one more for each target with two entries)
    IX* seen;                   // entries made, in order (the targets first; without a path: not in it)
    IX* ready;                  // entries whose children are done, in order
    IX* node_x;                 // a DAG arc's tail
    IX* node_next;              // the next arc with the same head

    __host__ __device__ static constexpr size_t entry_bytes() {
        return sizeof(uint64_t) * 3 + sizeof(DT) + 2 * sizeof(int32_t) + sizeof(uint16_t) + 2 * sizeof(IX);
    }
    __host__ __device__ static constexpr size_t bytes(size_t entries, size_t nodes) {
        return ((entries + (entries & 1)) * entry_bytes() + nodes * 2 * sizeof(IX) + 15) & ~(size_t)15;
    }
    __device__ __forceinline__ WalkTable(unsigned char* p, size_t entries, size_t nodes) {
        entries += entries & 1;
        auto take = [&](size_t b) {
            unsigned char* q = p;
            p += b;
            return q;
        };
        sig = reinterpret_cast<uint64_t*>(take(8 * entries));
        acc = reinterpret_cast<unsigned long long*>(take(8 * entries));
        low = reinterpret_cast<unsigned long long*>(take(8 * entries));
        d = reinterpret_cast<DT*>(take(sizeof(DT) * entries));
        key = reinterpret_cast<int32_t*>(take(4 * entries));
        head = reinterpret_cast<int32_t*>(take(4 * entries));
        cnt = reinterpret_cast<uint32_t*>(take(2 * entries));
        seen = reinterpret_cast<IX*>(take(sizeof(IX) * entries));
        ready = reinterpret_cast<IX*>(take(sizeof(IX) * entries));
        node_x = reinterpret_cast<IX*>(take(sizeof(IX) * nodes));
        node_next = reinterpret_cast<IX*>(take(sizeof(IX) * nodes));
    }
    __device__ __forceinline__ void free_entry(int e) const {
        key[e] = -1;
        head[e] = kNone;
        reinterpret_cast<uint16_t*>(cnt)[e] = 0;
        acc[e] = low[e] = 0ull;
    }
    __device__ __forceinline__ bool no_children(int e) const { return reinterpret_cast<const uint16_t*>(cnt)[e] == 0; }
    __device__ __forceinline__ void count_child(int e) const { atomicAdd(cnt + (e >> 1), 1u << ((e & 1) << 4)); }
    __device__ __forceinline__ bool last_child(int e) const {
        const int sh = (e & 1) << 4;
        return ((atomicSub(cnt + (e >> 1), 1u << sh) >> sh) & 0xFFFFu) == 1u;
    }
    __device__ __forceinline__ __int128 sum(int e) const {
        const long long hi = (long long)*(volatile unsigned long long*)(acc + e);
        return ((__int128)hi << 64) + *(volatile unsigned long long*)(low + e);
    }
    // The low word's carry goes along; most shares have nothing below 2^-55.
    __device__ __forceinline__ void add(int e, __int128 v) const {
        unsigned long long hi = (unsigned long long)(v >> 64);
        const unsigned long long lo = (unsigned long long)v;
        if (lo) hi += atomicAdd(low + e, lo) + lo < lo;
        atomicAdd(acc + e, hi);
    }
    // All m entries (a multiple of four; the arrays start on 16-byte boundaries).
    __device__ __forceinline__ void free_all(int m, int rank, int threads) const {
        for (int i = rank; i < m / 4; i += threads) {
            reinterpret_cast<int4*>(key)[i] = make_int4(-1, -1, -1, -1);
            reinterpret_cast<int4*>(head)[i] = make_int4(kNone, kNone, kNone, kNone);
            reinterpret_cast<int2*>(cnt)[i] = make_int2(0, 0);
            const ulonglong2 none = make_ulonglong2(0ull, 0ull);
            reinterpret_cast<ulonglong2*>(acc)[2 * i] = reinterpret_cast<ulonglong2*>(acc)[2 * i + 1] = none;
            reinterpret_cast<ulonglong2*>(low)[2 * i] = reinterpret_cast<ulonglong2*>(low)[2 * i + 1] = none;
        }
    }
};

// v in (-2^8, 2^8) to units of 2^-119 and back.  A share is at least 2^-64 (one path of fewer
// than 2^64), so these keep every bit of a float-float, and sums of them by integer atomics
// are exact whatever their order.  (With 2^-55 and one word a share of 2^-40 kept 15 bits.)
// h - a, r - c and the products with powers of two are exact.
__device__ __forceinline__ __int128 to_units(ff v) {
    const float h = v.hi * 0x1p24f, a = rintf(h);
    float r0 = (h - a) * 0x1p31f, r1 = v.lo * 0x1p55f;   // units of 2^-55
    const float b0 = rintf(r0), b1 = rintf(r1);
    const long long hi = __float2ll_rn(a) * (1ll << 31) + __float2ll_rn(b0) + __float2ll_rn(b1);
    r0 -= b0;
    r1 -= b1;
    __int128 x = (__int128)hi << 64;
    if (r0 != 0.f || r1 != 0.f) {
        r0 *= 0x1p32f;
        r1 *= 0x1p32f;
        const float c0 = rintf(r0), c1 = rintf(r1);
        x += (__int128)(__float2ll_rn(c0) + __float2ll_rn(c1)) << 32;
        x += __float2ll_rn((r0 - c0) * 0x1p32f) + __float2ll_rn((r1 - c1) * 0x1p32f);
    }
    return x;
}
__device__ __forceinline__ float pow2f(int e) { return e < -126 ? 0.f : __int_as_float((e + 127) << 23); }
__device__ __forceinline__ ff from_units(__int128 v) {
    const unsigned __int128 m = v < 0 ? -(unsigned __int128)v : (unsigned __int128)v;
    const uint64_t m1 = (uint64_t)(m >> 64), m0 = (uint64_t)m;
    // its 64 leading bits, in units of 2^(-55 - z)
    const int z = m1 ? __clzll((long long)m1) : 64 + __clzll((long long)m0);
    const uint64_t top = z == 0 ? m1 : z < 64 ? (m1 << z) | (m0 >> (64 - z)) : z < 128 ? m0 << (z - 64) : 0ull;
    const ff r = ff_add(two_sum((float)(uint32_t)(top >> 40) * pow2f(-15 - z),
                                (float)((uint32_t)(top >> 16) & 0xFFFFFFu) * pow2f(-39 - z)),
                        ff{(float)((uint32_t)top & 0xFFFFu) * pow2f(-55 - z), 0.f});
    return v < 0 ? ff{-r.hi, -r.lo} : r;
}
constexpr long long kOne = 1ll << 55;   // 1 in acc

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// GS threads work on a row: a warp, or the CTA.  H: entries of the hash table (0: dense,
// entry = vertex, or n + j for the j-th target's old one, which the vertex's head names);
// NODES: room for DAG arcs (dense: none are kept, the arcs are read again).
template <typename DT, typename UPD, typename IX, int GS, int H, int NODES>
struct RowWalk {
    const WalkGraph<DT>& a;
    const UPD& upd;
    const WalkTable<DT, IX>& t;
    WalkShared& sh;
    int limit;   // entries from which the hash table counts as too small
    int s, T;    // the row and its changed targets
    unsigned long long* totals;   // vertices found, arcs examined (of this lane 0)

    __device__ __forceinline__ static void sync() {
        if (GS == 32) __syncwarp();
        else __syncthreads();
    }
    __device__ __forceinline__ static int rank() { return GS == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x; }
    __device__ __forceinline__ static int home(int k) {
        constexpr int bits = H == 0 ? 1 : 31 - __builtin_clz(H | 1);
        return (int)(((uint32_t)k * 2654435761u) >> (32 - bits));
    }
    // The entry of key k, or -1.  A hash table always has a free entry, so the probe ends:
    // past the limit every thread makes at most one more (see over()).
    __device__ __forceinline__ int find(int k) const {
        if constexpr (H == 0) {
            if (!(k & 1)) return *(volatile int32_t*)(t.head + (k >> 1));
            return *(volatile int32_t*)(t.key + (k >> 1)) == k ? k >> 1 : -1;
        } else {
            for (int e = home(k);; e = (e + 1) & (H - 1)) {
                const int c = *(volatile int32_t*)(t.key + e);
                if (c == k) return e;
                if (c == -1) return -1;
            }
        }
    }
    // The entry of key k (the j-th target's old one), made if there is none.
    __device__ __forceinline__ int insert(int k, int j, DT d, bool count, bool* made) const {
        for (int e = H != 0 ? home(k) : (k & 1) ? k >> 1 : a.n + j;; e = (e + 1) & (H - 1)) {
            const int c = atomicCAS(t.key + e, -1, k);
            if (c != -1 && c != k) continue;
            *made = c == -1;
            if (c == -1) {
                t.d[e] = d;
                if (H == 0 && !(k & 1)) t.head[k >> 1] = e;
                if (count) {
                    const int u = atomicAdd(&sh.seen, 1);
                    t.seen[u] = (IX)e;
                    if (H != 0 && u + *(volatile int*)&sh.bare >= limit) *(volatile int*)&sh.over = 1;
                } else {
                    atomicAdd(&sh.bare, 1);
                }
            }
            return e;
        }
    }
    // Warp-uniform; asked before each step that makes at most one entry per thread.
    __device__ __forceinline__ bool over() const { return H != 0 && __any_sync(FULL, *(volatile int*)&sh.over); }

    // The old weight of an arc between x and y that weighs w now (negative: it did not exist).
    __device__ __forceinline__ DT old_weight(DT w, int x, int y) const {
        if (y == upd.v || x == upd.v) {
            const int o = y == upd.v ? x : y;
            for (int u = 0; u < upd.k; ++u)
                if (upd.x(u) == o) w = (DT)min(upd.wold(u), Inf<DT>::v);
        }
        return w;
    }

    // The changed targets, each with an entry per state (2 * kPairCap of them fit any table).
    __device__ __forceinline__ void seed() const {
        const size_t rs = (size_t)s * a.ld;
        for (int j0 = 0; j0 < 2 * T; j0 += GS) {
            const int j = j0 + rank();
            if (j < 2 * T) {
                const int x = a.tlist[(size_t)s * a.tcap + (j >> 1)], st = j & 1;
                const uint64_t sg = st ? a.S[rs + x] : a.oS[rs + x];
                DT d = st ? a.D[rs + x] : a.oD[rs + x];
                if (sg == 0) d = (DT)Inf<DT>::v;
                bool made;
                const bool path = (int64_t)d != Inf<DT>::v;
                const int e = insert(2 * x + st, j >> 1, d, path, &made);
                t.sig[e] = sg;
                if (path) {
                    t.acc[e] = (unsigned long long)(st ? kOne : -kOne);
                    prefetch_l2(a.Dl + rs + x);
                }
            }
        }
    }

    // The arcs [0, tot) of a warp's vertices (lane's: entry and state in ey, distance dy, slots
    // from off + excl on), 32 * U at a time so that the loads of U arcs per
    // lane overlap.  ONE: all are vertex `one`'s; else an arc's owner is the last vertex j < nb
    // whose arcs start at or before it.
    template <bool ONE>
    __device__ __forceinline__ void expand(int ey, DT dy, int off, int excl, int tot, int nb, int one) const {
        const int lane = threadIdx.x & 31;
        const size_t rs = (size_t)s * a.ld;
        const int top = nb > 1 ? 1 << (31 - __clz(nb - 1)) : 0;
        if (ONE) {
            ey = __shfl_sync(FULL, ey, one);
            dy = __shfl_sync(FULL, dy, one);
            off = __shfl_sync(FULL, off, one);
        }
        constexpr int U = ONE ? 4 : 1;
        for (int k0 = 0; k0 < tot; k0 += 32 * U) {
            int ej[U], x[U];
            DT dyj[U], dx[U], w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                x[u] = -1;
                ej[u] = ey;
                dyj[u] = dy;
                if (k0 + 32 * u >= tot) continue;   // uniform
                const int k = k0 + 32 * u + lane;
                int at = off + k;
                if (!ONE) {
                    int j = 0;
                    for (int step = top; step >= 1; step >>= 1) {
                        const int c = j + step;
                        const int ex = __shfl_sync(FULL, excl, c & 31);
                        if (c < nb && ex <= k) j = c;
                    }
                    ej[u] = __shfl_sync(FULL, ey, j);
                    dyj[u] = __shfl_sync(FULL, dy, j);
                    at = __shfl_sync(FULL, off, j) + k;
                }
                if (k < tot) {
                    const Arc arc = a.e_arc[at];
                    x[u] = arc.dst();
                    w[u] = sizeof(DT) == 4 ? (DT)arc.w : (DT)a.e_w64[at];
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (x[u] < 0) continue;
                if (!(ej[u] & 1)) w[u] = old_weight(w[u], x[u], t.key[ej[u] >> 1] >> 1);
                if (x[u] == s || w[u] < 0 || w[u] > dyj[u]) x[u] = -1;   // no predecessor
                else dx[u] = a.D[rs + x[u]];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (k0 + 32 * u >= tot) continue;   // uniform
                bool is = false;
                int f = -1;
                int k = (x[u] << 1) | 1;
                const DT want = dyj[u] - w[u];   // below INF: dyj is
                if (x[u] >= 0) {
                    is = dx[u] == want;
                    if (!(ej[u] & 1)) {   // old: a target's distance is that of its old entry
                        f = find(k ^ 1);
                        if (f >= 0) {
                            k ^= 1;
                            is = t.d[f] == want;
                        }
                    }
                }
                if (!__any_sync(FULL, is)) continue;
                if (over()) return;
                if (is) {
                    if (f < 0) {
                        bool made;
                        f = insert(k, 0, want, true, &made);
                        if (made) {
                            prefetch_l2(a.S + rs + x[u]);
                            prefetch_l2(a.Dl + rs + x[u]);
                        }
                    }
                    t.count_child(f);
                    if (H != 0) {
                        const int q = atomicAdd(&sh.nodes, 1);
                        if (q < NODES) {
                            t.node_x[q] = (IX)f;
                            t.node_next[q] = (IX)atomicExch(t.head + (ej[u] >> 1), q);
                        } else {
                            *(volatile int*)&sh.over = 1;
                        }
                    }
                }
                __syncwarp();
            }
        }
    }

    // Backwards from the entries seen, level by level, a level's vertices shared out to the
    // warps.  Every DAG arc (x,y) counts in cnt[x], and is linked into y's list.
    __device__ __forceinline__ void walk() const {
        const int lane = threadIdx.x & 31;
        constexpr int W = GS / 32;
        const int wid = rank() >> 5;
        for (int lo = 0;;) {
            sync();
            const int hi = *(volatile int*)&sh.seen;
            const int ov = *(volatile int*)&sh.over;
            sync();
            if (lo >= hi || ov) break;
            const int per = W == 1 ? 32 : min(32, (hi - lo + W - 1) / W);
            for (int b0 = lo + wid * per; b0 < hi; b0 += W * per) {
                const int nb = min(per, hi - b0);
                int ey = 0;
                int off = 0, len = 0;
                DT dy = 0;
                if (lane < nb) {
                    const int e = t.seen[b0 + lane], k = t.key[e];
                    ey = 2 * e + (k & 1);
                    off = a.e_off[k >> 1];
                    len = a.e_len[k >> 1];
                    dy = t.d[e];
                }
                const int arcs = __reduce_add_sync(FULL, len);
                if (lane == 0) totals[1] += (unsigned)arcs;
                // vertices with many arcs one by one, the others together
                for (unsigned m = __ballot_sync(FULL, len >= kManyArcs); m; m &= m - 1) {
                    const int one = __ffs(m) - 1;
                    expand<true>(ey, dy, off, 0, __shfl_sync(FULL, len, one), nb, one);
                }
                if (len >= kManyArcs) len = 0;
                int incl = len;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int z = __shfl_up_sync(FULL, incl, o);
                    if (lane >= o) incl += z;
                }
                const int tot = __shfl_sync(FULL, incl, 31);
                expand<false>(ey, dy, off - (incl - len), incl - len, tot, nb, 0);
            }
            lo = hi;
        }
    }

    // What a vertex y whose children are done has for its DAG parents: its sum c, and the
    // sum over its path count, r, for parents with another count.
    struct Share {
        __int128 c;
        uint64_t sig;
        ff r;
    };
    __device__ __forceinline__ void share(int e, Share& h) const {
        h.c = t.sum(e);
        h.sig = t.sig[e];
        h.r.hi = -1.f;
        h.r.lo = 2.f;   // not computed (no float-float has |lo| > |hi|)
    }
    // One DAG arc (x,y): sigma_sx / sigma_sy of y's sum, which is the whole of it where x is
    // y's only parent, mostly.
    __device__ __forceinline__ void push(int f, Share& h) const {
        const uint64_t sx = t.sig[f];
        __int128 c = h.c;
        if (sx != h.sig) {
            if (h.r.lo == 2.f) h.r = ff_mul(from_units(h.c), ff_rcp(ff_from_u64(h.sig)));
            c = to_units(ff_mul(h.r, ff_from_u64(sx)));
        }
        t.add(f, c);
        if (t.last_child(f)) t.ready[atomicAdd(&sh.ready, 1)] = (IX)f;
    }

    // The recurrence: an entry pushes to its DAG parents once its own children are done.
    __device__ __forceinline__ void pull(int nseed) const {
        const size_t rs = (size_t)s * a.ld;
        const int seen = *(volatile int*)&sh.seen;
        for (int i = rank(); i < seen; i += GS) {
            const int e = t.seen[i];
            if (i >= nseed) t.sig[e] = a.S[rs + (t.key[e] >> 1)];
            if (t.no_children(e)) t.ready[atomicAdd(&sh.ready, 1)] = (IX)e;
        }
        for (int lo = 0;;) {
            sync();
            const int hi = *(volatile int*)&sh.ready;
            sync();
            if (lo >= hi) break;
            if (H != 0) {
                for (int i = lo + rank(); i < hi; i += GS) {
                    const int e = t.ready[i];
                    int q = t.head[e];
                    if (q < 0) continue;
                    Share r;
                    share(e, r);
                    while (q >= 0) {   // the list of y: at most NODES arcs
                        push(t.node_x[q], r);
                        q = t.node_next[q];
                        if (q == (int)(IX)kNone) q = kNone;
                    }
                }
            } else {   // a warp per entry; the arcs are read again
                for (int i = lo + (rank() >> 5); i < hi; i += GS / 32) {
                    const int e = t.ready[i], y = t.key[e] >> 1, st = t.key[e] & 1;
                    const int off = a.e_off[y], len = a.e_len[y];
                    const DT dy = t.d[e];
                    Share r;
                    share(e, r);
                    for (int k = threadIdx.x & 31; k < len; k += 32) {
                        const Arc arc = a.e_arc[off + k];
                        const int x = arc.dst();
                        DT w = sizeof(DT) == 4 ? (DT)arc.w : (DT)a.e_w64[off + k];
                        if (!st) w = old_weight(w, x, y);
                        if (x == s || w < 0 || w > dy) continue;
                        int f = st ? -1 : find(2 * x);
                        if (f < 0) f = find(2 * x + 1);
                        if (f >= 0 && t.d[f] == dy - w) push(f, r);
                    }
                }
            }
            lo = hi;
        }
    }

    // delta_s(x) and BC(x) change by the difference; a target's in its two entries.
    __device__ __forceinline__ void finish(int e) const {
        const int k = t.key[e];
        if (k < 0 || !(k & 1)) return;
        const int o = find(k ^ 1);
        __int128 v = t.sum(e);
        if (o >= 0) v += t.sum(o);
        if (v == 0) return;
        const int x = k >> 1;
        ff* p = a.Dl + (size_t)s * a.ld + x;
        *p = ff_add(*p, from_units(v));
        // units of 2^-24, 2^-71 and, of a small one, 2^-112
        FixWords w{(long long)(v >> 95), (long long)(v >> 48) & ((1ll << 47) - 1), 0};
        const long long rest = (long long)v & ((1ll << 48) - 1);
        if (w.A == 0 || w.A == -1) w.C = (rest + 64) >> 7;
        else w.B += rest >> 47;
        fix_add(a.bcfix, a.n, x, w);
    }

    // The whole row; false: it outgrew the table and nothing was written but the table.
    // The table is free before and after.
    __device__ __forceinline__ bool run() const {
        if (rank() == 0) sh.seen = sh.bare = sh.nodes = sh.ready = sh.over = 0;
        sync();
        seed();
        sync();
        const int nseed = *(volatile int*)&sh.seen;
        walk();
        const bool ok = *(volatile int*)&sh.over == 0;   // (walk ends with a sync)
        if (ok) {
            pull(nseed);
            for (int i = rank(); i < nseed; i += GS) {
                const int e = t.seen[i];
                t.acc[e] -= (unsigned long long)(t.key[e] & 1 ? kOne : -kOne);
            }
            sync();
            const int seen = *(volatile int*)&sh.seen;
            for (int i = rank(); i < seen; i += GS) finish(t.seen[i]);
            if (rank() == 0) totals[0] += (unsigned)(seen - nseed);
        }
        sync();
        if constexpr (H != 0) {
            t.free_all(H, rank(), GS);
        } else {
            const int m = *(volatile int*)&sh.seen;
            for (int i = rank(); i < m; i += GS) t.free_entry(t.seen[i]);
            for (int j = rank(); j < T; j += GS) {
                t.free_entry(a.tlist[(size_t)s * a.tcap + j]);
                t.free_entry(a.n + j);
            }
        }
        sync();
        return ok;
    }
};

// Light rows: a warp each.  16 CTAs' tables (with 32-bit distances) leave an SM 60 KB of L1, as
// do four of the CTA rows' (below): both are kept under 196 KB an SM.  With 6.4 and 51 KB, past
// it, 16 updates at n = 16384 took 9.5 ms instead of 9.1.
constexpr int kLightPerSm = 16, kLightWarps = 2, kLightH = 128, kLightLimit = kLightH - 33, kLightNodes = 192;
static_assert(kLightH <= 255 && kLightNodes < 255, "numbered in 8 bits");
template <typename DT> using LightTable = WalkTable<DT, uint8_t>;
template <typename DT>
__host__ __device__ constexpr size_t light_bytes() { return LightTable<DT>::bytes(kLightH, kLightNodes); }

template <typename DT, typename UPD>
__device__ __forceinline__ bool light_row(const WalkGraph<DT>& g, const UPD& upd, const LightTable<DT>& t,
                                          WalkShared& sh, int s, unsigned long long* totals) {
    const RowWalk<DT, UPD, uint8_t, 32, kLightH, kLightNodes> w{g, upd, t, sh, min(g.cap, kLightLimit), s, g.tcnt[s], totals};
    return w.run();
}
__device__ __forceinline__ void walk_totals(int64_t* stats, unsigned long long* totals) {
    if (totals[0]) atomicAdd(reinterpret_cast<unsigned long long*>(stats + 11), totals[0]);
    if (totals[1]) atomicAdd(reinterpret_cast<unsigned long long*>(stats + 12), totals[1]);
    totals[0] = totals[1] = 0ull;
}

template <typename DT>
__global__ void __launch_bounds__(kLightWarps * 32, kLightPerSm) k_walk_light(const __grid_constant__ WalkArgs<DT> a) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char wsm[];
    __shared__ WalkShared s_sh[kLightWarps];
    if (*a.err) return;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const LightTable<DT> t(wsm + wib * light_bytes<DT>(), kLightH, kLightNodes);
    t.free_all(kLightH, lane, 32);
    __syncwarp();
    const OneWalkUpd upd{a.upd.v, a.upd.k, a.upd};
    const int cnt = a.ctl[0], nw = gridDim.x * kLightWarps;
    unsigned long long totals[2] = {0ull, 0ull};
    for (int i = blockIdx.x * kLightWarps + wib; i < cnt;) {
        int nx = 0;   // the next row's number arrives while this one is worked on
        if (lane == 0) nx = nw + atomicAdd(a.ctl + 3, 1);
        const int s = a.list[0][i];
        if (!light_row(a.g, upd, t, s_sh[wib], s, totals) && lane == 0) a.list[2][atomicAdd(a.ctl + 2, 1)] = s;
        i = __shfl_sync(FULL, nx, 0);
    }
    if (lane == 0) walk_totals(a.g.stats, totals);
}

// The same over a batch: rows are (graph, row) pairs, a warp's graph is in shared memory.
template <typename DT>
__global__ void __launch_bounds__(kLightWarps * 32, kLightPerSm) kb_walk_light(BatchArgs b, int r) {
    extern __shared__ __align__(16) unsigned char wsm[];
    __shared__ WalkShared s_sh[kLightWarps];
    __shared__ WalkGraph<DT> s_g[kLightWarps];
    __shared__ BatchWalkUpd s_u[kLightWarps];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const LightTable<DT> t(wsm + wib * light_bytes<DT>(), kLightH, kLightNodes);
    t.free_all(kLightH, lane, 32);
    const int cnt = b.wctl[0], nw = gridDim.x * kLightWarps;
    unsigned long long totals[2] = {0ull, 0ull};
    int cg = -1;
    for (int i = blockIdx.x * kLightWarps + wib; i < cnt;) {
        int nx = 0;
        if (lane == 0) nx = nw + atomicAdd(b.wctl + 3, 1);
        const int2 gs = b.wlist[i];
        if (gs.x != cg) {
            if (lane == 0) {
                if (cg >= 0) walk_totals(s_g[wib].stats, totals);
                s_g[wib] = walk_graph<DT>(b.devs[gs.x]);
                s_u[wib] = batch_upd(b, r, gs.x);
            }
            cg = gs.x;
        }
        __syncwarp();
        if (!light_row(s_g[wib], s_u[wib], t, s_sh[wib], gs.y, totals) && lane == 0)
            b.wlist[2 * b.wrows + atomicAdd(b.wctl + 2, 1)] = gs;
        i = __shfl_sync(FULL, nx, 0);
    }
    if (lane == 0 && cg >= 0) walk_totals(s_g[wib].stats, totals);
}

// Rows with more targets (RETRY: rows that outgrew their table, in the dense arrays if
// they outgrow this one too): a CTA each.  A light row has at most 16 targets (22 entries
// in the mean, and up to 95 fit); one of more has some hundred entries.  256 threads and 1024
// entries, four CTAs an SM, took 421 us an update at n = 16384 where 512 entries and eight
// CTAs took 432, and a CTA of 64 threads 475.
template <bool RETRY>
struct Cta {
    static_assert(4 * kPairCap <= 512 && 2 * kLightTargets < kLightH, "room for the targets");
    static constexpr int threads = RETRY ? 512 : 256, h = RETRY ? 2048 : 1024, limit = h - threads - 1,
                         nodes = RETRY ? 3072 : 1408, per_sm = RETRY ? 1 : 4;
    template <typename DT>
    __host__ __device__ static constexpr size_t bytes() { return WalkTable<DT, uint16_t>::bytes(h, nodes); }
};

// A dense table: the vertices, then the targets' old entries.
__host__ __device__ constexpr int dense_entries(int n) { return n + (n < kPairCap ? n : kPairCap); }

template <typename DT, bool RETRY, typename UPD>
__device__ __forceinline__ bool cta_row(const WalkGraph<DT>& g, const UPD& upd, const WalkTable<DT, uint16_t>& t,
                                        WalkShared& sh, int s, unsigned long long* totals, bool& dense_free) {
    using C = Cta<RETRY>;
    const int T = g.tcnt[s];
    const RowWalk<DT, UPD, uint16_t, C::threads, C::h, C::nodes> w{g, upd, t, sh, min(g.cap, C::limit), s, T, totals};
    if (w.run()) return true;
    if constexpr (RETRY) {
        const int m = dense_entries(g.n);
        const WalkTable<DT, int32_t> dt(g.dense + blockIdx.x * WalkTable<DT, int32_t>::bytes(m, 0), m, 0);
        if (!dense_free) {   // (what was there before: another update's plan)
            for (int e = threadIdx.x; e < m; e += C::threads) dt.free_entry(e);
            __syncthreads();
        }
        dense_free = true;
        const RowWalk<DT, UPD, int32_t, C::threads, 0, 0> dw{g, upd, dt, sh, 0, s, T, totals};
        return dw.run();
    }
    return false;
}

template <typename DT, bool RETRY>
__global__ void __launch_bounds__(Cta<RETRY>::threads, Cta<RETRY>::per_sm) k_walk_cta(const __grid_constant__ WalkArgs<DT> a) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char wsm[];
    __shared__ WalkShared sh;
    if (*a.err) return;
    using C = Cta<RETRY>;
    constexpr int L = RETRY ? 2 : 1;
    const int cnt = a.ctl[L];
    if ((int)blockIdx.x >= cnt) return;
    const WalkTable<DT, uint16_t> t(wsm, C::h, C::nodes);
    t.free_all(C::h, threadIdx.x, C::threads);
    const OneWalkUpd upd{a.upd.v, a.upd.k, a.upd};
    unsigned long long totals[2] = {0ull, 0ull};
    bool dense_free = false;
    for (int i = blockIdx.x; i < cnt;) {
        int nx = 0;
        if (threadIdx.x == 0) nx = (int)gridDim.x + atomicAdd(a.ctl + 3 + L, 1);
        const int s = a.list[L][i];
        if (!cta_row<DT, RETRY>(a.g, upd, t, sh, s, totals, dense_free) && threadIdx.x == 0)
            a.list[2][atomicAdd(a.ctl + 2, 1)] = s;
        if (threadIdx.x == 0) sh.row = nx;
        __syncthreads();
        i = sh.row;
        __syncthreads();
    }
    if ((threadIdx.x & 31) == 0) walk_totals(a.g.stats, totals);
}

template <typename DT, bool RETRY>
__global__ void __launch_bounds__(Cta<RETRY>::threads, Cta<RETRY>::per_sm) kb_walk_cta(BatchArgs b, int r) {
    extern __shared__ __align__(16) unsigned char wsm[];
    __shared__ WalkShared sh;
    __shared__ WalkGraph<DT> s_g;
    __shared__ BatchWalkUpd s_u;
    using C = Cta<RETRY>;
    constexpr int L = RETRY ? 2 : 1;
    const int cnt = b.wctl[L];
    if ((int)blockIdx.x >= cnt) return;
    const WalkTable<DT, uint16_t> t(wsm, C::h, C::nodes);
    t.free_all(C::h, threadIdx.x, C::threads);
    unsigned long long totals[2] = {0ull, 0ull};
    int cg = -1;
    bool dense_free = false;
    for (int i = blockIdx.x; i < cnt;) {
        int nx = 0;
        if (threadIdx.x == 0) nx = (int)gridDim.x + atomicAdd(b.wctl + 3 + L, 1);
        const int2 gs = b.wlist[L * b.wrows + i];
        if (gs.x != cg) {
            if (cg >= 0 && (threadIdx.x & 31) == 0) walk_totals(s_g.stats, totals);
            __syncthreads();
            if (threadIdx.x == 0) {
                s_g = walk_graph<DT>(b.devs[gs.x]);
                s_u = batch_upd(b, r, gs.x);
            }
            cg = gs.x;
            dense_free = false;
        }
        __syncthreads();
        if (!cta_row<DT, RETRY>(s_g, s_u, t, sh, gs.y, totals, dense_free) && threadIdx.x == 0)
            b.wlist[2 * b.wrows + atomicAdd(b.wctl + 2, 1)] = gs;
        if (threadIdx.x == 0) sh.row = nx;
        __syncthreads();
        i = sh.row;
        __syncthreads();
    }
    if (cg >= 0 && (threadIdx.x & 31) == 0) walk_totals(s_g.stats, totals);
}

template <typename DT>
WalkArgs<DT> walk_args(const Dev& d) {
    WalkArgs<DT> a{};
    a.g = walk_graph<DT>(d);
    a.rows = d.acc_rows;
    a.count = d.counts + 1;
    a.full_rows = d.full_rows;
    a.full_count = d.counts + 3;
    a.list[0] = d.pair_rows;
    a.list[1] = d.walk_rows;
    a.list[2] = d.walk_rows + d.n;
    a.ctl = d.counts + 8;
    a.err = d.err;
    return a;
}

// The dense tables take the place of the column test's plan, which an update that walks has
// no use for: as many of them as fit.
template <typename DT>
int dense_tables(int n) {
    return (int)((size_t)n * kPairCap * kPairPlanBytes / WalkTable<DT, int32_t>::bytes(dense_entries(n), 0));
}
// The least of dense_tables (n = 1, 64-bit distances; a batch's graphs have any n).
constexpr int kDenseTablesMin =
    (int)((size_t)kPairCap * kPairPlanBytes / WalkTable<int64_t, int32_t>::bytes(dense_entries(1), 0));
static_assert(kDenseTablesMin >= 40, "CTAs for the rows that outgrow shared memory");

template <typename DT>
void walks(const Dev& d, const WalkUpd& upd, cudaEvent_t ready) {
    WalkArgs<DT> a = walk_args<DT>(d);
    a.upd = upd;
    // rows of CTAs on the third stream beside the light ones, then those that outgrew
    // their table
    const cudaStream_t sr = ready ? d.st3 : d.st;
    if (ready) cudaStreamWaitEvent(sr, ready, 0);
    launch_k(k_walk_cta<DT, false>, d.nsm * Cta<false>::per_sm, Cta<false>::threads, Cta<false>::bytes<DT>(), sr, a);
    if (ready) cudaEventRecord(d.ev3_join, sr);
    launch_k(k_walk_light<DT>, d.nsm * kLightPerSm, kLightWarps * 32, kLightWarps * light_bytes<DT>(), d.st, a);
    if (ready) cudaStreamWaitEvent(d.st, d.ev3_join, 0);
    launch_k(k_walk_cta<DT, true>, std::min(d.nsm, dense_tables<DT>(d.n)), Cta<true>::threads, Cta<true>::bytes<DT>(), d.st, a);
}

template <typename DT>
cudaError_t setup() {
    auto allow = [](auto kern, size_t smem) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    };
    cudaError_t e = allow(k_walk_cta<DT, false>, Cta<false>::bytes<DT>());
    if (e == cudaSuccess) e = allow(kb_walk_cta<DT, false>, Cta<false>::bytes<DT>());
    if (e == cudaSuccess) e = allow(k_walk_cta<DT, true>, Cta<true>::bytes<DT>());
    if (e == cudaSuccess) e = allow(kb_walk_cta<DT, true>, Cta<true>::bytes<DT>());
    return e;
}

template <typename DT>
void batch_walks(const BatchArgs& b, int nsm, int r, cudaStream_t st) {
    kb_walk_cta<DT, false><<<nsm * Cta<false>::per_sm, Cta<false>::threads, Cta<false>::bytes<DT>(), st>>>(b, r);
    kb_walk_light<DT><<<nsm * kLightPerSm, kLightWarps * 32, kLightWarps * light_bytes<DT>(), st>>>(b, r);
    kb_walk_cta<DT, true><<<std::min(nsm, kDenseTablesMin), Cta<true>::threads, Cta<true>::bytes<DT>(), st>>>(b, r);
}

}  // namespace

cudaError_t walk_setup() {
    const cudaError_t e = setup<int32_t>();
    return e == cudaSuccess ? setup<int64_t>() : e;
}

void batch_walk_class(const BatchArgs& b, const BatchLaunch& L, int r, cudaStream_t st) {
    kb_walk_class<<<L.nsm * 8, 256, 0, st>>>(b, r);
}
void batch_walk_launches(const BatchArgs& b, const BatchLaunch& L, int r, int dbytes, cudaStream_t st) {
    if (dbytes == 4) batch_walks<int32_t>(b, L.nsm, r, st);
    else batch_walks<int64_t>(b, L.nsm, r, st);
}

void launch_walk_class(const Dev& d) {
    const int grid = std::max(1, std::min((d.n + 255) / 256, d.nsm * 4));
    if (d.dbytes == 4) launch_k(k_walk_class<int32_t>, grid, 256, 0, d.st, walk_args<int32_t>(d));
    else launch_k(k_walk_class<int64_t>, grid, 256, 0, d.st, walk_args<int64_t>(d));
}

void launch_walks(const Dev& d, const WalkUpd& upd, cudaEvent_t ready) {
    if (d.dbytes == 4) walks<int32_t>(d, upd, ready);
    else walks<int64_t>(d, upd, ready);
}

}  // namespace bcg
