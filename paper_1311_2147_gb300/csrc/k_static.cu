// k_static.cu -- the all-pairs distances of the static computation.
//
// bc_init_static needs d(s,t) for every pair before E* can be read off it.  Brandes
// (Appendix, Algorithm 7) runs Dijkstra from every source; a priority queue does not
// map well onto a CTA, so each CTA runs a label-correcting (Bellman-Ford) search from a
// group of sources at a time: every round relaxes, a lane per arc, the arcs whose tail's
// distance dropped in the round before, until no distance drops.  With positive weights
// this ends after at most n-1 rounds with the same distances Dijkstra settles.
//
// What bounds it: shared-memory gathers (two per arc, source and round in which the tail
// changed; the random one takes about three bank cycles) and, for few sources per group,
// the arcs' L2 reads of every round.  The arcs are read in order, 8 bytes each, once per
// round for all sources of the group (or, in rounds of few changed vertices, these
// vertices' arcs); before, a warp took the changed vertices of one source one after the
// other, a chain of two L2 reads each.  Static search, before and now: BA n = 4096 5.04 and
// 1.66 ms, ER n = 3001 (int64) 2.31 and 0.64 ms, BA n = 16384 90 and 42 ms, grid 128 x 128
// 300 and 112 ms.
//
// E* (Section 1: arcs on some shortest path) is then {(a,b) : w(a,b) = d(a,b)}: the
// one-arc path a->b is shortest exactly when the arc lies on a shortest path (a
// sub-path of a shortest path is shortest).
//
// Dense graphs (Section 6, Algorithm 6 step 1: the Hidden Paths algorithm examines only
// arcs of E*; a search may use any set of arcs that contains E*): a first search over each
// vertex's lightest arcs bounds every distance from above, arcs longer than that bound
// are not in E*, and the search runs over the others.  Hidden Paths finds E* exactly, in
// one global distance order over all sources; this finds a little more than E* and keeps
// the sources independent.
#include <algorithm>
#include <type_traits>

#include "bc_internal.cuh"

namespace bcg {

constexpr int kSsspMaxSources = 16;   // sources of a group (bits of a change mask)

__device__ __forceinline__ void atomic_min_dist(uint32_t* p, uint32_t v) { atomicMin(p, v); }
__device__ __forceinline__ void atomic_min_dist(int64_t* p, int64_t v) {
    atomicMin(reinterpret_cast<long long*>(p), (long long)v);
}
template <typename DS> struct Far;
template <> struct Far<uint32_t> { static constexpr uint32_t v = INT32_MAX; };
template <> struct Far<int64_t> { static constexpr int64_t v = INT64_MAX; };

// d(s,b) through an arc of weight w, or at least Far where the sum does not fit.
__device__ __forceinline__ uint32_t through(uint32_t d, uint32_t w) { return d + w; }   // both below 2^31
__device__ __forceinline__ int64_t through(int64_t d, int64_t w) { return w > INT64_MAX - 1 - d ? INT64_MAX : d + w; }

template <typename DT>
struct SsspArgs {
    int n, ld;
    const Arc* arc;        // arcs, by tail
    const int64_t* w64;    // their weights in full (int64 distances)
    const unsigned long long* arcs;   // their number
    const int32_t* off;    // [n + 1] first arc of each tail (NULL: they are in no order)
    DT* D;
    int32_t* err;
    int S;                 // sources of a group
    int check;             // a distance might not fit its type
};

// What a CTA keeps in shared memory.  Groups: S distance rows and 16 mask bits per vertex.
// Where not even one such row and its masks fit (n above 28672, or 19104 with 64-bit
// rows), one source at a time: its row and one mask bit per vertex, and where that does not
// fit either (64-bit rows, n above 27776), the mask bits alone, the distances in the
// source's row of D.  bc_init_static's device time, G(n, 4n) directed: kOne 129 ms at
// n = 29100 (32-bit) and 72 ms at n = 20000 (64-bit rows), kOneInD 328 ms at n = 32768; with a
// search of the changed vertices' arcs, source by source, these took 565, 297 and 560 ms.
enum class SsspForm { kGroups, kOne, kOneInD };

// Two change masks, one bit per vertex and source of the group: whether its distance
// dropped in the last round (cur) or in this one (nxt).
template <bool GROUPS>
struct SsspMask {
    static __host__ __device__ constexpr int words(int np) { return GROUPS ? np / 2 : np / 32; }
    static __device__ __forceinline__ unsigned get(const uint32_t* m, int x) {
        if (GROUPS) return reinterpret_cast<const volatile uint16_t*>(m)[x];
        return (*reinterpret_cast<const volatile uint32_t*>(m + (x >> 5)) >> (x & 31)) & 1u;
    }
    static __device__ __forceinline__ void set(uint32_t* m, int x, int k) {
        if (GROUPS) atomicOr(m + (x >> 1), (1u << k) << ((x & 1) << 4));
        else atomicOr(m + (x >> 5), 1u << (x & 31));
    }
    // Returns x's bits before.
    static __device__ __forceinline__ unsigned set_old(uint32_t* m, int x, int k) {
        if (GROUPS) return (atomicOr(m + (x >> 1), (1u << k) << ((x & 1) << 4)) >> ((x & 1) << 4)) & 0xFFFFu;
        return (atomicOr(m + (x >> 5), 1u << (x & 31)) >> (x & 31)) & 1u;
    }
    // By x's own thread alone.
    static __device__ __forceinline__ void clear(uint32_t* m, int x) {
        if (GROUPS) *reinterpret_cast<volatile uint16_t*>(reinterpret_cast<uint16_t*>(m) + x) = 0;
        else atomicAnd(m + (x >> 5), ~(1u << (x & 31)));
    }
};

// Rounds in which few vertices changed go over these vertices' arcs only (LISTS).  A round
// over all arcs costs the same however few changed, and on a path or a cycle nearly every
// round has a vertex or two per source.  Search without and with lists: path of n = 1024
// 1.56 and 0.91 ms, 4096 22.6 and 8.6 ms (64-bit rows 46 and 15.7), 16384 2860 and 590 ms;
// BA n = 4096, whose last rounds change few, 1.72 and 1.66 ms.  A round goes over a list where
// that is at most a quarter as long as there are vectors of 32 arcs.
constexpr int kSsspList = 512;
constexpr int kListsMinN = 2048;
struct SsspLists {
    int n[3];                      // vertices listed for a round, by round modulo 3
    uint16_t v[2][kSsspList];      // by round modulo 2 (more than fit are only counted)
};

// A group of S sources per CTA: their distance rows (DS) and the two change masks.  A round
// goes over all arcs, a lane per arc; a vector of 32 arcs is skipped for the sources in
// which none of its tails changed.  Or, where few vertices are listed as changed, over the
// arcs of 32 of these at a time.
template <typename DT, typename DS, int T, SsspForm F, bool LISTS>
__global__ void __launch_bounds__(T, 1024 / T) k_sssp(SsspArgs<DT> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SsspLists sh;
    constexpr bool kRowInD = F == SsspForm::kOneInD;
    static_assert(!kRowInD || sizeof(DS) == sizeof(DT), "the search's rows are D's");
    using Mask = SsspMask<F == SsspForm::kGroups>;
    const int n = a.n, np = (n + 31) & ~31, words = Mask::words(np);
    DS* const rows = reinterpret_cast<DS*>(smem);
    uint32_t* cur = reinterpret_cast<uint32_t*>(smem + (kRowInD ? 0 : (size_t)a.S * np * sizeof(DS)));
    uint32_t* nxt = cur + words;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = T / 32, U = 4;
    const int64_t arcs = (int64_t)*a.arcs;
    const int nchunk = (int)((arcs + 31) >> 5);
    const int few = LISTS && a.off ? min(kSsspList, nchunk / 4) : 0;   // vertices, for a round over a list
    for (int s0 = blockIdx.x * a.S; s0 < n; s0 += gridDim.x * a.S) {
        if (block_err(a.err)) return;
        const int S = min(a.S, n - s0);
        DS* const dist = kRowInD ? reinterpret_cast<DS*>(a.D + (size_t)s0 * a.ld) : rows;
        for (int t = tid; t < (kRowInD ? a.ld : S * np); t += T) dist[t] = Far<DS>::v;
        for (int t = tid; t < words; t += T) cur[t] = nxt[t] = 0u;
        __syncthreads();
        if (tid < S) {
            dist[(size_t)tid * np + s0 + tid] = (DS)0;
            Mask::set(cur, s0 + tid, tid);
            sh.v[0][tid] = (uint16_t)(s0 + tid);
        }
        if (tid < 3) sh.n[tid] = tid == 0 ? S : 0;
        __syncthreads();
        bool converged = false;
        bool listed = LISTS && S <= few;   // the vertices in cur are all in this round's list
        for (int round = 0; round <= n; ++round) {
            const uint16_t* const list = sh.v[round & 1];
            uint16_t* const list_next = sh.v[(round + 1) & 1];
            int* const n_next = &sh.n[(round + 1) % 3];
            int changed;
            if (LISTS && listed) {
                const int count = sh.n[round % 3], per = min(32, (count + NW - 1) / NW);
                if (tid == 0) sh.n[(round + 2) % 3] = 0;
                for (int b0 = warp * per; b0 < count; b0 += NW * per) {   // warp-uniform
                    int x = 0, beg = 0, len = 0;
                    unsigned mine = 0;
                    if (lane < min(per, count - b0)) {
                        x = list[b0 + lane];
                        beg = a.off[x];
                        len = a.off[x + 1] - beg;
                        mine = Mask::get(cur, x);
                        Mask::clear(cur, x);
                    }
                    int incl = len;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int z = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += z;
                    }
                    const int tot = __shfl_sync(0xffffffffu, incl, 31), excl = incl - len;
                    for (int k0 = 0; k0 < tot; k0 += 32) {
                        // the arc's tail: the last vertex whose arcs start at or before it
                        int j = 0;
#pragma unroll
                        for (int step = 16; step >= 1; step >>= 1) {
                            const int ex = __shfl_sync(0xffffffffu, excl, j + step);
                            if (ex <= k0 + lane) j += step;
                        }
                        const int xj = __shfl_sync(0xffffffffu, x, j);
                        const int64_t e = __shfl_sync(0xffffffffu, beg - excl, j) + k0 + lane;
                        unsigned m = __shfl_sync(0xffffffffu, mine, j);
                        if (k0 + lane >= tot) continue;
                        const Arc r = a.arc[e];
                        const DS w = sizeof(DS) == 8 ? (DS)a.w64[e] : (DS)r.w;
                        for (; m; m &= m - 1u) {
                            const int k = __ffs(m) - 1, b = r.dst();
                            DS* d = dist + (size_t)k * np;
                            const DS nd = through(*(volatile DS*)(d + xj), w);
                            if (nd >= *(volatile DS*)(d + b)) continue;
                            atomic_min_dist(d + b, nd);
                            if (Mask::set_old(nxt, b, k) != 0u) continue;   // listed already
                            const int p = atomicAdd(n_next, 1);
                            if (p < kSsspList) list_next[p] = (uint16_t)b;
                        }
                    }
                }
                __syncthreads();
                changed = *n_next;
                listed = changed <= few;
            } else {
                bool any = false;
                if (tid == 0) sh.n[(round + 2) % 3] = 0;
                for (int c0 = warp * U; c0 < nchunk; c0 += U * NW) {
                    Arc r[U];
                    int64_t w[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int64_t e = ((int64_t)(c0 + u) << 5) + lane;
                        r[u] = empty_arc();
                        w[u] = 0;
                        if (e < arcs) {
                            r[u] = a.arc[e];
                            if (sizeof(DS) == 8) w[u] = a.w64[e];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int x = r[u].src(), b = r[u].dst();
                        const unsigned mine = r[u].empty() ? 0u : Mask::get(cur, x);
                        for (unsigned m = __reduce_or_sync(0xffffffffu, mine); m; m &= m - 1u) {
                            const int k = __ffs(m) - 1;
                            if (!((mine >> k) & 1u)) continue;
                            DS* d = dist + (size_t)k * np;
                            const DS dx = *(volatile DS*)(d + x);
                            const DS nd = through(dx, sizeof(DS) == 8 ? (DS)w[u] : (DS)r[u].w);
                            if (nd < *(volatile DS*)(d + b)) {
                                atomic_min_dist(d + b, nd);
                                Mask::set(nxt, b, k);
                                any = true;
                            }
                        }
                    }
                }
                changed = __syncthreads_count(any);   // threads that found one
                listed = false;
                for (int q = tid; q < words; q += T) cur[q] = 0u;
                if (LISTS && changed <= min(few, T / 4)) {   // block-uniform: perhaps few vertices
                    for (int q = tid; q < words; q += T) {
                        constexpr int per_word = F == SsspForm::kGroups ? 2 : 32;
                        uint32_t w = nxt[q];
                        for (int i = 0; w; ++i, w = per_word == 2 ? w >> 16 : w >> 1) {
                            if (!(w & (per_word == 2 ? 0xFFFFu : 1u))) continue;
                            const int p = atomicAdd(n_next, 1);
                            if (p < kSsspList) list_next[p] = (uint16_t)(q * per_word + i);
                        }
                    }
                    __syncthreads();
                    listed = *n_next <= few;
                } else {
                    __syncthreads();
                }
            }
            if (changed == 0) {
                converged = true;
                break;
            }
            uint32_t* t = cur;
            cur = nxt;
            nxt = t;
        }
        // positive weights converge within n-1 rounds; anything else is reported
        if (!converged && tid == 0) set_err(a.err, ERRF_TIMEOUT);
        // An arc from a vertex with a distance to one without: their sum did not fit, so
        // that vertex has a distance the type cannot hold.
        if (a.check)
            for (int64_t e = tid; e < arcs; e += T) {
                const Arc r = a.arc[e];
                for (int k = 0; k < S; ++k)
                    if (dist[(size_t)k * np + r.src()] != Far<DS>::v && dist[(size_t)k * np + r.dst()] == Far<DS>::v)
                        set_err(a.err, ERRF_DIST);
            }
        if constexpr (!kRowInD)
            for (int k = 0; k < S; ++k) {
                DT* row = a.D + (size_t)(s0 + k) * a.ld;
                for (int t = tid; t < a.ld; t += T) {   // the entries past n: no path
                    const DS d = t < n ? dist[(size_t)k * np + t] : Far<DS>::v;
                    row[t] = d == Far<DS>::v ? (DT)Inf<DT>::v : (DT)d;
                }
            }
        __syncthreads();
    }
}

template <typename DT>
__global__ void k_estar_flags(int ld, int64_t arcs, const Arc* arc, const int64_t* w64, const DT* D, uint8_t* flags) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= arcs) return;
    const Arc r = arc[e];
    const int64_t w = sizeof(DT) == 8 ? w64[e] : (int64_t)r.w;
    flags[e] = ((int64_t)D[(size_t)r.src() * ld + r.dst()] == w) ? 1 : 0;
}

// ---- dense graphs: arcs that cannot be in E* left out before the search
//
// A path is at most as long as one over each vertex's lightest arcs only, so an arc longer
// than that path is not shortest and not in E*, and the search may leave it out.

constexpr int kLight = 12;   // lightest arcs of a vertex, at least (with equal weights up to twice that)

// A warp per vertex: appends its kLight lightest arcs (all of them when there are no more)
// to the list, the threshold found by bisection on the weight.
__global__ void __launch_bounds__(256) k_light_arcs(int n, const int32_t* off, const Arc* arc, const int64_t* w64,
                                                    int64_t w_max, Arc* l_arc, int64_t* l_w64,
                                                    unsigned long long* l_count) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    for (int x = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < n; x += (gridDim.x * blockDim.x) >> 5) {
        const int beg = off[x], end = off[x + 1];
        auto weight = [&](int e) { return w64 ? w64[e] : (int64_t)arc[e].w; };
        int64_t lo = 0, hi = w_max;
        while (lo < hi && end - beg > kLight) {   // least threshold with kLight arcs at or below it
            const int64_t mid = lo + (hi - lo) / 2;
            int c = 0;
            for (int e = beg + lane; e < end; e += 32) c += weight(e) <= mid;
            if (__reduce_add_sync(0xffffffffu, c) >= kLight) hi = mid;
            else lo = mid + 1;
        }
        int left = 2 * kLight;   // warp-uniform
        for (int e0 = beg; e0 < end && left > 0; e0 += 32) {
            const int e = e0 + lane;
            const bool light = e < end && weight(e) <= hi;
            const unsigned b = __ballot_sync(0xffffffffu, light);
            const int c = min(__popc(b), left), rank = __popc(b & lt);
            left -= c;
            unsigned long long p = 0;
            if (lane == 0 && c) p = atomicAdd(l_count, (unsigned long long)c);
            p = __shfl_sync(0xffffffffu, p, 0);
            if (light && rank < c) {
                l_arc[p + rank] = arc[e];
                if (w64) l_w64[p + rank] = w64[e];
            }
        }
    }
}

// Appends the arcs that are no longer than the distances of the search over the light ones.
template <typename DT>
__global__ void __launch_bounds__(256) k_filter_arcs(int ld, int64_t arcs, const Arc* arc, const int64_t* w64,
                                                     const DT* D, Arc* f_arc, int64_t* f_w64,
                                                     unsigned long long* f_count) {
    const int lane = threadIdx.x & 31;
    for (int64_t e0 = (int64_t)blockIdx.x * blockDim.x; e0 < arcs; e0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = e0 + threadIdx.x;
        bool keep = false;
        Arc r = empty_arc();
        int64_t w = 0;
        if (e < arcs) {
            r = arc[e];
            w = sizeof(DT) == 8 ? w64[e] : (int64_t)r.w;
            keep = w <= (int64_t)D[(size_t)r.src() * ld + r.dst()];
        }
        const unsigned b = __ballot_sync(0xffffffffu, keep);
        unsigned long long p = 0;
        if (lane == 0 && b) p = atomicAdd(f_count, (unsigned long long)__popc(b));
        p = __shfl_sync(0xffffffffu, p, 0) + __popc(b & ((1u << lane) - 1u));
        if (keep) {
            f_arc[p] = r;
            if (sizeof(DT) == 8) f_w64[p] = w;
        }
    }
}

// Most shared memory of a search CTA, and what its kernels are allowed (the allowance
// belongs to the kernel, which other host threads may be launching: none sets less).
constexpr size_t kSsspSmemMax = 224 * 1024;

template <typename DT, typename DS, int T, SsspForm F, bool LISTS>
static void sssp_launch(const Dev& d, const SsspArgs<DT>& a, size_t smem) {
    auto kern = k_sssp<DT, DS, T, F, LISTS>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSsspSmemMax);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, T, smem);
    const int grid = std::min(d.nsm * std::max(per_sm, 1), (d.n + a.S - 1) / a.S);
    kern<<<grid, T, smem, d.st>>>(a);
}

// arcs_about: the number of arcs, for the choice of S (it is known only on the device).
template <typename DT, typename DS>
static void sssp_search(const Dev& d, const Arc* arc, const int64_t* w64, const unsigned long long* arcs,
                        const int32_t* off, double arcs_about, bool check) {
    const size_t np = ((size_t)d.n + 31) & ~(size_t)31;
    SsspArgs<DT> a{d.n, d.ld, arc, w64, arcs, off, (DT*)d.D, d.err, 1, check ? 1 : 0};
    auto bytes = [&](int S) { return (size_t)S * np * sizeof(DS) + 2 * np * 2; };
    if (bytes(1) > kSsspSmemMax) {
        const size_t masks = 2 * (np / 8), one = np * sizeof(DS) + masks;
        if constexpr (sizeof(DS) == sizeof(int64_t)) {
            // (a row of D: as many threads an SM, in small CTAs, which wait for it one by one)
            if (one > kSsspSmemMax) return sssp_launch<DT, DS, 256, SsspForm::kOneInD, true>(d, a, masks);
        }
        return sssp_launch<DT, DS, 1024, SsspForm::kOne, true>(d, a, one);   // 32-bit rows fit up to kMaxVertices
    }
    auto resident = [&](int S) {   // groups an SM holds at a time
        const int groups = (d.n + S - 1) / S;
        return std::max(1, std::min({4, (int)((227 * 1024) / (bytes(S) + sizeof(SsspLists) + 1088)), (groups + d.nsm - 1) / d.nsm}));
    };
    // Sources per group: an SM's groups cost about their arcs once per source, the masks of
    // the arcs' tails twice that once per group, and a round's latency, times the rounds,
    // for every set of groups that run side by side.
    double best = 0;
    for (int k = 1; k <= kSsspMaxSources && bytes(k) <= kSsspSmemMax; ++k) {
        const int groups = (d.n + k - 1) / k, per_sm = (groups + d.nsm - 1) / d.nsm;
        const double cost = per_sm * arcs_about * (k + 2.0) + (per_sm + resident(k) - 1) / resident(k) * 20000.0;
        if (k == 1 || cost < best) {
            best = cost;
            a.S = k;
        }
    }
    // about 1024 threads per SM
    const size_t smem = bytes(a.S);
    auto go = [&](auto lists) {
        constexpr bool L = decltype(lists)::value;
        if (resident(a.S) >= 3) sssp_launch<DT, DS, 256, SsspForm::kGroups, L>(d, a, smem);
        else if (resident(a.S) == 2) sssp_launch<DT, DS, 512, SsspForm::kGroups, L>(d, a, smem);
        else sssp_launch<DT, DS, 1024, SsspForm::kGroups, L>(d, a, smem);
    };
    // Lists for large graphs and for those with about one edge per vertex (k_sssp): they cost a
    // small one some 3 us for their part of the kernel (G(256, 2048) 20.1 us without, 23.4 with;
    // G(1024, 8192) 85.7 and 87.0).
    if (off && (d.n >= kListsMinN || 2 * d.g_arcs <= 5 * (int64_t)d.n)) go(std::true_type{});
    else go(std::false_type{});
}
static_assert((size_t)kMaxVertices * sizeof(uint32_t) + 2 * kMaxVertices / 8 <= kSsspSmemMax, "SsspForm::kOne of 32-bit rows");

// Arcs per vertex from which the light search pays: its own kLight arcs per vertex, twice
// (bc_init_static's device time, complete n = 1024:
// 4.9 ms so, 25 ms over every arc; complete n = 600, int32: 2.4 ms so, 2.9 ms before).
constexpr int kDenseDegree = 4 * kLight;

template <typename DT, typename DS>
static void sssp(const Dev& d, int64_t w_max, bool all_arcs, bool check) {
    if (!all_arcs && d.g_off && d.g_arcs >= (int64_t)kDenseDegree * d.n) {
        // the lists live in the memory of the path counts and the dependency rows, which the
        // accumulation writes only afterwards: each holds n * ld >= arcs entries of 8 bytes
        Arc* f_arc = reinterpret_cast<Arc*>(d.S);
        int64_t* f_w64 = reinterpret_cast<int64_t*>(d.Dl);
        const size_t light = (size_t)2 * kLight * d.n;   // <= arcs / 2
        Arc* l_arc = reinterpret_cast<Arc*>(d.Dl);
        int64_t* l_w64 = reinterpret_cast<int64_t*>(l_arc + light);
        unsigned long long* counts = reinterpret_cast<unsigned long long*>(d.g_count);
        k_light_arcs<<<std::min((d.n + 7) / 8, d.nsm * 8), 256, 0, d.st>>>(d.n, d.g_off, d.g_arc, d.g_w64, w_max, l_arc,
                                                                         l_w64, counts + 1);
        sssp_search<DT, DS>(d, l_arc, l_w64, counts + 1, nullptr, (double)light, false);
        k_filter_arcs<DT><<<(int)std::min<int64_t>((d.g_arcs + 255) / 256, d.nsm * 8), 256, 0, d.st>>>(
            d.ld, d.g_arcs, d.g_arc, d.g_w64, (const DT*)d.D, f_arc, f_w64, counts + 2);
        sssp_search<DT, DS>(d, f_arc, f_w64, counts + 2, nullptr, (double)light, check);
        return;
    }
    sssp_search<DT, DS>(d, d.g_arc, d.g_w64, d.g_count, d.g_off, (double)d.g_arcs, check);
}

// w_max: the largest weight (0: not known).
void launch_sssp(const Dev& d, int64_t w_max, bool all_arcs) {
    const int64_t inf = d.dbytes == 4 ? (int64_t)INT32_MAX : INT64_MAX;
    auto below = [&](int64_t bound) { return w_max > 0 && w_max <= (bound - 1) / std::max(d.n - 1, 1); };
    if (d.dbytes == 4) sssp<int32_t, uint32_t>(d, w_max, all_arcs, !below(inf));
    else if (below(INT32_MAX)) sssp<int64_t, uint32_t>(d, w_max, all_arcs, false);
    else sssp<int64_t, int64_t>(d, w_max, all_arcs, !below(inf));
}

void launch_estar_flags(const Dev& d, uint8_t* flags) {
    if (d.g_arcs <= 0) return;
    const int blocks = (int)((d.g_arcs + 255) / 256);
    if (d.dbytes == 4)
        k_estar_flags<int32_t><<<blocks, 256, 0, d.st>>>(d.ld, d.g_arcs, d.g_arc, d.g_w64, (const int32_t*)d.D, flags);
    else
        k_estar_flags<int64_t><<<blocks, 256, 0, d.st>>>(d.ld, d.g_arcs, d.g_arc, d.g_w64, (const int64_t*)d.D, flags);
}

}  // namespace bcg
