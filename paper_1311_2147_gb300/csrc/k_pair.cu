// k_pair.cu -- dependency rows of an undirected update by pair corrections.
//
// delta_s(x) is the sum over targets t of the pair dependency
// delta_st(x) = sigma_sx * sigma_xt / sigma_st, taken where d(s,x) + d(x,t) = d(s,t) and
// x is neither s nor t (Section 2, the definition that Eq. 4 turns into a recurrence).
// Under a decrease, a pair (s,t) whose distance and path count are both unchanged keeps
// its whole set of shortest paths: no old shortest path uses a changed edge (it would
// now be shorter, so d(s,t) would have dropped), so each one keeps its weight and stays
// shortest, and since sigma_st did not grow no path joined them.  Every delta_st(x) of
// such a pair is unchanged, hence
//     delta'_s(x) = delta_s(x) + sum over changed pairs (s,t) of [delta'_st(x) - delta_st(x)].
// The passes that write D and sigma (the rank-1 passes of Lemma 2 / Lemma 4 and the
// write of row v) record each pair's first change in an update: a bit in the n x n
// change map, the pair's old distance and path count, and t in the target list of row
// s (record_change).  A row with at most kPairCap changed targets is corrected by the
// sum above.  The state before the update is the state after it except at the set
// bits, where the saved values hold, so both terms read the current rows plus a few
// saved values.  In G_D of an undirected graph d(x,t) = d(t,x) and sigma_xt = sigma_tx
// before and after the update, so the column t of the formula is row t, read
// contiguously.  Rows with more targets than the cap are re-accumulated by Algorithm 1.
#include "bc_batch.cuh"
#include "bc_device.cuh"
#include "ff.cuh"

static_assert(bcg::kPairCap <= 1024, "the targets of a row are sorted by one CTA");

namespace bcg {

constexpr int kPairThreads = 256;
constexpr int kPairCtasPerSm = 4;
// targets whose rows are loaded together: one with int32 distances (eight columns per
// thread, whose two loads per target already overlap), two with int64 ones
template <int VN> struct PairGroup { static constexpr int value = VN >= 8 ? 1 : 2; };
constexpr int kPairPieces = 8;  // pieces of equal weight per CTA of the grid

// Per-update records of the rows listed in rows[0..count) back to zero (a pair (s,t)
// changes only in a changed row s), a warp per row: a row with at most tcap changed
// targets has its bits only in the words of its listed targets, a longer one is
// cleared whole.
__device__ __forceinline__ void dev_pair_clear_row(int s, int32_t* tcnt, const int32_t* tlist, int tcap,
                                                   uint32_t* chg, int words) {
    const int lane = threadIdx.x & 31;
    const int T = tcnt[s];
    uint32_t* row = chg + (size_t)s * words;
    if (T <= tcap) {
        for (int j = lane; j < T; j += 32) row[tlist[(size_t)s * tcap + j] >> 5] = 0u;
    } else {
        for (int j = lane; j < words; j += 32) row[j] = 0u;
    }
    __syncwarp();
    if (lane == 0) tcnt[s] = 0;
}

// One changed target t of a row s, as prepared by k_pair_plan: the pair's distance and
// reciprocal path count before and after the update (-1: no path).
struct PairTgt {
    int32_t t;
    int32_t pad;
    int64_t dold;
    int64_t dnew;
    ff rold;
    ff rnew;
};
static_assert(sizeof(PairTgt) == kPairPlanBytes, "the plan is allocated with these bytes per target");

template <typename DT>
struct PairArgs {
    int n;
    int ld;                 // entries of a state row
    const DT* D;            // state after the update
    const uint64_t* S;
    const uint32_t* chg;    // change map: bit (s,x) set where the pair changed
    int words;
    const DT* oD;           // old values where the bit is set
    const uint64_t* oS;
    int32_t* tcnt;          // changed targets per row
    const int32_t* tlist;
    PairTgt* plan;          // [n * tcap]
    int64_t* wpre;          // [n + 1] prefix of the item weights of the listed rows
    int32_t* next_piece;    // pieces of the work handed out so far past the first wave
    const int32_t* prows;   // the rows corrected pair by pair, most targets first
    const int32_t* pcount;
    int tcap;
    const int32_t* rows;
    const int32_t* count;
    int32_t* full_rows;     // rows with more targets than tcap
    int32_t* full_count;
    ff* Dl;
    int64_t* bcfix;         // [3n + 1] BC change of this update (fixed point, see fix_add)
    int32_t* err;
};

// BC(x) += v for one corrected entry delta_s(x) (fix_add): each pair term delta_st(x)
// lies in [0, 1] and a row has at most kPairCap targets, so |v| <= 128, and a column
// receives at most one entry per row.
__device__ __forceinline__ void bc_fix_add(int64_t* fix, int n, int x, ff v) {
    FixWords w = fix_words(v);
    if (fix_small(v)) w.C = fix_rest(v);
    fix_add(fix, n, x, w);
}

// One warp per listed row: a row with more changed targets than the cap goes to the list of
// those re-accumulated in full; one with 1..tcap (most rows have a few): rank
// them (the sums then run in a fixed order) and write the per-target scalars of the
// plan.  Every target of row s has its bit set, so its old values are the saved ones.
constexpr int kPlanThreads = 256;

// (One warp; sv: kPairCap ints of shared memory.)
template <typename DT>
__device__ __forceinline__ void dev_pair_plan_row(const PairArgs<DT>& a, int s, int32_t* sv) {
    const int64_t INF = Inf<DT>::v;
    const int lane = threadIdx.x & 31;
    const int T = a.tcnt[s];
    if (T > a.tcap && lane == 0) a.full_rows[atomicAdd(a.full_count, 1)] = s;
    if (T == 0 || T > a.tcap) return;   // warp-uniform
    for (int j = lane; j < T; j += 32) sv[j] = a.tlist[(size_t)s * a.tcap + j];
    __syncwarp();
    for (int j = lane; j < T; j += 32) {
        const int val = sv[j];
        int pos = 0;
        for (int k = 0; k < T; ++k) pos += sv[k] < val;   // targets are distinct
        const size_t it = (size_t)s * a.ld + val;
        const int64_t dol = a.oD[it], dnw = a.D[it];
        const uint64_t sol = a.oS[it], snw = a.S[it];
        PairTgt p;
        p.t = val;
        p.pad = 0;
        p.dold = (dol == INF || sol == 0) ? -1 : dol;
        p.dnew = (dnw == INF || snw == 0) ? -1 : dnw;
        p.rold = sol ? ff_rcp(ff_from_u64(sol)) : ff{0.f, 0.f};
        p.rnew = snw ? ff_rcp(ff_from_u64(snw)) : ff{0.f, 0.f};
        a.plan[(size_t)s * a.tcap + pos] = p;
    }
    __syncwarp();
}

template <typename DT>
__global__ void __launch_bounds__(kPlanThreads) k_pair_plan(PairArgs<DT> a) {
    pdl_enter();
    __shared__ int32_t s_val[kPlanThreads / 32][kPairCap];
    if (*a.err) return;
    const int cnt = *a.count;
    const int wib = threadIdx.x >> 5;
    const int nw = gridDim.x * (kPlanThreads / 32);
    for (int i = blockIdx.x * (kPlanThreads / 32) + wib; i < cnt; i += nw) dev_pair_plan_row<DT>(a, a.rows[i], s_val[wib]);
}

// sigma_sx * sigma_xt / sigma_st in float-float (the quotient as a product with the
// reciprocal of sigma_st).
__device__ __forceinline__ ff pair_term(uint64_t a, uint64_t b, const ff& rcp) {
    return ff_mul(ff_mul(ff_from_u64(a), ff_from_u64(b)), rcp);
}

// VN consecutive distances in 16-byte loads.
template <typename DT, int VN>
struct DVec {
    DT v[VN];
    __device__ __forceinline__ void load(const DT* p) {
        if constexpr (sizeof(DT) == 4) {
            static_assert(VN == 8, "two 16-byte loads");
            const int4 x = *reinterpret_cast<const int4*>(p);
            const int4 y = *reinterpret_cast<const int4*>(p + 4);
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
            v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
        } else {
            static_assert(VN == 2, "one 16-byte load");
            const longlong2 x = *reinterpret_cast<const longlong2*>(p);
            v[0] = x.x; v[1] = x.y;
        }
    }
};

// Bits of columns x0 .. x0+VN-1 of row r in the change map (x0 is a multiple of VN, so
// they sit in one word).
template <int VN>
__device__ __forceinline__ unsigned chg_bits(const uint32_t* chg, int words, int r, int x0) {
    return (chg[(size_t)r * words + (x0 >> 5)] >> (x0 & 31)) & ((1u << VN) - 1u);
}

// The old values of row r at the columns whose bit is set (one vector load; the saved
// values at the other columns are stale and not used).
template <typename DT, int VN>
__device__ __forceinline__ void patch_old(DVec<DT, VN>& d, unsigned bits, const DT* oD_row, int x0) {
    DVec<DT, VN> o;
    o.load(oD_row + x0);
#pragma unroll
    for (int q = 0; q < VN; ++q)
        if ((bits >> q) & 1u) d.v[q] = o.v[q];
}

template <typename DT> struct Unsigned;
template <> struct Unsigned<int32_t> { using T = uint32_t; };
template <> struct Unsigned<int64_t> { using T = uint64_t; };

// Bit q set where column x0+q lies on a shortest s-t path of one state:
// d(s,x) + d(x,t) = d(s,t) and d(x,t) > 0 (x != t; x != s is ensured by the caller,
// which replaces d(s,s) by INF).  Distances are below INF = DT max, so their unsigned
// sum never wraps, and a sum with an INF term exceeds every finite d(s,t); "no path"
// is passed as all ones, which no sum equals.
template <typename DT, int VN>
__device__ __forceinline__ unsigned on_path(const DVec<DT, VN>& ds, const DVec<DT, VN>& dt,
                                            typename Unsigned<DT>::T dst) {
    using U = typename Unsigned<DT>::T;
    unsigned m = 0;
#pragma unroll
    for (int q = 0; q < VN; ++q)
        m |= (((U)ds.v[q] + (U)dt.v[q] == (U)dst) && dt.v[q] != 0) ? (1u << q) : 0u;
    return m;
}

// Per-target scalars of the row being processed, as staged in shared memory: what
// every column test reads (row t of D and of the change map, and the distances, with
// -1 for "no path": in unsigned arithmetic no sum of two distances equals it) and
// what only a matched column reads.
template <typename DT>
struct TgtFast {
    const DT* Dt;
    const uint32_t* Ct;
    DT dold, dnew;
};
struct TgtSlow {
    int64_t rt;      // t * ld
    ff rold, rnew;
};


// Weight of one work item of a listed row: its targets plus one (the row's own loads),
// or 0 when the row takes the full path or has nothing to correct.
__device__ __forceinline__ int64_t item_weight(int T, int tcap) { return (T == 0 || T > tcap) ? 0 : T + 1; }

// prows[0..*pcount) = the listed rows with 1..tcap targets, most targets first;
// wpre[i] = total weight of the items of rows prows[0..i-1] (nchunks items per row).
// One CTA: a counting sort (the lanes of a warp with the same target count add to its
// bucket with one shared-memory atomic), then each warp scans a contiguous run of the
// sorted rows and one block scan joins the runs.
// Also adds the rows with a correction and their targets to stats[8], stats[9].
// Listed rows the weights pass stages in shared memory (up to n; none past the limit).
constexpr int kWeightsStageMax = 20480;   // 160 KB of row ids and counts
static int weights_stage(int n) { return n <= kWeightsStageMax ? n : 0; }

struct PairWeightsSmem {
    int64_t wsum[32];
    int64_t s_total;
    int64_t s_rows[32], s_tgts[32];
    int s_hist[kPairCap + 1];
};

// (CTA-wide, 1024 threads.)  s_r and s_T: scap ints each of shared memory; when the
// listed rows fit, they and their target counts are staged there first, every load
// issued before any is used (the passes below would otherwise wait on a row id and then
// on its count, tile after tile).  The sorted rows' counts are staged in wpre, which
// the last pass overwrites with the prefix.
__device__ __forceinline__ void dev_pair_weights(const int32_t* rows, const int32_t* count, const int32_t* tcnt,
                                                 int tcap, int nchunks, int32_t* prows, int32_t* pcount,
                                                 int64_t* wpre, int64_t* stats, PairWeightsSmem& sm,
                                                 int32_t* s_r, int32_t* s_T, int scap) {
    int64_t* wsum = sm.wsum;
    int64_t& s_total = sm.s_total;
    int64_t* s_rows = sm.s_rows;
    int64_t* s_tgts = sm.s_tgts;
    int* s_hist = sm.s_hist;
    const int cnt_all = *count;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nw = blockDim.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    // the rows with 1..tcap targets, most targets first (a counting sort): the heaviest
    // items are handed out first and the light ones fill the end of the kernel.  The
    // order inside a bucket follows the atomics; a row's result does not depend on it.
    for (int b = tid; b <= kPairCap; b += blockDim.x) s_hist[b] = 0;
    const bool staged = cnt_all <= scap;
    if (staged) {
        for (int i = tid; i < cnt_all; i += blockDim.x) s_r[i] = rows[i];
        __syncthreads();
        for (int i = tid; i < cnt_all; i += blockDim.x) s_T[i] = tcnt[s_r[i]];
    }
    __syncthreads();
    for (int i0 = 0; i0 < cnt_all; i0 += blockDim.x) {   // warp-uniform bounds (the match)
        const int i = i0 + tid;
        const int T = i < cnt_all ? (staged ? s_T[i] : tcnt[rows[i]]) : 0;
        const bool ok = T > 0 && T <= tcap;
        const unsigned peers = __match_any_sync(0xffffffffu, ok ? T : -1);
        if (ok && lane == __ffs(peers) - 1) atomicAdd(&s_hist[T], __popc(peers));
    }
    __syncthreads();
    if (tid == 0) {
        int acc = 0;
        for (int b = kPairCap; b >= 1; --b) {
            const int h = s_hist[b];
            s_hist[b] = acc;
            acc += h;
        }
        s_hist[0] = acc;
        *pcount = acc;
    }
    __syncthreads();
    const int cnt = s_hist[0];
    for (int i0 = 0; i0 < cnt_all; i0 += blockDim.x) {
        const int i = i0 + tid;
        const int r = i < cnt_all ? (staged ? s_r[i] : rows[i]) : 0;
        const int T = i < cnt_all ? (staged ? s_T[i] : tcnt[r]) : 0;
        const bool ok = T > 0 && T <= tcap;
        const unsigned peers = __match_any_sync(0xffffffffu, ok ? T : -1);
        const int leader = __ffs(peers) - 1;
        int p0 = 0;
        if (ok && lane == leader) p0 = atomicAdd(&s_hist[T], __popc(peers));
        p0 = __shfl_sync(0xffffffffu, p0, leader);
        if (ok) {
            const int pos = p0 + __popc(peers & below);
            prows[pos] = r;
            wpre[pos] = T;
        }
    }
    __syncthreads();
    int64_t my_rows = 0, my_tgts = 0;
    // a contiguous run of the sorted rows per warp, 32 rows per step
    const int per = (cnt + nw - 1) / nw;
    const int w0 = min(cnt, wid * per), w1 = min(cnt, w0 + per);
    auto warp_incl = [&](int64_t x) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        return x;
    };
    int64_t run = 0;
    for (int b0 = w0; b0 < w1; b0 += 32) {
        const int i = b0 + lane;
        const int64_t iw = i < w1 ? item_weight((int)wpre[i], tcap) : 0;
        if (iw) {
            ++my_rows;
            my_tgts += iw - 1;
        }
        run += __shfl_sync(0xffffffffu, warp_incl(iw * nchunks), 31);
    }
    if (lane == 0) wsum[wid] = run;
    __syncthreads();
    if (wid == 0) {
        const int64_t x = lane < nw ? wsum[lane] : 0;
        const int64_t winc = warp_incl(x);
        if (lane < nw) wsum[lane] = winc - x;
        if (lane == 31) s_total = winc;
    }
    __syncthreads();
    run = wsum[wid];
    for (int b0 = w0; b0 < w1; b0 += 32) {
        const int i = b0 + lane;
        const int64_t x = i < w1 ? item_weight((int)wpre[i], tcap) * nchunks : 0;
        const int64_t incl = warp_incl(x);
        if (i < w1) wpre[i] = run + incl - x;
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    const int64_t base = s_total;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        my_rows += __shfl_xor_sync(0xffffffffu, my_rows, o);
        my_tgts += __shfl_xor_sync(0xffffffffu, my_tgts, o);
    }
    if (lane == 0) {
        s_rows[wid] = my_rows;
        s_tgts[wid] = my_tgts;
    }
    __syncthreads();
    if (tid == 0) {
        int64_t r = 0, t = 0;
        for (int k = 0; k < nw; ++k) {
            r += s_rows[k];
            t += s_tgts[k];
        }
        wpre[cnt] = base;
        stats[8] += r;
        stats[9] += t;
    }
}

__global__ void __launch_bounds__(1024) k_pair_weights(const int32_t* rows, const int32_t* count,
                                                       const int32_t* tcnt, int tcap, int nchunks,
                                                       int32_t* prows, int32_t* pcount,
                                                       int64_t* wpre, int64_t* stats, const int32_t* err,
                                                       int scap) {
    pdl_enter();
    __shared__ PairWeightsSmem sm;
    extern __shared__ int32_t s_stage[];   // 2 * scap ints
    if (*err) return;
    dev_pair_weights(rows, count, tcnt, tcap, nchunks, prows, pcount, wpre, stats,
                     sm, s_stage, s_stage + scap, scap);
}

// Queue of one warp's matches: entry = lane (5 bits) | q (3) | target index u (7) |
// new state (1) | old d/sigma of s saved (1) | old d/sigma of t saved (1); the terms are
// evaluated by all lanes together and summed by the owning lane in queue order.
constexpr int kPairQueue = 64;
struct PairQueue {
    uint32_t e[kPairQueue];
    ff term[kPairQueue];
};

// One work item: the VN columns x0 .. x0+VN-1 of this thread in row s, whose U_
// targets are staged in s_fa / s_sl.  Targets go in groups of kPairGroup: the group's
// rows are loaded together (one memory round trip), then tested with one add and
// compare per column and state.  The matches (columns on a shortest s-t path of either
// state) are appended to the warp's queue in target order, old state first; when the
// queue is full and at the end of the item, the warp evaluates all queued terms at once
// (one match per lane, its two path counts loaded together with the others) and each
// lane adds its own terms to its column sums in queue order.  A column's sum thus runs
// in target order whatever the lanes' loads are -- one column on the paths to every
// target (a hub) no longer serialises its lane -- and does not depend on how the work
// is shared out.
template <typename DT, int VN>
__device__ __forceinline__ void pair_item(const PairArgs<DT>& a, int s, int U_, int x0, const TgtFast<DT>* s_fa,
                                          const TgtSlow* s_sl, ff (*s_acc)[kPairThreads], PairQueue& wq) {
    constexpr int kPairGroup = PairGroup<VN>::value;
    static_assert(2 * VN * kPairGroup <= 32 && VN <= 8, "a group's matches fit one 32-bit mask");
    using U = typename Unsigned<DT>::T;
    constexpr unsigned kMask = (1u << VN) - 1u;
    const int lane = threadIdx.x & 31;
    const size_t rs = (size_t)s * a.ld;
    const bool active = x0 < a.n;   // the warp runs the item together (the queue needs every lane)
    DVec<DT, VN> dsn, dso;
    unsigned bs = 0;
    if (active) {
        dsn.load(a.D + rs + x0);
        bs = chg_bits<VN>(a.chg, a.words, s, x0);
        dso = dsn;
        if (bs) patch_old<DT, VN>(dso, bs, a.oD + rs, x0);
        if (s >= x0 && s < x0 + VN) {
#pragma unroll
            for (int q = 0; q < VN; ++q)
                if (x0 + q == s) dso.v[q] = dsn.v[q] = (DT)Inf<DT>::v;
        }
    }
    unsigned any = 0;   // bit q: s_acc[q][tid] holds the sum of column x0 + q
    int qlen = 0;       // warp-uniform
    const int lane_x0 = x0 - lane * VN;   // column of lane 0's first vector
    // evaluate the queued terms (all lanes), then add each lane's terms in queue order
    auto flush = [&]() {
        __syncwarp();
        for (int e = lane; e < qlen; e += 32) {
            const uint32_t en = wq.e[e];
            const int L = en & 31, q = (en >> 5) & 7, u = (en >> 8) & 127;
            const bool is_new = (en >> 15) & 1u;
            const int x = lane_x0 + L * VN + q;
            const TgtSlow& sl = s_sl[u];
            const size_t rt = (size_t)sl.rt;
            const uint64_t ssx = (!is_new && ((en >> 16) & 1u)) ? a.oS[rs + x] : a.S[rs + x];
            const uint64_t stx = (!is_new && ((en >> 17) & 1u)) ? a.oS[rt + x] : a.S[rt + x];
            ff t = pair_term(ssx, stx, is_new ? sl.rnew : sl.rold);
            if (!is_new) t = ff{-t.hi, -t.lo};
            wq.term[e] = t;
        }
        __syncwarp();
        for (int e = 0; e < qlen; ++e) {
            const uint32_t en = wq.e[e];
            if ((int)(en & 31) == lane) {
                const int q = (en >> 5) & 7;
                const ff prev = ((any >> q) & 1u) ? s_acc[q][threadIdx.x] : ff{0.f, 0.f};
                s_acc[q][threadIdx.x] = ff_add(prev, wq.term[e]);
                any |= 1u << q;
            }
        }
        __syncwarp();
        qlen = 0;
    };
    const int wofs = x0 >> 5, bsh = x0 & 31;
    for (int u0 = 0; u0 < U_; u0 += kPairGroup) {
        DVec<DT, VN> dtg[kPairGroup];
        unsigned btg[kPairGroup];
        if (active) {
#pragma unroll
            for (int k = 0; k < kPairGroup; ++k)
                if (u0 + k < U_) {
                    const TgtFast<DT> f = s_fa[u0 + k];
                    dtg[k].load(f.Dt + x0);
                    btg[k] = f.Ct[wofs];
                }
        }
        uint32_t mm = 0, btp = 0;
#pragma unroll
        for (int k = 0; k < kPairGroup; ++k) {
            if (!active || u0 + k >= U_) break;
            const TgtFast<DT> f = s_fa[u0 + k];
            const DVec<DT, VN>& dtn = dtg[k];
            const unsigned bt = (btg[k] >> bsh) & kMask;
            DVec<DT, VN> dto = dtn;
            bool hit = false;
            if (!(bs | bt)) {
                // no saved values at these columns: the old and new sums are the same
#pragma unroll
                for (int q = 0; q < VN; ++q) {
                    const U sum = (U)dsn.v[q] + (U)dtn.v[q];
                    hit |= (sum == (U)f.dold) | (sum == (U)f.dnew);
                }
            } else {
                if (bt) patch_old<DT, VN>(dto, bt, a.oD + (f.Dt - a.D), x0);
#pragma unroll
                for (int q = 0; q < VN; ++q) {
                    hit |= (U)dso.v[q] + (U)dto.v[q] == (U)f.dold;
                    hit |= (U)dsn.v[q] + (U)dtn.v[q] == (U)f.dnew;
                }
            }
            if (!hit) continue;
            const unsigned mo = on_path<DT, VN>(dso, dto, (U)f.dold);
            const unsigned mn = on_path<DT, VN>(dsn, dtn, (U)f.dnew);
            mm |= (mo | (mn << VN)) << (2 * VN * k);
            btp |= bt << (VN * k);
        }
        // append this group's matches, each lane's in (target, state, q) order; a group
        // that does not fit goes in parts, with a flush in between
        while (__any_sync(0xffffffffu, mm != 0)) {
            if (qlen == kPairQueue) flush();
            const int cnt = __popc(mm);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int tot = __shfl_sync(0xffffffffu, incl, 31);
            const int space = kPairQueue - qlen;
            for (int pos = incl - cnt; mm && pos < space; ++pos) {
                const int b = __ffs(mm) - 1;
                mm &= mm - 1;
                const int k = b / (2 * VN), j = b - k * 2 * VN;
                const unsigned is_new = j >= VN ? 1u : 0u;
                const int q = is_new ? j - VN : j;
                wq.e[qlen + pos] = (uint32_t)lane | ((uint32_t)q << 5) | ((uint32_t)(u0 + k) << 8) | (is_new << 15) |
                                   (((bs >> q) & 1u) << 16) | (((btp >> (VN * k + q)) & 1u) << 17);
            }
            qlen += min(tot, space);
            __syncwarp();
        }
    }
    if (qlen) flush();
#pragma unroll
    for (int q = 0; q < VN; ++q)
        if ((any >> q) & 1u) {
            const ff acc = s_acc[q][threadIdx.x];
            ff* p = a.Dl + rs + x0 + q;
            *p = ff_add(*p, acc);
            bc_fix_add(a.bcfix, a.n, x0 + q, acc);
        }
}

// Work item = (listed row s, chunk of CW = threads x VN columns), in row-major order;
// an item weighs the row's targets plus one.  The items are cut into kPairPieces x grid
// pieces of equal weight (a piece runs the items whose start falls in it, so rows with
// many targets spread over several pieces).  The first wave of CTAs takes the first
// pieces and every CTA that finishes one takes the next from a counter: item costs
// vary more than their weights (the matches, the per-item loads), and a static share
// per CTA left half of the SMs idle for half of the kernel.  The plan of a row is
// staged in shared memory when the CTA meets the row.
template <typename DT, int VN>
__global__ void __launch_bounds__(kPairThreads, kPairCtasPerSm) k_pairdep(PairArgs<DT> a) {
    pdl_enter();
    __shared__ TgtFast<DT> s_fa[kPairCap];
    __shared__ TgtSlow s_sl[kPairCap];
    __shared__ ff s_acc[VN][kPairThreads];   // per thread: the sums of its VN columns
    __shared__ PairQueue s_wq[kPairThreads / 32];
    __shared__ int s_i, s_c, s_p;
    if (*a.err) return;
    constexpr int CW = kPairThreads * VN;
    const int n = a.n;
    const int nchunks = (n + CW - 1) / CW;
    const int cnt = *a.pcount;
    const int64_t W = a.wpre[cnt];
    const int npieces = gridDim.x * kPairPieces;
    int cur = -1, s = -1, U_ = 0;   // the row whose plan is staged
    for (int piece = blockIdx.x; piece < npieces;) {
        const int64_t lo = W * piece / npieces, hi = W * (piece + 1) / npieces;
        if (lo < hi) {   // block-uniform
            if (threadIdx.x == 0) {
                // last row whose items start at or before lo: wpre[L] <= lo < wpre[R]
                int L = 0, R = cnt;
                while (R - L > 1) {
                    const int m = (L + R) >> 1;
                    if (a.wpre[m] <= lo) L = m; else R = m;
                }
                const int64_t wc = (a.wpre[L + 1] - a.wpre[L]) / nchunks;   // > 0: lo lies in row L
                s_i = L;
                s_c = (int)((lo - a.wpre[L] + wc - 1) / wc);
            }
            __syncthreads();
            int i = s_i, c = s_c;
            int64_t wc = (a.wpre[i + 1] - a.wpre[i]) / nchunks;
            for (;;) {
                if (c >= nchunks) {   // next row with items (block-uniform)
                    do {
                        ++i;
                    } while (i < cnt && a.wpre[i + 1] == a.wpre[i]);
                    if (i >= cnt) break;
                    wc = (a.wpre[i + 1] - a.wpre[i]) / nchunks;
                    c = 0;
                }
                if (a.wpre[i] + (int64_t)c * wc >= hi) break;
                if (i != cur) {
                    cur = i;
                    s = a.prows[i];
                    U_ = (int)wc - 1;
                    __syncthreads();   // the previous row's plan is no longer read
                    if (threadIdx.x < U_) {
                        const PairTgt p = a.plan[(size_t)s * a.tcap + threadIdx.x];
                        const size_t rt = (size_t)p.t * a.ld;
                        s_fa[threadIdx.x] =
                            TgtFast<DT>{a.D + rt, a.chg + (size_t)p.t * a.words, (DT)p.dold, (DT)p.dnew};
                        s_sl[threadIdx.x] = TgtSlow{(int64_t)rt, p.rold, p.rnew};
                    }
                    __syncthreads();
                }
                const int x0 = c * CW + threadIdx.x * VN;
                ++c;
                // a warp with at least one column in the row runs the item (all its lanes)
                if (x0 - (int)(threadIdx.x & 31) * VN < n)
                    pair_item<DT, VN>(a, s, U_, x0, s_fa, s_sl, s_acc, s_wq[threadIdx.x >> 5]);
            }
        }
        // the next piece: the first wave takes pieces 0 .. grid-1, later ones go in
        // order to the CTAs that finish first
        if (threadIdx.x == 0) s_p = gridDim.x + atomicAdd(a.next_piece, 1);
        __syncthreads();
        piece = s_p;
        __syncthreads();   // s_p is read by all before thread 0 writes it again
    }
}

// BC (hi, lo) += the fixed-point change of each column, then its words are zeroed for the
// next update: B's high bits are carried into A, so that A * 2^-24 and B * 2^-71 are exact
// doubles, the first added with TwoSum.  third: some column has a C.
__device__ __forceinline__ void dev_bc_fix(int t, int n, int64_t* fix, bool third, double* hi, double* lo) {
    const longlong2 f = *reinterpret_cast<const longlong2*>(fix + 2 * (size_t)t);
    FixWords w{f.x, f.y, 0};
    if (third) w.C = fix[2 * (size_t)n + t];
    if ((w.A | w.B | w.C) == 0) return;
    *reinterpret_cast<longlong2*>(fix + 2 * (size_t)t) = make_longlong2(0, 0);
    if (third) fix[2 * (size_t)n + t] = 0;
    fix_carry(w);
    const double x1 = (double)w.A * 0x1p-24;
    const double x2 = (double)w.B * 0x1p-71 + (double)w.C * 0x1p-112;
    const double h = hi[t];
    const double s = h + x1;
    const double bp = s - h;
    const double e = (h - (s - bp)) + (x1 - bp);
    hi[t] = s;
    lo[t] += e + x2;
}

// Counters of a finished update, from its lists: [0] rows changed [1] updates without any
// [2] most rows [3] updates [7] rows re-accumulated in full among those with corrections.
__device__ __forceinline__ void dev_update_stats(int64_t* stats, int changed, int full) {
    stats[0] += changed;
    if (changed == 0) stats[1] += 1;
    if (changed > stats[2]) stats[2] = changed;
    stats[3] += 1;
    stats[7] += full;
}

// The last kernel of an update: BC takes its change, the changed rows' flags and records go
// back to zero, and the CTA that finishes last adds the counters and zeroes the lists'
// counts for the next update.
struct EndArgs {
    int n;
    int64_t* fix;
    double* hi;
    double* lo;
    const int32_t* rows;
    int32_t* counts;
    uint32_t* changed;
    int32_t* tcnt;       // NULL: no records
    const int32_t* tlist;
    int tcap;
    uint32_t* chg;
    int words;
    int64_t* stats;
    const int32_t* err;
};
__global__ void __launch_bounds__(256) k_update_end(EndArgs a) {
    pdl_enter();
    if (*a.err) return;   // the handle is poisoned: no further update
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const bool third = a.fix[3 * (size_t)a.n] != 0;
    for (int x = t; x < a.n; x += gridDim.x * blockDim.x) dev_bc_fix(x, a.n, a.fix, third, a.hi, a.lo);
    const int cnt = a.counts[1];
    for (int i = t; i < cnt; i += gridDim.x * blockDim.x) a.changed[a.rows[i]] = 0u;
    if (a.tcnt)
        for (int i = t >> 5; i < cnt; i += (gridDim.x * blockDim.x) >> 5)
            dev_pair_clear_row(a.rows[i], a.tcnt, a.tlist, a.tcap, a.chg, a.words);
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(a.counts + 6, 1) == (int)gridDim.x - 1) {
        dev_update_stats(a.stats, cnt, a.counts[3]);
        for (int k = 0; k < 16; ++k) a.counts[k] = 0;
        if (third) a.fix[3 * (size_t)a.n] = 0;
    }
}

// ------------------------------------------------------------------ launches

PairRec pair_rec(const Dev& d) { return make_pair_rec(d); }

void launch_update_end(const Dev& d) {
    EndArgs a{d.n, d.bcfix, d.bc_hi, d.bc_lo, d.acc_rows, d.counts, d.changed, d.pair_on ? d.tcnt : nullptr, d.tlist,
              d.tcap, d.chg, d.chg_words, d.stats, d.err};
    launch_k(k_update_end, std::min(d.nsm * 4, std::max(1, (d.n + 31) / 32)), 256, 0, d.st, a);
}

template <typename DT>
__host__ __device__ inline PairArgs<DT> pair_args(const Dev& d) {
    PairArgs<DT> a;
    a.n = d.n;
    a.ld = d.ld;
    a.D = (const DT*)d.D;
    a.S = d.S;
    a.chg = d.chg;
    a.words = d.chg_words;
    a.oD = (const DT*)d.oldD;
    a.oS = d.oldS;
    a.tcnt = d.tcnt;
    a.tlist = d.tlist;
    a.plan = reinterpret_cast<PairTgt*>(d.plan);
    a.wpre = d.pair_w;
    a.next_piece = d.counts + 4;
    a.prows = d.pair_rows;
    a.pcount = d.counts + 5;
    a.tcap = d.tcap;
    a.rows = d.acc_rows;
    a.count = d.counts + 1;
    a.full_rows = d.full_rows;
    a.full_count = d.counts + 3;
    a.Dl = d.Dl;
    a.bcfix = d.bcfix;
    a.err = d.err;
    return a;
}

// ------------------------------------------------------------------ batches
//
// The pair corrections of round r of a batch, for every graph that has them (the rest of
// the round is in k_batch.cu).  Each kernel runs the single-graph kernel's device
// function on the concatenated work of all graphs, a task mapped to its graph by binary
// search over prefix offsets, so a graph's result in a batch is bit-identical to its
// result alone.  Graphs whose update walks are k_walk.cu's.

__device__ __forceinline__ bool batch_pair_graph(const BatchArgs& b, int r, int g) {
    const Dev& d = b.devs[g];
    return d.pair_on && b.upd[(int64_t)r * b.G + g].present && *d.err == 0 && !batch_walks_graph(b, r, g);
}

// A warp per listed row of every graph (k_pair_plan); plan_pr offsets the rows.
template <typename DT>
__global__ void __launch_bounds__(kPlanThreads) kb_pair_plan(BatchArgs b, int r) {
    __shared__ int32_t s_val[kPlanThreads / 32][kPairCap];
    const int G = b.G;
    const int64_t total = b.plan_pr[G];
    const int wib = threadIdx.x >> 5;
    const int64_t nw = (int64_t)gridDim.x * (kPlanThreads / 32);
    for (int64_t j = (int64_t)blockIdx.x * (kPlanThreads / 32) + wib; j < total; j += nw) {
        const int g = graph_of(b.plan_pr, G, j);
        const Dev& d = b.devs[g];
        if (!d.pair_on || batch_walks_graph(b, r, g)) continue;
        const PairArgs<DT> a = pair_args<DT>(d);
        dev_pair_plan_row<DT>(a, d.acc_rows[j - b.plan_pr[g]], s_val[wib]);
    }
}

// One CTA per graph in turn: rows most targets first and their weight prefix
// (k_pair_weights).
__global__ void __launch_bounds__(1024) kb_pair_weights(BatchArgs b, int r, int scap) {
    __shared__ PairWeightsSmem sm;
    extern __shared__ int32_t s_stage[];   // 2 * scap ints
    for (int g = blockIdx.x; g < b.G; g += gridDim.x) {
        if (!batch_pair_graph(b, r, g)) continue;   // block-uniform
        const Dev& d = b.devs[g];
        const int cw = kPairThreads * pair_vn(d.dbytes);
        const int nchunks = (d.n + cw - 1) / cw;
        dev_pair_weights(d.acc_rows, d.counts + 1, d.tcnt, d.tcap, nchunks, d.pair_rows, d.counts + 5, d.pair_w,
                         d.stats, sm, s_stage, s_stage + scap, scap);
        __syncthreads();
    }
}

// The column test (k_pairdep) over every graph with corrections: their weight lines laid
// end to end (plan_pw), cut into kPairPieces x grid pieces of equal weight; a piece runs
// the items whose start falls in it, across row and graph boundaries, and later pieces go
// to the CTAs that finish first (counter pctr).
template <typename DT, int VN>
__global__ void __launch_bounds__(kPairThreads, kPairCtasPerSm) kb_pairdep(BatchArgs b) {
    __shared__ TgtFast<DT> s_fa[kPairCap];
    __shared__ TgtSlow s_sl[kPairCap];
    __shared__ ff s_acc[VN][kPairThreads];
    __shared__ PairQueue s_wq[kPairThreads / 32];
    __shared__ int s_g, s_i, s_c, s_p;
    constexpr int CW = kPairThreads * VN;
    const int G = b.G;
    const int64_t* off = b.plan_pw;
    const int64_t W = off[G];
    const int npieces = gridDim.x * kPairPieces;
    int cg = -1;                     // the graph whose arguments are loaded
    int sg = -1, cur = -1, s = -1;   // the graph and row whose plan is staged
    int U_ = 0, nchunks = 1, cnt = 0;
    PairArgs<DT> a{};
    for (int piece = blockIdx.x; piece < npieces;) {
        const int64_t lo = W * piece / npieces, hi = W * (piece + 1) / npieces;
        if (lo < hi) {   // block-uniform
            if (threadIdx.x == 0) {
                // the graph holding lo (off[g] <= lo < off[g + 1]), then its last row whose
                // items start at or before lo
                const int g = graph_of(off, G, lo);
                const Dev& d = b.devs[g];
                const int nch = (d.n + CW - 1) / CW;
                const int64_t l = lo - off[g];
                int L = 0, R = d.counts[5];
                while (R - L > 1) {
                    const int m = (L + R) >> 1;
                    if (d.pair_w[m] <= l) L = m; else R = m;
                }
                const int64_t wc = (d.pair_w[L + 1] - d.pair_w[L]) / nch;   // > 0: l lies in row L
                s_g = g;
                s_i = L;
                s_c = (int)((l - d.pair_w[L] + wc - 1) / wc);
            }
            __syncthreads();
            int g = s_g, i = s_i, c = s_c;
            if (g != cg) {
                cg = g;
                a = pair_args<DT>(b.devs[g]);
                nchunks = (a.n + CW - 1) / CW;
                cnt = *a.pcount;
            }
            int64_t wc = (a.wpre[i + 1] - a.wpre[i]) / nchunks;
            for (;;) {
                if (c >= nchunks) {   // next row with items, in this graph or the next ones (block-uniform)
                    do {
                        ++i;
                    } while (i < cnt && a.wpre[i + 1] == a.wpre[i]);
                    while (i >= cnt) {
                        do {
                            ++g;
                        } while (g < G && off[g + 1] == off[g]);
                        if (g >= G) break;
                        cg = g;
                        a = pair_args<DT>(b.devs[g]);
                        nchunks = (a.n + CW - 1) / CW;
                        cnt = *a.pcount;
                        i = 0;
                        while (i < cnt && a.wpre[i + 1] == a.wpre[i]) ++i;
                    }
                    if (g >= G) break;
                    wc = (a.wpre[i + 1] - a.wpre[i]) / nchunks;
                    c = 0;
                }
                if (off[g] + a.wpre[i] + (int64_t)c * wc >= hi) break;
                if (i != cur || g != sg) {
                    cur = i;
                    sg = g;
                    s = a.prows[i];
                    U_ = (int)wc - 1;
                    __syncthreads();   // the previous row's plan is no longer read
                    if (threadIdx.x < U_) {
                        const PairTgt p = a.plan[(size_t)s * a.tcap + threadIdx.x];
                        const size_t rt = (size_t)p.t * a.ld;
                        s_fa[threadIdx.x] =
                            TgtFast<DT>{a.D + rt, a.chg + (size_t)p.t * a.words, (DT)p.dold, (DT)p.dnew};
                        s_sl[threadIdx.x] = TgtSlow{(int64_t)rt, p.rold, p.rnew};
                    }
                    __syncthreads();
                }
                const int x0 = c * CW + threadIdx.x * VN;
                ++c;
                if (x0 - (int)(threadIdx.x & 31) * VN < a.n)
                    pair_item<DT, VN>(a, s, U_, x0, s_fa, s_sl, s_acc, s_wq[threadIdx.x >> 5]);
            }
        }
        if (threadIdx.x == 0) s_p = gridDim.x + atomicAdd(b.pctr, 1);
        __syncthreads();
        piece = s_p;
        __syncthreads();
    }
}

// The end of a round (k_update_end): BC takes its change in every graph with an update, the
// changed rows' flags and records go back to zero (a warp per listed row); then, a thread
// per graph, the counters and the lists' counts.
__global__ void kb_update_end(BatchArgs b, int r) {
    const int G = b.G;
    const int64_t total = b.coff[G];
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < total;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int g = graph_of(b.coff, G, j);
        const Dev& d = b.devs[g];
        if (*d.err || b.upd[(int64_t)r * G + g].present == 0) continue;
        dev_bc_fix((int)(j - b.coff[g]), d.n, d.bcfix, d.bcfix[3 * (size_t)d.n] != 0, d.bc_hi, d.bc_lo);
    }
    const int64_t rows = b.plan_pr[G];
    const int wpb = blockDim.x >> 5;
    for (int64_t j = (int64_t)blockIdx.x * wpb + (threadIdx.x >> 5); j < rows; j += (int64_t)gridDim.x * wpb) {
        const int g = graph_of(b.plan_pr, G, j);
        const Dev& d = b.devs[g];
        const int s = d.acc_rows[j - b.plan_pr[g]];
        if ((threadIdx.x & 31) == 0) d.changed[s] = 0u;
        if (d.pair_on) dev_pair_clear_row(s, d.tcnt, d.tlist, d.tcap, d.chg, d.chg_words);
    }
}
__global__ void kb_update_stats(BatchArgs b, int r) {
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < b.G; g += gridDim.x * blockDim.x) {
        const Dev& d = b.devs[g];
        if (*d.err || b.upd[(int64_t)r * b.G + g].present == 0) continue;
        dev_update_stats(d.stats, d.counts[1], d.counts[3]);
        for (int k = 0; k < 8; ++k) d.counts[k] = 0;
        d.bcfix[3 * (size_t)d.n] = 0;
    }
}

void batch_pair_plan(const BatchArgs& b, const BatchLaunch& L, int r, int dbytes, cudaStream_t st) {
    if (dbytes == 4) kb_pair_plan<int32_t><<<L.nsm * 8, kPlanThreads, 0, st>>>(b, r);
    else kb_pair_plan<int64_t><<<L.nsm * 8, kPlanThreads, 0, st>>>(b, r);
}

void batch_round_end(const BatchArgs& b, const BatchLaunch& L, int r, cudaStream_t st) {
    kb_update_end<<<L.nsm * 4, 256, 0, st>>>(b, r);
    kb_update_stats<<<std::max(1, (b.G + 255) / 256), 256, 0, st>>>(b, r);
}

template <typename DT>
static void batch_pairs(const BatchArgs& b, const BatchLaunch& L, int r, cudaStream_t st) {
    const int G = b.G, nsm = L.nsm;
    const int scap = weights_stage(b.n_max);
    kb_pair_weights<<<std::min(G, nsm * 2), 1024, 2 * sizeof(int32_t) * (size_t)scap, st>>>(b, r, scap);
    const int pgrid = nsm * kPairCtasPerSm;
    batch_plan(b, r, 4, 2, b.plan_pw, L.scan_unroll, st);
    kb_pairdep<DT, pair_vn(sizeof(DT))><<<pgrid, kPairThreads, 0, st>>>(b);
}

void batch_pair_launches(const BatchArgs& b, const BatchLaunch& L, int r, int dbytes, cudaStream_t st) {
    if (dbytes == 4) batch_pairs<int32_t>(b, L, r, st);
    else batch_pairs<int64_t>(b, L, r, st);
}

cudaError_t pair_setup() {
    const int wmax = 2 * (int)sizeof(int32_t) * kWeightsStageMax;
    cudaError_t e = cudaFuncSetAttribute(k_pair_weights, cudaFuncAttributeMaxDynamicSharedMemorySize, wmax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kb_pair_weights, cudaFuncAttributeMaxDynamicSharedMemorySize, wmax);
    return e;
}

void launch_pair_plan(const Dev& d) {
    const int pgrid = d.nsm * 8;
    if (d.dbytes == 4) launch_k(k_pair_plan<int32_t>, pgrid, kPlanThreads, 0, d.st, pair_args<int32_t>(d));
    else launch_k(k_pair_plan<int64_t>, pgrid, kPlanThreads, 0, d.st, pair_args<int64_t>(d));
}

void launch_pairdep(const Dev& d) {
    const int vn = pair_vn(d.dbytes);
    const int cw = kPairThreads * vn;
    const int nchunks = (d.n + cw - 1) / cw;
    const int scap = weights_stage(d.n);
    launch_k(k_pair_weights, 1, 1024, 2 * sizeof(int32_t) * (size_t)scap, d.st, d.acc_rows, d.counts + 1, d.tcnt,
             d.tcap, nchunks, d.pair_rows, d.counts + 5, d.pair_w, d.stats, d.err, scap);
    const int grid = d.nsm * kPairCtasPerSm;   // one resident wave; later pieces go to the first free CTA
    if (d.dbytes == 4) launch_k(k_pairdep<int32_t, 8>, grid, kPairThreads, 0, d.st, pair_args<int32_t>(d));
    else launch_k(k_pairdep<int64_t, 2>, grid, kPairThreads, 0, d.st, pair_args<int64_t>(d));
}

}  // namespace bcg
