// bc_device.cuh -- device functions shared by the single-graph kernels and the batched
// (many graphs per launch) kernels, so that both run the same arithmetic and give
// bit-identical results.  What each function computes is described at its definition;
// the translation units that launch them describe the method (k_update.cu: the
// all-pairs passes; k_accum.cu: the dependency accumulation and BC).
#pragma once

#include "bc_internal.cuh"

namespace bcg {

// Algorithm 4 (Compute-Dist-to-v) for source s = this thread, over the in-edges
// (x_j, v) of the update, followed by the affected-row test of the IN phase: row s can
// change only if d'(s,v) < d(s,v) or new shortest paths reach v (sigma-hat > 0).
// SYM: the graph is undirected and the state is the one before the update, whose d and
// sigma are symmetric, so d(s,x) is read as d(x,s) (consecutive threads then read
// consecutive entries of row x instead of one entry of each row).
// Returns whether row s can change.
template <typename DT, bool SYM = false>
__device__ __forceinline__ bool dev_alg4_in(int s, int ld, const DT* __restrict__ D, const uint64_t* __restrict__ S,
                          int v, const VEdge* __restrict__ e, int k, int directed,
                          DT* fD, uint64_t* fS, uint64_t* fM, int32_t* err) {
    const int64_t INF = Inf<DT>::v;
    const size_t rs = (size_t)s * ld;
    auto at = [&](int x) { return SYM ? (size_t)x * ld + s : rs + x; };
    const int64_t old = D[at(v)];
    int64_t cur = old;
    uint64_t sig = S[at(v)];
    uint64_t hat = 0;
    bool sat = false;
    for (int j = 0; j < k; ++j) {
        const VEdge ed = e[j];
        if (directed && ed.dir != 0) continue;
        const int64_t dx = D[at(ed.x)];
        if (dx == INF) continue;
        const int64_t dj = dsum<DT>(dx, ed.w);
        if (dj == SAT) {
            sat = true;
            continue;
        }
        const uint64_t sx = S[at(ed.x)];
        if (cur == dj) {
            sig = add_chk(sig, sx, err);
            hat += sx;
        } else if (cur > dj) {
            cur = dj;
            sig = sx;
        }
    }
    // v reachable from s only through a sum that does not fit: d'(s,v) overflows.
    if (sat && cur == INF) set_err(err, ERRF_DIST);
    const bool dec = cur < old;
    const bool aff = dec || hat != 0;
    fD[s] = (DT)cur;
    fS[s] = sig;
    fM[s] = dec ? sig : hat;
    return aff;
}

// OUT phase, row test: row s (s != v) can change only through a new shortest path
// s ~> v -> x_j, i.e. d'(s,v) + w'(v,x_j) <= d'(s,x_j) for some out-edge of the update.
// Returns that.
template <typename DT>
__device__ __forceinline__ bool dev_rows_out(int s, int ld, const DT* __restrict__ D, const uint64_t* __restrict__ S,
                           int v, const VEdge* __restrict__ e, int k, int directed,
                           DT* fD, uint64_t* fS, uint64_t* fM, int32_t* err) {
    const int64_t INF = Inf<DT>::v;
    const size_t rs = (size_t)s * ld;
    const int64_t dsv = D[rs + v];
    const uint64_t ssv = S[rs + v];
    bool aff = false;
    if (s != v && dsv != INF) {
        for (int j = 0; j < k; ++j) {
            const VEdge ed = e[j];
            if (directed && ed.dir != 1) continue;
            const int64_t dy = D[rs + ed.x];
            const int64_t c = dsum<DT>(dsv, ed.w);
            // A sum that does not fit can only matter where d'(s,x_j) is INF; the row is
            // then kept so that the scan decides (and reports a distance overflow).
            if (c == SAT) {
                if (dy == INF) aff = true;
                continue;
            }
            if (c <= dy) aff = true;
        }
    }
    fD[s] = (DT)dsv;
    fS[s] = ssv;
    fM[s] = ssv;
    return aff;
}

// Algorithm 4 on the reversed graph G'_R, for "source" t of G'_R = target t of G: the
// out-edges (v, x_j) of the update are in-edges of v in G'_R, and d_R(t, x_j) is
// d'(x_j, t), read from row x_j.  Produces row v of the result;
// returns whether its entry t changes.
template <typename DT>
__device__ __forceinline__ bool dev_alg4_out(int t, int ld, const DT* __restrict__ D, const uint64_t* __restrict__ S,
                           int v, const VEdge* __restrict__ e, int k, int directed,
                           DT* cD, uint64_t* cS, uint64_t* cM, int32_t* err) {
    const int64_t INF = Inf<DT>::v;
    const size_t rv = (size_t)v * ld;
    const int64_t old = D[rv + t];
    int64_t cur = old;
    uint64_t sig = S[rv + t];
    uint64_t hat = 0;
    bool sat = false;
    for (int j = 0; j < k; ++j) {
        const VEdge ed = e[j];
        if (directed && ed.dir != 1) continue;
        const size_t ry = (size_t)ed.x * ld;
        const int64_t dy = D[ry + t];
        if (dy == INF) continue;
        const int64_t dj = dsum<DT>(ed.w, dy);
        if (dj == SAT) {
            sat = true;
            continue;
        }
        const uint64_t sy = S[ry + t];
        if (cur == dj) {
            sig = add_chk(sig, sy, err);
            hat += sy;
        } else if (cur > dj) {
            cur = dj;
            sig = sy;
        }
    }
    if (sat && cur == INF) set_err(err, ERRF_DIST);
    const bool dec = cur < old;
    cD[t] = (DT)cur;
    cS[t] = sig;
    cM[t] = dec ? sig : hat;
    return dec || hat != 0;
}

// Appends s to a list where the lane wants to: one atomic per warp (every lane of the
// warp calls it).
__device__ __forceinline__ void append_row(bool want, int s, int32_t* rows, int32_t* count) {
    const unsigned b = __ballot_sync(0xffffffffu, want);
    if (!b) return;
    const int lane = threadIdx.x & 31;
    int p = 0;
    if (lane == 0) p = atomicAdd(count, __popc(b));
    p = __shfl_sync(0xffffffffu, p, 0) + __popc(b & ((1u << lane) - 1u));
    if (want) rows[p] = s;
}

// One write into the E* superset.
__device__ __forceinline__ void dev_estar_write(const EOp& o, Arc* e_arc, int64_t* e_w64, int32_t* e_len) {
    if (o.slot >= 0) {
        e_arc[o.slot] = make_arc(o.a, o.b, o.w);
        if (e_w64) e_w64[o.slot] = o.w;
    }
    atomicMax(e_len + o.a, o.len_a);   // lengths only grow between rebuilds
}

// BC's change in an update is summed per column as fixed-point words (A in units of 2^-24,
// B of 2^-71) by integer atomics, so the total does not depend on the order in which rows
// and CTAs add (the result is deterministic) and is exact up to the rounding of each
// dependency to 2^-71, its own last bit or less from 2^-23 on.  Where pairs have very many
// shortest paths dependencies, and BC with them, are smaller; what those have below 2^-71
// goes to a third word (C in units of 2^-112), which few updates touch (fix[3n] tells).
//
// A dependency v = hi + lo, |v| < 2^15, as these words, in single precision only (fp64
// runs at a small fraction of the fp32 rate here): with h = hi * 2^24 and a = rint(h), h
// and h - a are exact, and (h - a) * 2^47 and lo * 2^71 (|lo| <= 2^-10) are exact
// scalings, each rounded to an integer once.  |A| <= 2^39, |B| <= 2^61 + 2^46, |C| <= 2^41.
struct FixWords {
    long long A, B, C;
};
__device__ __forceinline__ FixWords fix_words(ff v) {   // but C
    const float h = v.hi * 0x1p24f, a = rintf(h);
    return FixWords{__float2ll_rn(a), __float2ll_rn((h - a) * 0x1p47f) + __float2ll_rn(v.lo * 0x1p71f), 0};
}
// 0 < |v| < 2^-23, and its C: what the two roundings of B leave, exactly.
__device__ __forceinline__ bool fix_small(ff v) { return (__float_as_uint(v.hi) & 0x7FFFFFFFu) - 1u < 0x33FFFFFFu; }
__device__ __forceinline__ long long fix_rest(ff v) {
    const float h = v.hi * 0x1p24f, r = (h - rintf(h)) * 0x1p47f, l = v.lo * 0x1p71f;
    return __float2ll_rn((r - rintf(r)) * 0x1p41f) + __float2ll_rn((l - rintf(l)) * 0x1p41f);
}
// B's high bits carried into A: |B| <= 2^46 is left.
__device__ __forceinline__ void fix_carry(FixWords& w) {
    const long long c = (w.B + (1ll << 46)) >> 47;
    w.A += c;
    w.B -= c << 47;
}
// Adds w to column x's words (A and B side by side, the C of all n columns behind them): a
// column has at most 2^15 addends of each kind, so |A| < 2^55, |B| <= 2^62 and |C| < 2^58.
__device__ __forceinline__ void fix_add(int64_t* fix, int n, int x, FixWords w) {
    fix_carry(w);
    unsigned long long* p = reinterpret_cast<unsigned long long*>(fix + 2 * (size_t)x);
    if (w.A) atomicAdd(p, (unsigned long long)w.A);
    if (w.B) atomicAdd(p + 1, (unsigned long long)w.B);
    if (w.C) {
        atomicAdd(reinterpret_cast<unsigned long long*>(fix + 2 * (size_t)n + x), (unsigned long long)w.C);
        fix[3 * (size_t)n] = 1;
    }
}
// BC(x) changes by delta_s(x)'s change from old to now.
__device__ __forceinline__ void bc_fix_change(int64_t* fix, int n, int x, ff old, ff now) {
    if (old.hi == now.hi && old.lo == now.lo) return;
    const FixWords w0 = fix_words(old), w1 = fix_words(now);
    FixWords w{w1.A - w0.A, w1.B - w0.B, 0};
    if (fix_small(old) || fix_small(now)) w.C = fix_rest(now) - fix_rest(old);
    fix_add(fix, n, x, w);
}

// Vector access of VEC consecutive distances (16 bytes).
template <typename DT> struct Vec;
template <> struct Vec<int32_t> {
    static constexpr int N = 4;
    using T = int4;
    __device__ static void unpack(const T& x, int64_t* o) { o[0] = x.x; o[1] = x.y; o[2] = x.z; o[3] = x.w; }
    __device__ static void set(T& x, int i, int64_t val) {
        if (i == 0) x.x = (int32_t)val; else if (i == 1) x.y = (int32_t)val;
        else if (i == 2) x.z = (int32_t)val; else x.w = (int32_t)val;
    }
};
template <> struct Vec<int64_t> {
    static constexpr int N = 2;
    using T = longlong2;
    __device__ static void unpack(const T& x, int64_t* o) { o[0] = x.x; o[1] = x.y; }
    __device__ static void set(T& x, int i, int64_t val) { if (i == 0) x.x = val; else x.y = val; }
};

constexpr int kScanThreads = 256;

template <typename DT>
struct ScanArgs {
    int ld;                // entries of a state row: the columns of a pass (those past n hold INF)
    DT* D;
    uint64_t* S;
    const int32_t* rows;
    const int32_t* count;
    const DT* fD;          // per row s: distance to v (after the IN phase)
    const uint64_t* fS;    // per row s: path count to v
    const uint64_t* fM;    // per row s: multiplier of a tie
    const DT* cD;          // per column t: distance from v
    const uint64_t* cS;    // per column t: path count from v
    const uint64_t* cM;    // per column t: multiplier of a tie
    int skip_row;
    // Ties with a zero tie multiplier add no paths (sigma += rowM * colM = 0), so for
    // integer distances such a pair can change only if cand < d, i.e. cand + 1 <= d.
    // tie_rows: rows with rowM = 0 take the quick test with rd + 1 (the IN phase, where
    // every finite column has colM = sigma(v,t) > 0);  tie_cols: columns with colM = 0
    // are staged as c + 1 (the OUT phase, where every finite row has rowM = sigma(s,v)
    // > 0).  Never both in one pass: cand + 2 <= d would miss an improvement by one.
    int tie_rows;
    int tie_cols;
    int32_t* err;
    int64_t* stats;        // [4] pairs with a lower distance [5] pairs with new tied paths [6] rows
    PairRec rec;           // when rec.tcnt is set: record the changed pairs (pair corrections)
    // Second row list with its own column vector (the fused pass of an undirected edge
    // update: the rows whose new paths use the edge as v -> u); rows2 = NULL: one list.
    const int32_t* rows2;
    const int32_t* count2;
    const DT* cD2;
    const uint64_t* cS2;
    const uint64_t* cM2;
};

// The rank-1 rule of Lemma 2 / Lemma 4 for one pair, given the candidate distance
// cand = rd + cd through v:  cand > d: unchanged;  cand == d: sigma += rowM * colM
// (new shortest paths through v);  cand < d: d = cand, sigma = rowS * colS.
template <typename DT>
__device__ __forceinline__ bool pair_rule(int64_t cand, int64_t old, size_t idx, uint64_t rs,
                                          uint64_t rm, uint64_t cs, uint64_t cm,
                                          uint64_t* S, int32_t* err, int64_t* newd, int* ties) {
    if (cand == SAT) {
        if (old == Inf<DT>::v) set_err(err, ERRF_DIST);
        return false;
    }
    if (cand > old) return false;
    if (cand < old) {
        S[idx] = mul_chk(rs, cs, err);
        *newd = cand;
        return true;
    }
    const uint64_t p = mul_chk(rm, cm, err);
    if (p != 0ull) {
        S[idx] = add_chk(S[idx], p, err);
        ++*ties;
    }
    return false;
}

// Quick test of the rank-1 rule on VN consecutive pairs (s, t .. t+VN-1) of row s with
// distances dv and column distances cv: can any of them change?  (False positives only
// cost time: scan_vec applies the exact rule.)
// small: rd plus every finite column value stays below INF, so no finite sum can
// overflow and a pair with d = INF and an INF column term cannot pass.
template <typename DT>
__device__ __forceinline__ bool quick_vec(const typename Vec<DT>::T& dv, const typename Vec<DT>::T& cv, int64_t rd,
                                          bool small = false) {
    using V = Vec<DT>;
    constexpr int VN = V::N;
    const int64_t INF = Inf<DT>::v;
    bool any = false;
    if constexpr (sizeof(DT) == 4) {
        // both terms are below 2^31, so their sum fits 32 bits: a pair can change only if
        // the sum does not exceed d (or d is INF, where a sum that does not fit must be
        // reported).  An INF column term passes only where d is INF or rd is 0; the rule
        // skips it.
        const uint32_t r32 = (uint32_t)rd;
        const int32_t* dp = reinterpret_cast<const int32_t*>(&dv);
        const int32_t* cp = reinterpret_cast<const int32_t*>(&cv);
        if (small) {
#pragma unroll
            for (int q = 0; q < VN; ++q) any |= r32 + (uint32_t)cp[q] <= (uint32_t)dp[q];
        } else {
#pragma unroll
            for (int q = 0; q < VN; ++q) {
                const uint32_t sum = r32 + (uint32_t)cp[q];
                any |= (sum <= (uint32_t)dp[q]) | (dp[q] == INT32_MAX);
            }
        }
    } else {
        int64_t dd0[VN], cd0[VN];
        V::unpack(dv, dd0);
        V::unpack(cv, cd0);
#pragma unroll
        for (int q = 0; q < VN; ++q) {
            if (cd0[q] == INF) continue;
            const int64_t cand = dsum<DT>(rd, cd0[q]);
            any |= (cand <= dd0[q]) || (cand == SAT);
        }
    }
    return any;
}

// The rank-1 rule on the VN consecutive pairs (s, t .. t+VN-1) of row s, given their
// distances dv (updated in place) and the column distances cv; sigma is read only on
// ties and written only where the pair changes.  Returns whether a distance changed
// (dv must then be written back).
template <typename DT>
__device__ __forceinline__ bool rule_vec(const ScanArgs<DT>& a, int s, size_t rowoff, int t, typename Vec<DT>::T& dv,
                                         const typename Vec<DT>::T& cv, int64_t rd, uint64_t rs, uint64_t rm,
                                         int& n_changed, int& n_ties) {
    using V = Vec<DT>;
    constexpr int VN = V::N;
    const int64_t INF = Inf<DT>::v;
    int64_t dd[VN], cd[VN];
    V::unpack(dv, dd);
    V::unpack(cv, cd);
    bool wr = false;
#pragma unroll
    for (int q = 0; q < VN; ++q) {
        if (cd[q] == INF) continue;
        const int64_t cand = dsum<DT>(rd, cd[q]);
        int64_t nd;
        const int ties0 = n_ties;
        const uint64_t sig0 = a.rec.tcnt ? a.S[rowoff + t + q] : 0ull;
        if (pair_rule<DT>(cand, dd[q], rowoff + t + q, rs, rm, a.cS[t + q], a.cM[t + q], a.S, a.err, &nd,
                          &n_ties)) {
            V::set(dv, q, nd);
            wr = true;
            ++n_changed;
            if (a.rec.tcnt) record_change<DT>(a.rec, s, t + q, dd[q], sig0);
        } else if (n_ties != ties0 && a.rec.tcnt) {
            record_change<DT>(a.rec, s, t + q, dd[q], sig0);
        }
    }
    return wr;
}

// VN consecutive path counts from a 16-byte aligned address, in 16-byte loads.
template <int VN>
__device__ __forceinline__ void load_u64s(const uint64_t* p, uint64_t* o) {
#pragma unroll
    for (int h = 0; h < VN / 2; ++h) {
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(p + 2 * h);
        o[2 * h] = x.x;
        o[2 * h + 1] = x.y;
    }
}

// The rank-1 rule on a vector like rule_vec, recording nothing: returns the mask of
// pairs q whose distance dropped (bits 0..7) or that gained paths at the same distance
// (bits 8..15), with their values before the rule in dold / sold, for a caller that
// records the changes of a whole warp together.  The vector's path counts and the
// column's counts and multipliers are loaded together (16-byte loads: t is a multiple
// of VN and so is ld), and the changed counts written back together, so a vector costs
// one round trip to memory instead of one per pair.
template <typename DT>
__device__ __forceinline__ unsigned rule_vec_masked(const ScanArgs<DT>& a, const uint64_t* colS,
                                                    const uint64_t* colM, size_t rowoff, int t,
                                                    typename Vec<DT>::T& dv, const typename Vec<DT>::T& cv,
                                                    int64_t rd, uint64_t rs, uint64_t rm, int& n_changed,
                                                    int& n_ties, int64_t* dold, uint64_t* sold) {
    using V = Vec<DT>;
    constexpr int VN = V::N;
    const int64_t INF = Inf<DT>::v;
    int64_t dd[VN], cd[VN];
    uint64_t sg[VN], cs[VN], cm[VN];
    V::unpack(dv, dd);
    V::unpack(cv, cd);
    load_u64s<VN>(a.S + rowoff + t, sg);
    load_u64s<VN>(colS + t, cs);
    load_u64s<VN>(colM + t, cm);
    unsigned mask = 0;
#pragma unroll
    for (int q = 0; q < VN; ++q) {
        dold[q] = dd[q];
        sold[q] = sg[q];
        if (cd[q] == INF) continue;
        const int64_t cand = dsum<DT>(rd, cd[q]);
        if (cand == SAT) {
            if (dd[q] == INF) set_err(a.err, ERRF_DIST);
            continue;
        }
        if (cand > dd[q]) continue;
        if (cand < dd[q]) {
            sg[q] = mul_chk(rs, cs[q], a.err);
            V::set(dv, q, cand);
            ++n_changed;
            mask |= 1u << q;
        } else {
            const uint64_t p = mul_chk(rm, cm[q], a.err);
            if (p != 0ull) {
                sg[q] = add_chk(sg[q], p, a.err);
                ++n_ties;
                mask |= 1u << (q + 8);
            }
        }
    }
    if (mask) {
#pragma unroll
        for (int h = 0; h < VN / 2; ++h)
            *reinterpret_cast<ulonglong2*>(a.S + rowoff + t + 2 * h) = make_ulonglong2(sg[2 * h], sg[2 * h + 1]);
    }
    return mask;
}

// Records, for the whole warp, the changes one rule_vec_masked per lane found: lane
// holds row s (s < 0: nothing), the vector's first column t (a multiple of VN, so its
// pairs share one change-map word) and the changed pairs in bits; lanes with the same
// row must be consecutive.  One change-map OR per lane and one target-count atomic per
// run of lanes on the same row; the first change of a pair in the update saves its old
// values and lists it, as record_change does.  Every lane of the warp must call it.
template <typename DT>
__device__ __forceinline__ void record_changes_warp(const PairRec& r, int s, int t, unsigned bits,
                                                    const int64_t* dold, const uint64_t* sold) {
    const int lane = threadIdx.x & 31;
    if (s >= 0 && bits) {
        uint32_t* w = r.chg + (size_t)s * r.chg_words + (t >> 5);
        unsigned wb = bits << (t & 31);
        if (!r.first) wb &= ~*w;   // pairs already recorded in this update keep their saved values
        bits = wb >> (t & 31);
        if (wb) atomicOr(w, wb);
        const size_t i0 = (size_t)s * r.ld + t;
        for (unsigned b = bits; b; b &= b - 1) {
            const int q = __ffs(b) - 1;
            static_cast<DT*>(r.oldD)[i0 + q] = (DT)dold[q];
            r.oldS[i0 + q] = sold[q];
        }
    } else {
        bits = 0;
    }
    // segmented scan of the counts over runs of lanes with the same row
    const int c = __popc(bits);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int s_prev = __shfl_up_sync(0xffffffffu, s, 1);
    const unsigned starts = __ballot_sync(0xffffffffu, lane == 0 || s_prev != s);
    const unsigned upto = lane == 31 ? 0xffffffffu : ((2u << lane) - 1u);
    const int start = 31 - __clz(starts & upto);
    const unsigned after = starts & ~upto;
    const int end = after ? __ffs(after) - 2 : 31;
    const int before = __shfl_sync(0xffffffffu, incl, start > 0 ? start - 1 : 0);
    const int base_incl = start > 0 ? before : 0;
    const int total = __shfl_sync(0xffffffffu, incl, end) - base_incl;
    int base = 0;
    if (lane == start && s >= 0 && total > 0) base = atomicAdd(r.tcnt + s, total);
    base = __shfl_sync(0xffffffffu, base, start);
    int pos = base + (incl - c - base_incl);
    for (unsigned b = bits; b; b &= b - 1, ++pos)
        if (pos < r.tcap) r.tlist[(size_t)s * r.tcap + pos] = t + __ffs(b) - 1;
}

template <typename DT>
__device__ __forceinline__ bool scan_vec(const ScanArgs<DT>& a, int s, size_t rowoff, int t, typename Vec<DT>::T& dv,
                                         const typename Vec<DT>::T& cv, int64_t rd, uint64_t rs, uint64_t rm,
                                         int& n_changed, int& n_ties) {
    if (!quick_vec<DT>(dv, cv, rd)) return false;
    return rule_vec<DT>(a, s, rowoff, t, dv, cv, rd, rs, rm, n_changed, n_ties);
}

// One work item of the rank-1 pass: row s (scalars rd, rs, rm), chunk c of CW columns.
template <typename DT, int U>
__device__ __forceinline__ void dev_scan_item(const ScanArgs<DT>& a, int s, int64_t rd, uint64_t rs, uint64_t rm,
                                              int c, int& n_changed, int& n_ties) {
    using V = Vec<DT>;
    constexpr int VN = V::N;
    constexpr int CW = kScanThreads * VN * U;
    const int ld = a.ld;
    const size_t rowoff = (size_t)s * ld;
    DT* __restrict__ Drow = a.D + rowoff;
    const int t0 = c * CW;
    const int tid = threadIdx.x % kScanThreads;
    typename V::T dv[U], cv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int t = t0 + (u * kScanThreads + tid) * VN;
        if (t < ld) {
            dv[u] = __ldcs(reinterpret_cast<const typename V::T*>(Drow + t));
            cv[u] = __ldg(reinterpret_cast<const typename V::T*>(a.cD + t));
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int t = t0 + (u * kScanThreads + tid) * VN;
        if (t >= ld) break;
        if (scan_vec<DT>(a, s, rowoff, t, dv[u], cv[u], rd, rs, rm, n_changed, n_ties))
            *reinterpret_cast<typename V::T*>(Drow + t) = dv[u];
    }
}

// Fold the per-thread counters of the scan into the handle's statistics (whole warps).
__device__ __forceinline__ void scan_stats(int64_t* stats, int n_changed, int n_ties) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        n_changed += __shfl_xor_sync(0xffffffffu, n_changed, o);
        n_ties += __shfl_xor_sync(0xffffffffu, n_ties, o);
    }
    if ((threadIdx.x & 31) == 0 && (n_changed | n_ties)) {
        atomicAdd(reinterpret_cast<unsigned long long*>(stats + 4), (unsigned long long)n_changed);
        atomicAdd(reinterpret_cast<unsigned long long*>(stats + 5), (unsigned long long)n_ties);
    }
}

template <typename DT>
__device__ __forceinline__ void dev_write_row(int t, int ld, DT* D, uint64_t* S, int v, const DT* cD, const uint64_t* cS,
                            const int32_t* err) {
    D[(size_t)v * ld + t] = cD[t];
    S[(size_t)v * ld + t] = cS[t];
}

template <typename DT>
struct AccArgs {
    int n;
    int ld;
    const DT* D;
    uint64_t* S;
    ff* Dl;
    const int32_t* e_off;
    const int32_t* e_len;
    const Arc* e_arc;
    const int64_t* e_w64;
    int64_t e_used;      // slots in use, a multiple of kGroupSlots (the rest of the last group is empty)
    const int32_t* rows;
    const int32_t* count;
    int32_t* ws;
    int64_t ws_stride;
    int32_t* err;
    int64_t* bcfix;      // BC's change (updates)
    AccLayout lay;
};

constexpr uint32_t FULL = 0xffffffffu;

// DAG in-degrees still to be taken, in 16-bit halves of 32-bit words (below 32768).  Most
// vertices have one: they are marked kOneTail and need no atomic, which the levels'
// chains would wait for (an update's vertices without DAG out-arcs are marked 0, they
// join no level).  The others count down, and the last tail to be taken is told.
constexpr uint32_t kOneTail = 0x8000;
__device__ __forceinline__ void cnt_inc(uint32_t* cnt, int b) {
    atomicAdd(cnt + (b >> 1), 1u << ((b & 1) << 4));
}
__device__ __forceinline__ bool cnt_last(uint32_t* cnt, int b) {
    const uint32_t sh = (b & 1) << 4;
    return ((atomicSub(cnt + (b >> 1), 1u << sh) >> sh) & 0xFFFFu) == 1u;
}
__device__ __forceinline__ uint32_t cnt_get(const uint32_t* cnt, int b) {
    return reinterpret_cast<const volatile uint16_t*>(cnt)[b];
}
// To the marks above, by the vertex's own thread, once all are counted.
__device__ __forceinline__ void cnt_mark(uint32_t* cnt, int x, bool leave_out) {
    uint16_t* c = reinterpret_cast<uint16_t*>(cnt) + x;
    if (leave_out) *c = 0;
    else if (*c == 1) *c = (uint16_t)kOneTail;
}

__device__ __forceinline__ ff warp_sum(ff x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = ff_add(x, ff_shfl_xor(x, o));
    return x;
}

// ---- one source's dependencies
//
constexpr int kNearLevels = 512;
// The arrays of one accumulation CTA (acc_layout says where each lives).
struct AccMem {
    uint32_t* row;     // [np] the source's distances in 32 bits; dead once the DAG is read off
    uint16_t* first;   // [np] (over row) first pool entry of a vertex's heads
    uint32_t* cnt;     // [np / 2] (over row) in-degrees
    uint32_t* mask;    // [words] bit per slot of the superset: its arc is in DAG'(s)
    uint16_t* base;    // [words] first pool entry of a mask word's arcs
    uint16_t* order;   // [np] (over mask and base; without the pool over first) vertices with DAG
                       // out-arcs, level by level
    uint16_t* pool;    // [pcap + 4] heads of the DAG arcs
    uint64_t* cell;    // [np] sigma_sx, then rho(x) once x is finished
    uint32_t* sink;    // [np / 32] bit per vertex: no DAG out-arc
    uint32_t* big;     // [np / 32] bit per vertex: kBigDag DAG out-arcs or more
    uint16_t* level;   // [kNearLevels] start of each level in order, the later ones in far
    uint16_t* far;     // [np] (work space)
    __device__ __forceinline__ uint16_t& level_at(int l) const { return l < kNearLevels ? level[l] : far[l]; }
};
// cp.async of 16 bytes into shared memory, read back after async_wait_all and a barrier.
__device__ __forceinline__ void async_copy16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

struct AccShared {
    int arcs;          // pool entries handed out
    int q[3];          // vertices appended for the next level, by level modulo 3
};

// SM: every array is in shared memory (the compiler then addresses it as such).
template <bool SM>
__device__ __forceinline__ AccMem acc_mem(const AccLayout& l, unsigned char* smem, int32_t* wsb) {
    unsigned char* ws = reinterpret_cast<unsigned char*>(wsb);
    AccMem m;
    auto at = [&](int32_t off, bool in_ws) { return (SM || !in_ws) ? smem + off : ws + off; };
    m.row = reinterpret_cast<uint32_t*>(smem + l.row);
    m.first = reinterpret_cast<uint16_t*>(smem + l.row);
    m.cnt = reinterpret_cast<uint32_t*>(smem + l.cnt);
    m.level = reinterpret_cast<uint16_t*>(smem + l.level);
    m.far = reinterpret_cast<uint16_t*>(ws + l.far);
    m.sink = reinterpret_cast<uint32_t*>(smem + l.sink);
    m.big = reinterpret_cast<uint32_t*>(smem + l.big);
    m.mask = reinterpret_cast<uint32_t*>(at(l.mask, l.mask_ws));
    m.base = reinterpret_cast<uint16_t*>(at(l.base, l.mask_ws));
    m.order = reinterpret_cast<uint16_t*>(m.mask);
    m.pool = reinterpret_cast<uint16_t*>(at(l.pool, l.pool_ws));
    m.cell = reinterpret_cast<uint64_t*>(at(l.cell, l.cell_ws));
    return m;
}

__device__ __forceinline__ uint64_t cell_rho(ff r) {
    return ((uint64_t)__float_as_uint(r.hi) << 32) | __float_as_uint(r.lo);
}
__device__ __forceinline__ ff cell_ff(uint64_t c) {
    return ff{__uint_as_float((uint32_t)(c >> 32)), __uint_as_float((uint32_t)c)};
}

// The last head of a vertex carries kLastHead.  A vertex with kBigDag DAG out-arcs or
// more is taken by a whole warp; its first pool entry is their number and the heads
// follow.
constexpr int kBigDag = 31;
constexpr uint32_t kLastHead = 0x8000, kHeadMask = 0x7FFF;
constexpr int kHugeDag = 256;
constexpr uint16_t kPlaceLater = 0xFFFF;   // (no pool entry: the pool is shorter)

__device__ __forceinline__ bool bit_of(const uint32_t* w, int x) { return (w[x >> 5] >> (x & 31)) & 1u; }

// The heads of a vertex from pool entry p on, four at a time (a chain of one head after
// the other costs two or three shared-memory latencies a head): f(h, valid) with up to
// four heads, bit u of valid set where h[u] is one.  All lanes of a warp call it together,
// those without a vertex with go false, and f is called by all of them.
template <typename F>
__device__ __forceinline__ void four_heads(const AccMem& m, int p, bool go, F&& f) {
    while (__any_sync(FULL, go)) {
        uint32_t h[4] = {0u, 0u, 0u, 0u};
        if (go) {
#pragma unroll
            for (int u = 0; u < 4; ++u) h[u] = m.pool[p + u];   // the pool is four entries longer
        }
        // up to the first that is marked last
        const unsigned last = (h[0] & kLastHead) >> 15 | (h[1] & kLastHead) >> 14 | (h[2] & kLastHead) >> 13 |
                              (h[3] & kLastHead) >> 12;
        const unsigned valid = go ? (last ^ (last - 1u)) & 15u : 0u;
        go = go && last == 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) h[u] = (valid >> u) & 1u ? h[u] & kHeadMask : 0u;
        f(h, valid);
        p += 4;
    }
}

// Appends the lanes' vertices (u < 4, where bit u of ready is set) to the next level.
__device__ __forceinline__ void append4(const AccMem& m, int* q, int at, unsigned ready, const uint32_t* b) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    unsigned bal[4];
    int tot = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        bal[u] = __ballot_sync(FULL, (ready >> u) & 1u);
        tot += __popc(bal[u]);
    }
    if (!tot) return;
    int p = 0;
    if (lane == 0) p = atomicAdd(q, tot);
    p = at + __shfl_sync(FULL, p, 0);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if ((ready >> u) & 1u) m.order[p + __popc(bal[u] & lt)] = (uint16_t)b[u];
        p += __popc(bal[u]);
    }
}

// DAG'(s) read off the distance row: a lane per slot of the superset (the loads of a
// group of slots are issued before any is used).  The heads of the DAG arcs go to the
// pool, those of a group together in slot order.  Arc (x, b, w) is in DAG'(s) where
// d(s,x) + w = d(s,b) (Eq. 1).  On the row in shared memory INF is 2^31 - 1, a weight that
// does not fit 31 bits is held as that too and an empty slot's as 2^31, so one 32-bit
// sum and compare decides: a sum with INF or an empty slot's exceeds every entry of the
// row, none wraps, and no finite sum equals INF (where b is unreachable no arc from a
// reachable x leads to it).  WIDE: some finite distance of the row does not fit;
// distances and weights then come from memory.
template <typename DT, int T, bool WIDE>
__device__ __forceinline__ void dag_slots(const AccArgs<DT>& a, const AccMem& m, const DT* Ds, int* s_arcs) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    constexpr int NW = T / 32, U = kGroupSlots / 32;
    const int ngroup = (int)(a.e_used / kGroupSlots);
    for (int g = warp; g < ngroup; g += NW) {
        const Arc* ap = a.e_arc + (int64_t)g * kGroupSlots + lane;
        Arc r[U];
#pragma unroll
        for (int u = 0; u < U; ++u) r[u] = ap[32 * u];
        unsigned word[U];
        int tot = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            bool on;
            if constexpr (WIDE) {
                const int64_t dx = __ldg(Ds + r[u].src());
                on = !r[u].empty() && dx != Inf<DT>::v &&
                     dx + a.e_w64[(int64_t)g * kGroupSlots + 32 * u + lane] == (int64_t)__ldg(Ds + r[u].dst());
            } else {
                on = m.row[r[u].src()] + (uint32_t)r[u].w == m.row[r[u].dst()];
            }
            word[u] = __ballot_sync(FULL, on);
            tot += __popc(word[u]);
        }
        int p = 0;
        if (lane == 0 && tot) p = atomicAdd(s_arcs, tot);
        p = __shfl_sync(FULL, p, 0);
        const bool fits = p + tot <= a.lay.pcap;   // past the end the arcs are only counted
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (fits && ((word[u] >> lane) & 1u)) m.pool[p + __popc(word[u] & lt)] = (uint16_t)r[u].dst();
            if (lane == u) {
                m.mask[g * U + u] = word[u];
                m.base[g * U + u] = (uint16_t)p;
            }
            p += __popc(word[u]);
        }
    }
}

// DAG out-degree of the vertex whose segment is [beg, beg + len), and its heads' first
// pool entry where they lie in one group.
__device__ __forceinline__ int count_dag(const AccMem& m, int beg, int len, int* p) {
    if (len <= 0) return 0;
    const int w = beg >> 5, sh = beg & 31;
    const uint32_t m0 = m.mask[w];
    *p = (int)m.base[w] + __popc(m0 & ((1u << sh) - 1u));
    if (sh + len <= 32) return __popc((m0 >> sh) & (0xffffffffu >> (32 - len)));
    int k = __popc(m0 >> sh);
    const int end = beg + len, w1 = (end - 1) >> 5;
    for (int v = w + 1; v < w1; ++v) k += __popc(m.mask[v]);
    return k + __popc(m.mask[w1] & (0xffffffffu >> (31 - ((end - 1) & 31))));
}

// Mask word w of the segment of slots [beg, end].
__device__ __forceinline__ uint32_t segment_word(const AccMem& m, int w, int beg, int end) {
    uint32_t b = m.mask[w];
    if (w == beg >> 5) b &= 0xffffffffu << (beg & 31);
    if (w == end >> 5) b &= 0xffffffffu >> (31 - (end & 31));
    return b;
}
// First pool entry of the heads of a vertex with 0 < k < kHugeDag DAG out-arcs; p as count_dag
// gives it.  Marks the last head.  Heads that lie in several groups, and those of a big vertex
// behind their number, are copied to the end of the pool (past its end they are only
// counted).
__device__ __forceinline__ uint16_t place_heads(const AccMem& m, int pcap, int* s_arcs, int beg, int len, int k, int p) {
    const int h = k >= kBigDag ? 1 : 0, end = beg + len - 1;
    if (h || beg / kGroupSlots != end / kGroupSlots) {
        p = atomicAdd(s_arcs, k + h);
        if (p + k + h > pcap) return 0;
        int at = p;
        if (h) m.pool[at++] = (uint16_t)k;
        for (int w = beg >> 5; w <= end >> 5; ++w) {
            const uint32_t word = m.mask[w], low = w == beg >> 5 ? (1u << (beg & 31)) - 1u : 0u;
            uint32_t b = word & ~low;
            if (w == end >> 5) b &= 0xffffffffu >> (31 - (end & 31));
            const int p0 = (int)m.base[w] + __popc(word & low), c = __popc(b);
            for (int q = 0; q < c; ++q) m.pool[at++] = m.pool[p0 + q] & kHeadMask;
        }
    }
    if (p + k + h <= pcap) m.pool[p + k + h - 1] |= kLastHead;
    return (uint16_t)p;
}
// A vertex with more is placed by the whole warp (one with fewer by its thread: by warps they
// took 16 updates at BA n = 16384 from 9.19 to 9.41 ms).
__device__ __forceinline__ uint16_t place_big(const AccMem& m, int pcap, int* s_arcs, int beg, int len) {
    const int lane = threadIdx.x & 31, end = beg + len - 1;
    int k = 0;
    for (int w = (beg >> 5) + lane; w <= end >> 5; w += 32) k += __popc(segment_word(m, w, beg, end));
    k = __reduce_add_sync(FULL, k);
    int p = 0;
    if (lane == 0) p = atomicAdd(s_arcs, k + 1);
    p = __shfl_sync(FULL, p, 0);
    if (p + k + 1 > pcap) return 0;
    if (lane == 0) m.pool[p] = (uint16_t)k;
    int at = p + 1;
    for (int w0 = beg >> 5; w0 <= end >> 5; w0 += 32) {   // 32 words at a time
        const int w = w0 + lane;
        int c = 0, p0 = 0;
        if (w <= end >> 5) {
            c = __popc(segment_word(m, w, beg, end));
            p0 = (int)m.base[w] + (w == beg >> 5 ? __popc(m.mask[w] & ((1u << (beg & 31)) - 1u)) : 0);
        }
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int z = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += z;
        }
        const int words = min(32, (end >> 5) - w0 + 1);
        for (int j = 0; j < words; ++j) {
            const int cj = __shfl_sync(FULL, c, j), from = __shfl_sync(FULL, p0, j), to = __shfl_sync(FULL, at + incl - c, j);
            if (lane < cj) m.pool[to + lane] = m.pool[from + lane] & kHeadMask;
        }
        at += __shfl_sync(FULL, incl, 31);
    }
    return (uint16_t)p;
}

// ---- the heads of a DAG with more arcs than the pool holds (ties everywhere, a hub whose
// heads would be copied), from the masks and the superset: the masks stay and `order` takes
// the place of `first`.  One L2 read a head in place of a shared-memory one, as many at a time
// as in the pool's form.  Testing every slot of a vertex again, a thread a vertex, took 13.0 ms
// where this takes 3.7 (k_accum of the static computation, BA n = 4096 with unit weights; BA
// n = 12000 174 and 45 ms), and 27 and 1.1 ms for a star of 4096 vertices.

// As four_heads, for the vertex whose segment is [beg, beg + len).
template <typename F>
__device__ __forceinline__ void four_heads_masked(const Arc* e_arc, const AccMem& m, int beg, int len, bool go, F&& f) {
    const int end = beg + len - 1;
    int w = beg >> 5;
    uint32_t b = go ? segment_word(m, w, beg, end) : 0u;
    while (__any_sync(FULL, go)) {
        int at[4];
        unsigned valid = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            at[u] = 0;
            while (go && b == 0u && w < end >> 5) b = segment_word(m, ++w, beg, end);
            if (b == 0u) continue;
            at[u] = 32 * w + __ffs(b) - 1;
            valid |= 1u << u;
            b &= b - 1u;
        }
        go = go && (b != 0u || w < end >> 5);
        uint32_t h[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) h[u] = (valid >> u) & 1u ? (uint32_t)e_arc[at[u]].dst() : 0u;
        f(h, valid);
    }
}
// Position of bit number i (from 0) of b, which has more than i.
__device__ __forceinline__ int nth_bit(uint32_t b, int i) {
    int p = 0;
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const int c = __popc(b & ((1u << s) - 1u));
        if (i >= c) {
            i -= c;
            b >>= s;
            p += s;
        }
    }
    return p;
}
// The heads of one vertex by a whole warp, head number r by lane r mod 32 in increasing order,
// as from the pool (so a lane's sum has the same terms in the same order): f(have, head).
template <typename F>
__device__ __forceinline__ void big_heads_masked(const Arc* e_arc, const AccMem& m, int beg, int len, F&& f) {
    constexpr int U = 4;
    const int lane = threadIdx.x & 31, end = beg + len - 1;
    int rank = 0;   // warp-uniform
    for (int w0 = beg >> 5; w0 <= end >> 5; w0 += U) {
        uint32_t b[U];
        bool have[U];
        int h[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            b[u] = w0 + u <= end >> 5 ? segment_word(m, w0 + u, beg, end) : 0u;
            const int i = (lane - rank) & 31, c = __popc(b[u]);
            have[u] = i < c;
            h[u] = have[u] ? e_arc[32 * (w0 + u) + nth_bit(b[u], i)].dst() : 0;
            rank += c;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (b[u]) f(have[u], h[u]);
    }
}

// The levels of DAG'(s) forwards (Kahn): a vertex joins the next level when its last DAG
// in-arc is taken; vertices without DAG out-arcs are left out.  Statically the path
// counts go along: sigma_sb is the sum of sigma_sa over the DAG in-arcs (a, b).  Returns
// the number of levels; level l is order[level_at(l) .. level_at(l + 1)).
template <typename DT, bool STATIC, int T, bool POOLED>
__device__ __forceinline__ int dag_levels(const AccArgs<DT>& a, const AccMem& m, AccShared& sh, int s) {
    const int tid = threadIdx.x, lane = tid & 31;
    int lo = 0, hi = bit_of(m.sink, s) ? 0 : 1, L = 0;
    if (tid == 0) {
        m.order[0] = (uint16_t)s;
        m.level_at(0) = 0;
    }
    __syncthreads();   // what lies under order (POOLED: the masks) is dead from here on
    while (lo < hi) {
        int* q = &sh.q[L % 3];
        if (tid == 0) sh.q[(L + 1) % 3] = 0;
        // one more tail, with sx paths, of vertex b is taken: whether it was the last
        auto take = [&](int b, uint64_t sx) {
            const uint32_t c = cnt_get(m.cnt, b);
            if (c == kOneTail) {
                if (STATIC) m.cell[b] = sx;
                return true;
            }
            if (!STATIC && c == 0) return false;
            if (STATIC) {
                const unsigned long long old =
                    atomicAdd(reinterpret_cast<unsigned long long*>(m.cell + b), (unsigned long long)sx);
                if (old + sx < old) set_err(a.err, ERRF_OVERFLOW);
            }
            return cnt_last(m.cnt, b);
        };
        for (int i0 = lo + (tid & ~31); i0 < hi; i0 += T) {   // warp-uniform
            const int i = i0 + lane;
            const bool have = i < hi;
            const int x = have ? m.order[i] : 0;
            const uint64_t sx = STATIC ? m.cell[x] : 0ull;
            if constexpr (POOLED) {
                const bool big = have && bit_of(m.big, x);
                const int p = m.first[x];
                four_heads(m, p, have && !big, [&](const uint32_t* b, unsigned valid) {
                    // one tail only (nearly all): ready, without branches; then the others
                    unsigned ready = 0, others = 0;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const uint32_t c = cnt_get(m.cnt, (int)b[u]);
                        ready |= c == kOneTail ? 1u << u : 0u;
                        others |= c != 0 ? 1u << u : 0u;
                        if (STATIC && c == kOneTail && ((valid >> u) & 1u)) m.cell[b[u]] = sx;
                    }
                    ready &= valid;
                    others &= valid & ~ready;
                    if (others) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if ((others >> u) & 1u) ready |= take((int)b[u], sx) ? 1u << u : 0u;
                    }
                    if (STATIC) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) ready &= ~((unsigned)bit_of(m.sink, (int)b[u]) << u);
                    }
                    append4(m, q, hi, ready, b);
                });
                for (unsigned bb = __ballot_sync(FULL, big); bb; bb &= bb - 1u) {
                    const int src = __ffs(bb) - 1;
                    const int pb = __shfl_sync(FULL, p, src), k = m.pool[pb];
                    const uint64_t sb = STATIC ? m.cell[__shfl_sync(FULL, x, src)] : 0ull;
                    for (int c = 0; c < k; c += 32) {
                        uint32_t b[4] = {0u, 0u, 0u, 0u};
                        unsigned ready = 0;
                        if (c + lane < k) {
                            b[0] = m.pool[pb + 1 + c + lane] & kHeadMask;
                            ready = take((int)b[0], sb) && !bit_of(m.sink, (int)b[0]) ? 1u : 0u;
                        }
                        append4(m, q, hi, ready, b);
                    }
                }
            } else {
                const bool big = have && bit_of(m.big, x);
                const int beg = have ? a.e_off[x] : 0, len = have ? a.e_len[x] : 0;
                four_heads_masked(a.e_arc, m, beg, len, have && !big, [&](const uint32_t* b, unsigned valid) {
                    unsigned ready = 0;
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if ((valid >> u) & 1u) ready |= take((int)b[u], sx) && !bit_of(m.sink, (int)b[u]) ? 1u << u : 0u;
                    append4(m, q, hi, ready, b);
                });
                for (unsigned bb = __ballot_sync(FULL, big); bb; bb &= bb - 1u) {
                    const int src = __ffs(bb) - 1;
                    const uint64_t sb = STATIC ? m.cell[__shfl_sync(FULL, x, src)] : 0ull;
                    big_heads_masked(a.e_arc, m, __shfl_sync(FULL, beg, src), __shfl_sync(FULL, len, src), [&](bool got, int h) {
                        const uint32_t b[4] = {(uint32_t)h, 0u, 0u, 0u};
                        append4(m, q, hi, got && take(h, sb) && !bit_of(m.sink, h) ? 1u : 0u, b);
                    });
                }
            }
        }
        __syncthreads();
        const int c = *q;
        ++L;
        if (tid == 0) m.level_at(L) = (uint16_t)hi;
        lo = hi;
        hi += c;
    }
    return L;
}

// Eq. 4 back over the levels (level 0 is s: delta_s.(s) is not kept).
template <typename DT, bool STATIC, int T, bool POOLED>
__device__ __forceinline__ void dag_pull(const AccArgs<DT>& a, const AccMem& m, int L, ff* out) {
    const int tid = threadIdx.x, lane = tid & 31;
    for (int l = L - 1; l >= 1; --l) {
        const int lo = m.level_at(l), hi = m.level_at(l + 1);
        for (int i0 = lo + (tid & ~31); i0 < hi; i0 += T) {   // warp-uniform
            const int i = i0 + lane;
            const bool have = i < hi;
            const int x = have ? m.order[i] : 0;
            ff old{0.0f, 0.0f};
            if (!STATIC && have) old = out[x];   // used last: on its way meanwhile
            const ff sx = ff_from_u64(m.cell[x]), rx = ff_rcp(sx);
            ff acc{0.0f, 0.0f};
            if constexpr (POOLED) {
                const bool big = have && bit_of(m.big, x);
                const int p = m.first[x];
                four_heads(m, p, have && !big, [&](const uint32_t* b, unsigned valid) {
                    uint64_t c[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) c[u] = (valid >> u) & 1u ? m.cell[b[u]] : 0ull;
#pragma unroll
                    for (int u = 0; u < 4; ++u) acc = ff_add(acc, cell_ff(c[u]));   // + 0 past the end: exact
                });
                for (unsigned bb = __ballot_sync(FULL, big); bb; bb &= bb - 1u) {
                    const int src = __ffs(bb) - 1;
                    const int pb = __shfl_sync(FULL, p, src), k = m.pool[pb];
                    ff part{0.0f, 0.0f};
                    for (int c = lane; c < k; c += 32)
                        part = ff_add(part, cell_ff(m.cell[m.pool[pb + 1 + c] & kHeadMask]));
                    part = warp_sum(part);
                    if (lane == src) acc = part;
                }
            } else {
                const bool big = have && bit_of(m.big, x);
                const int beg = have ? a.e_off[x] : 0, len = have ? a.e_len[x] : 0;
                four_heads_masked(a.e_arc, m, beg, len, have && !big, [&](const uint32_t* b, unsigned valid) {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if ((valid >> u) & 1u) acc = ff_add(acc, cell_ff(m.cell[b[u]]));
                });
                for (unsigned bb = __ballot_sync(FULL, big); bb; bb &= bb - 1u) {
                    const int src = __ffs(bb) - 1;
                    ff part{0.0f, 0.0f};
                    big_heads_masked(a.e_arc, m, __shfl_sync(FULL, beg, src), __shfl_sync(FULL, len, src), [&](bool got, int h) {
                        if (got) part = ff_add(part, cell_ff(m.cell[h]));
                    });
                    part = warp_sum(part);
                    if (lane == src) acc = part;
                }
            }
            // delta(x) = sigma_sx * acc, rho(x) = (1 + delta(x)) / sigma_sx = acc + 1 / sigma_sx
            if (have) {
                m.cell[x] = cell_rho(ff_add(acc, rx));
                const ff now = ff_mul(sx, acc);
                out[x] = now;
                if (!STATIC) bc_fix_change(a.bcfix, a.n, x, old, now);
            }
        }
        __syncthreads();
    }
}

// Once the DAG's levels are known: the vertices without DAG out-arcs are finished, then
// the others back over the levels.
template <typename DT, bool STATIC, int T, bool POOLED>
__device__ __forceinline__ void dag_source(const AccArgs<DT>& a, const AccMem& m, AccShared& sh, int s, uint64_t* Ss,
                                           ff* out) {
    const int n = a.n, tid = threadIdx.x;
    if (!POOLED) {   // the pool's heads were counted as they came; now those of the masks
        for (int t = tid; t < (n + 1) / 2; t += T) m.cnt[t] = 0u;
        __syncthreads();
        constexpr int U = kGroupSlots / 32;
        for (int g = tid >> 5; g < (int)(a.e_used / kGroupSlots); g += T / 32)
#pragma unroll
            for (int u = 0; u < U; ++u)
                if ((m.mask[g * U + u] >> (tid & 31)) & 1u)
                    cnt_inc(m.cnt, a.e_arc[(int64_t)g * kGroupSlots + 32 * u + (tid & 31)].dst());
        __syncthreads();
        for (int x = tid; x < n; x += T) cnt_mark(m.cnt, x, !STATIC && bit_of(m.sink, x));
        __syncthreads();
    }
    const int L = dag_levels<DT, STATIC, T, POOLED>(a, m, sh, s);
    constexpr int VU = 8;
    for (int x0 = tid; x0 < n; x0 += VU * T) {
        ff old[VU];
        bool done[VU];
#pragma unroll
        for (int v = 0; v < VU; ++v) {
            const int x = x0 + v * T;
            done[v] = x < n && (x == s || bit_of(m.sink, x));
            old[v] = ff{0.0f, 0.0f};
            if (!STATIC && done[v]) old[v] = out[x];
        }
#pragma unroll
        for (int v = 0; v < VU; ++v) {
            const int x = x0 + v * T;
            if (x >= n) break;
            const uint64_t sg = m.cell[x];
            if (STATIC) Ss[x] = sg;
            if (done[v]) {
                const ff none{0.0f, 0.0f};
                if (!STATIC) bc_fix_change(a.bcfix, n, x, old[v], none);
                if (STATIC || old[v].hi != 0.0f) out[x] = none;
                if (sg != 0) m.cell[x] = cell_rho(ff_rcp(ff_from_u64(sg)));
            }
        }
    }
    if (STATIC && tid < a.ld - n) {   // the entries past n: no path
        Ss[n + tid] = 0ull;
        out[n + tid] = ff{0.0f, 0.0f};
    }
    __syncthreads();
    dag_pull<DT, STATIC, T, POOLED>(a, m, L, out);
}
template <typename DT, bool STATIC, int T>
__device__ __noinline__ void dag_source_unpooled(AccArgs<DT> a, AccMem m, AccShared* sh, int s) {
    m.order = m.first;   // the masks are still read
    const size_t row = (size_t)s * a.ld;
    dag_source<DT, STATIC, T, false>(a, m, *sh, s, a.S + row, a.Dl + row);
}

// Re-accumulate source s (whole block; every thread calls it): stage its distance row,
// read DAG'(s) off it, order it by levels, pull Eq. 4 back over them, write the delta row
// (and, statically, the sigma row).  A sum runs in slot order (kBigDag heads or more: by
// rank modulo 32, then a butterfly), so it does not depend on scheduling.
//
// What bounds it: instructions (about 25 per 32 slots of the superset, for every source)
// and two chains of shared-memory reads per level.  Everything after the slots is read
// once lives in shared memory; before, the levels read the superset, its heads and rho
// from L2, three dependent reads per level and direction, around a dozen barriers, now
// one.  Time per source over an update's changed rows, before and now: ER n = 256 (int64)
// 0.50 and 0.21 us, ER n = 4096 0.43 and 0.18, BA n = 8192 0.86 and 0.48, BA n = 16384
// 2.50 and 1.10.  Of the cycles of one source at ER n = 4096, 24 % go to the slots, 13 %
// to the heads, 36 % to the levels forwards, 20 % to the pull.  Measured and not kept:
// no order at all, each thread looking through its open vertices in sweeps until their
// heads are finished (0.22 at ER n = 4096); a thread per vertex instead of a lane per
// slot to read the DAG off (0.29: four dependent L2 reads per 256 vertices, and the hubs
// of a BA graph in the same few warps).
template <typename DT, bool STATIC, int T, bool SM>
__device__ __forceinline__ void dev_accum_source(const AccArgs<DT>& a, int s, const AccMem& m, AccShared& sh) {
    const int n = a.n;
    const int tid = threadIdx.x, lane = tid & 31;
    const DT* Ds = a.D + (size_t)s * a.ld;
    uint64_t* Ss = a.S + (size_t)s * a.ld;
    ff* out = a.Dl + (size_t)s * a.ld;
    int wide = 0;
    for (int t = tid * 4; t < n; t += T * 4) {   // rows start on 32-byte boundaries, np >= t + 4
        uint4 c;
        if constexpr (sizeof(DT) == 4) {
            c = *reinterpret_cast<const uint4*>(Ds + t);
        } else {
            longlong2 v[2];
            v[0] = *reinterpret_cast<const longlong2*>(Ds + t);
            v[1] = *reinterpret_cast<const longlong2*>(Ds + t + 2);
            const long long* vv = reinterpret_cast<const long long*>(v);
            uint32_t* cc = reinterpret_cast<uint32_t*>(&c);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                cc[q] = vv[q] < INT32_MAX ? (uint32_t)vv[q] : (uint32_t)INT32_MAX;
                wide |= vv[q] >= INT32_MAX && vv[q] != Inf<DT>::v;
            }
        }
        *reinterpret_cast<uint4*>(m.row + t) = c;
    }
    if (STATIC) {
        for (int t = tid; t < n; t += T) m.cell[t] = t == s ? 1ull : 0ull;
    } else {
        // the old dependencies are on their way to L2 and the path counts, which the cells
        // start as, here while the DAG is read off
        for (int t = tid * 16; t < n; t += T * 16) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(out + t));
        for (int t = tid * 2; t < n; t += T * 2) {
            if (SM) async_copy16(m.cell + t, Ss + t);
            else *reinterpret_cast<ulonglong2*>(m.cell + t) = *reinterpret_cast<const ulonglong2*>(Ss + t);
        }
        if (SM) async_commit();
    }
    if (tid == 0) sh.arcs = sh.q[0] = 0;
    wide = __syncthreads_or(wide);
    if constexpr (sizeof(DT) == 8) {
        if (wide) dag_slots<DT, T, true>(a, m, Ds, &sh.arcs);
        else dag_slots<DT, T, false>(a, m, Ds, &sh.arcs);
    } else {
        dag_slots<DT, T, false>(a, m, Ds, &sh.arcs);
    }
    __syncthreads();   // the distance row is dead from here on
    for (int t = tid; t < (n + 1) / 2; t += T) m.cnt[t] = 0u;
    const int arcs = sh.arcs;
    __syncthreads();
    if (arcs <= a.lay.pcap)
        for (int q = tid; q < arcs; q += T) cnt_inc(m.cnt, m.pool[q]);
    __syncthreads();   // the lists below mark and copy pool entries
    constexpr int VU = 8;
    unsigned any_huge = 0;
    for (int i0 = 0; i0 * T < n; i0 += VU) {
        int beg[VU], len[VU];
#pragma unroll
        for (int v = 0; v < VU; ++v) {
            const int x = (i0 + v) * T + tid;
            beg[v] = len[v] = 0;
            if (x < n) {
                beg[v] = a.e_off[x];
                len[v] = a.e_len[x];
            }
        }
#pragma unroll
        for (int v = 0; v < VU; ++v) {
            const int x = (i0 + v) * T + tid;
            if ((i0 + v) * T >= n) break;
            int p = 0;
            const int k = count_dag(m, beg[v], len[v], &p);
            if (x < n) {
                m.first[x] = k >= kHugeDag ? kPlaceLater
                             : k > 0       ? place_heads(m, a.lay.pcap, &sh.arcs, beg[v], len[v], k, p)
                                           : (uint16_t)0;
                cnt_mark(m.cnt, x, !STATIC && k == 0);
            }
            const unsigned sinks = __ballot_sync(FULL, k == 0), bigs = __ballot_sync(FULL, k >= kBigDag);
            any_huge |= __ballot_sync(FULL, k >= kHugeDag);
            if (lane == 0 && x < n) {
                m.sink[x >> 5] = sinks;
                m.big[x >> 5] = bigs;
            }
        }
    }
    __syncwarp();
    for (int q = tid >> 5; any_huge && q * 32 < n; q += T / 32)   // the words of big that this warp wrote
        for (uint32_t bb = m.big[q]; bb; bb &= bb - 1u) {
            const int x = 32 * q + __ffs(bb) - 1;
            if (m.first[x] != kPlaceLater) continue;
            const uint16_t first = place_big(m, a.lay.pcap, &sh.arcs, a.e_off[x], a.e_len[x]);
            if (lane == 0) m.first[x] = first;
        }
    if (SM && !STATIC) async_wait_all();
    __syncthreads();
    if (sh.arcs <= a.lay.pcap) dag_source<DT, STATIC, T, true>(a, m, sh, s, Ss, out);
    else dag_source_unpooled<DT, STATIC, T>(a, m, &sh, s);
}

}  // namespace bcg
