// k_accum.cu -- dependency accumulation and the BC reduction.
//
// For each source s whose row changed (and, in the static computation, for every s):
//   * DAG'(s) is rebuilt implicitly: an arc (a,b) of the E* superset is in DAG'(s)
//     iff d'(s,a) is finite and d'(s,a) + w(a,b) = d'(s,b) (Eq. 1; Algorithm 6 step 4
//     applied to E'; Section 6 notes any superset of E* gives the same DAGs).
//   * A topological order of DAG'(s) is built level by level (Kahn): in-degrees are
//     counted first, then a vertex joins level L+1 when its last in-arc from level L
//     is consumed.  Section 2 notes that any reverse topological order serves
//     Algorithm 1 as well as the order by distance; level order keeps the sequential
//     chain as short as the DAG is deep.  In the static computation the same sweep
//     carries the path counts forward (sigma_sb = sum of sigma_sa over DAG in-arcs,
//     Algorithm 6 step 7).
//   * delta_s. is pulled in reverse level order (Eq. 4), in float-float (ff.cuh):
//         delta(a) = sum over DAG out-arcs (a,b) of sigma_sa / sigma_sb * (1 + delta(b))
//                  = sigma_sa * sum over the same arcs of rho(b),
//     with rho(b) = (1 + delta(b)) / sigma_sb kept per vertex, a thread per vertex (a warp
//     for kBigDag DAG out-arcs or more), in slot order: the result does not depend on
//     scheduling.
// The kernel keeps in shared memory the source's distance row, then what it read off it:
// the heads of the DAG arcs, the levels and a cell per vertex (sigma, then rho); see
// dev_accum_source.
//
// BC is maintained as BC += sum over changed rows of (delta'_s - delta_s) (Algorithm 3
// step 1 recomputes BC from zero; rows that did not change contribute the same amount
// before and after, so only changed rows are touched): as an entry of delta_s is written,
// its change goes to BC's fixed-point change of the update (bc_fix_change), which
// k_update_end folds into the compensated (hi, lo) pair.  Summing the old and the new rows
// by columns instead took four launches and read every changed row twice (ER n = 4096,
// 8 updates: 0.33 of 3.6 ms; ER n = 256, 16 updates: 0.31 of 0.98 ms).  The static
// computation sums the columns in row blocks, in a fixed order.
#include <algorithm>
#include <type_traits>

#include "bc_device.cuh"

namespace bcg {

// One CTA per source at a time.
template <typename DT, bool STATIC, int T, bool SM>
__global__ void __launch_bounds__(T, 1024 / T) k_accum(AccArgs<DT> a) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ AccShared sh;
    const AccMem m = acc_mem<SM>(a.lay, smem, a.ws + (size_t)blockIdx.x * a.ws_stride);
    const int total = STATIC ? a.n : *a.count;
    for (int i = blockIdx.x; i < total; i += gridDim.x) {
        if (block_err(a.err)) return;
        dev_accum_source<DT, STATIC, T, SM>(a, STATIC ? i : a.rows[i], m, sh);
    }
}

// partial[rb][t] = sum over the rows of row block rb of Dl[s][t] (t != s), in increasing
// order, in float-float (all terms are non-negative), two adjacent columns per thread:
// 16-byte loads, eight rows' loads issued before they are added.
constexpr int kBcUnroll = 8;
__global__ void __launch_bounds__(256) k_bc_partial(int n, int ld, const ff* Dl, ff* partial,
                                                    const int32_t* err) {
    pdl_enter();
    if (*err) return;
    const int t = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int total = n;
    if (t >= ld) return;
    for (int rb = blockIdx.y; rb * kRowsPerBlock < total; rb += gridDim.y) {
        const int r0 = rb * kRowsPerBlock;
        const int r1 = min(total, r0 + kRowsPerBlock);
        ff a0{0.0f, 0.0f}, a1{0.0f, 0.0f};
        for (int r = r0; r < r1; r += kBcUnroll) {
            int sr[kBcUnroll];
            float4 v[kBcUnroll];
#pragma unroll
            for (int k = 0; k < kBcUnroll; ++k) sr[k] = r + k < r1 ? r + k : -1;
#pragma unroll
            for (int k = 0; k < kBcUnroll; ++k)
                if (sr[k] >= 0) v[k] = __ldcs(reinterpret_cast<const float4*>(Dl + (size_t)sr[k] * ld + t));
#pragma unroll
            for (int k = 0; k < kBcUnroll; ++k) {
                if (sr[k] < 0) break;
                if (sr[k] != t) a0 = ff_add(a0, ff{v[k].x, v[k].y});
                if (sr[k] != t + 1) a1 = ff_add(a1, ff{v[k].z, v[k].w});
            }
        }
        partial[(size_t)rb * ld + t] = a0;
        partial[(size_t)rb * ld + t + 1] = a1;
    }
}

// bc (hi, lo) = the sum of the row-block partials in block order.
__global__ void k_bc_finish(int n, int ld, const ff* partial, double* hi, double* lo, const int32_t* err) {
    pdl_enter();
    if (*err) return;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int nrb = (n + kRowsPerBlock - 1) / kRowsPerBlock;
    ff acc{0.0f, 0.0f};
    for (int rb = 0; rb < nrb; ++rb) acc = ff_add(acc, partial[(size_t)rb * ld + t]);
    hi[t] = ff_to_double(acc);
    lo[t] = 0.0;
}

// ------------------------------------------------------------------ launches

template <typename DT>
static AccArgs<DT> acc_args(const Dev& d, int is_static, const int32_t* rows, const int32_t* count) {
    AccArgs<DT> a;
    a.n = d.n;
    a.ld = d.ld;
    a.D = (const DT*)d.D;
    a.S = d.S;
    a.Dl = d.Dl;
    a.e_off = d.e_off;
    a.e_len = d.e_len;
    a.e_arc = d.e_arc;
    a.e_w64 = d.e_w64;
    a.e_used = group_slots(d.e_used);
    a.rows = rows;
    a.count = count;
    a.ws = d.ws;
    a.ws_stride = d.ws_stride;
    a.err = d.err;
    a.bcfix = d.bcfix;
    a.lay = d.acc_lay[is_static];
    return a;
}

// The cells (8 bytes per vertex, the largest array) stay in shared memory while two CTAs
// fit an SM with them: past that (n above ~5500) they go to the work space, in L2, and
// more threads per SM pay for it (BA n = 8192, every changed row: 0.48 us per row with
// two CTAs of 512 threads and the cells in L2, 0.54 with one of 1024 and the cells here).
constexpr int32_t kAccCellSmem = 100 * 1024;

AccLayout acc_layout(int n, int64_t e_cap, bool is_static) {
    AccLayout l{};
    const int64_t np = ((int64_t)n + 31) & ~(int64_t)31, words = group_slots(e_cap) / 32;
    auto up = [](int64_t x) { return (x + 15) & ~(int64_t)15; };
    int64_t sm = 0, ws = 0;
    auto place = [&](int32_t& off, uint8_t& in_ws, int64_t bytes, int64_t limit) {
        in_ws = sm + up(bytes) > limit;
        int64_t& at = in_ws ? ws : sm;
        off = (int32_t)at;
        at += up(bytes);
    };
    uint8_t no = 0;
    l.pcap = (int32_t)std::min<int64_t>(65532, 7 * np / 4);
    place(l.row, no, 4 * np, kAccSmemMax);
    l.cnt = (int32_t)(l.row + 2 * np);
    place(l.level, no, 2 * kNearLevels, kAccSmemMax);
    place(l.far, no, 2 * (np + 1), 0);
    place(l.sink, no, np / 8, kAccSmemMax);
    place(l.big, no, np / 8, kAccSmemMax);
    place(l.mask, l.mask_ws, std::max(6 * words, 2 * np), kAccSmemMax);
    l.base = (int32_t)(l.mask + 4 * words);
    place(l.pool, l.pool_ws, 2 * (int64_t)(l.pcap + 4), kAccSmemMax);
    place(l.cell, l.cell_ws, 8 * np, kAccCellSmem);
    l.all_smem = !(l.mask_ws || l.pool_ws || l.cell_ws);
    l.smem = (int32_t)sm;
    l.ws = (int32_t)ws;
    return l;
}

template <typename DT, bool STATIC, int T>
static int accum_occupancy(const AccLayout& l) {
    int per_sm = 1;
    if (acc_all_smem(l)) {
        cudaFuncSetAttribute(k_accum<DT, STATIC, T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAccSmemMax);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_accum<DT, STATIC, T, true>, T, l.smem);
    } else {
        cudaFuncSetAttribute(k_accum<DT, STATIC, T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAccSmemMax);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_accum<DT, STATIC, T, false>, T, l.smem);
    }
    return std::max(per_sm, 1);
}

// Calls f with the thread count as a type; the counts an accumulation CTA is built for.
template <typename F>
static auto with_threads(int threads, F&& f) {
    if (threads == 256) return f(std::integral_constant<int, 256>{});
    if (threads == 512) return f(std::integral_constant<int, 512>{});
    return f(std::integral_constant<int, kAccThreadsWide>{});
}

// Threads of a CTA by how many CTAs' shared memory fits an SM, so that an SM has about
// 1024 (us per row when every changed row is re-accumulated, with 256 / 512 / 1024
// threads: ER n = 1024 0.122 / 0.152 / 0.233, ER n = 4096 0.183 / 0.203 / 0.305, BA
// n = 8192 0.583 / 0.478 / 0.602, BA n = 16384 1.83 / 1.29 / 1.10; static n = 16384
// 140 / 130 / 126 ms).
static int acc_threads_for(const AccLayout& l) {
    const int ctas = (227 * 1024) / (l.smem + 1088);
    return ctas >= 3 ? 256 : ctas == 2 ? 512 : kAccThreadsWide;
}

void accum_config(Dev& d) {
    const int n = std::max(d.n, 1);
    d.acc_ctas = 0;
    d.ws_stride = 0;
    for (int k = 0; k < 2; ++k) {
        d.acc_lay[k] = acc_layout(d.n, d.e_cap, k == 1);
        d.acc_threads[k] = acc_threads_for(d.acc_lay[k]);
        auto grid = [&](int threads) {
            return std::min(n, d.nsm * with_threads(threads, [&](auto t) {
                constexpr int T = decltype(t)::value;
                const AccLayout& l = d.acc_lay[k];
                if (d.dbytes == 4) return k ? accum_occupancy<int32_t, true, T>(l) : accum_occupancy<int32_t, false, T>(l);
                return k ? accum_occupancy<int64_t, true, T>(l) : accum_occupancy<int64_t, false, T>(l);
            }));
        };
        d.acc_grid[k] = grid(d.acc_threads[k]);
        d.acc_grid_wide[k] = grid(kAccThreadsWide);
        d.acc_ctas = std::max({d.acc_ctas, d.acc_grid[k], d.acc_grid_wide[k]});
        d.ws_stride = std::max<int64_t>(d.ws_stride, (d.acc_lay[k].ws + 15) / 16 * 4);
    }
    d.acc_wide = d.n >= kAccWideMinN && !d.acc_narrow_only;
}

// Algorithm 1 for the sources listed in rows[0..*count), or for every source.
template <typename DT, bool STATIC>
static void accum_t(const Dev& d, bool wide, const int32_t* rows, const int32_t* count) {
    const AccArgs<DT> a = acc_args<DT>(d, STATIC, rows, count);
    const int grid = wide ? d.acc_grid_wide[STATIC] : d.acc_grid[STATIC];
    with_threads(wide ? kAccThreadsWide : d.acc_threads[STATIC], [&](auto t) {
        constexpr int T = decltype(t)::value;
        if (acc_all_smem(a.lay)) launch_k(k_accum<DT, STATIC, T, true>, grid, T, a.lay.smem, d.st, a);
        else launch_k(k_accum<DT, STATIC, T, false>, grid, T, a.lay.smem, d.st, a);
    });
}

// The wide CTAs serve a partial wave of sources (the rows over the target cap of an
// update with pair corrections: tens per update), where one source's latency is the time.
// Every changed row of an update without pair corrections (thousands of sources) and the
// static computation are served faster by more sources per SM.
static void accum(const Dev& d, int is_static, const int32_t* rows, const int32_t* count) {
    const bool wide = d.acc_wide && !is_static && d.pair_on != 0;
    if (d.dbytes == 4) {
        if (is_static) accum_t<int32_t, true>(d, wide, rows, count);
        else accum_t<int32_t, false>(d, wide, rows, count);
    } else {
        if (is_static) accum_t<int64_t, true>(d, wide, rows, count);
        else accum_t<int64_t, false>(d, wide, rows, count);
    }
}

void launch_accum(const Dev& d, int is_static) { accum(d, is_static, d.acc_rows, d.counts + 1); }

void launch_accum_rows(const Dev& d, const int32_t* rows, const int32_t* count) { accum(d, 0, rows, count); }

// BC of the static computation: the column sums of all rows.  The row blocks go to
// gridDim.y CTAs per column block in turn, about eight CTAs per SM in all.
void launch_bc_static(const Dev& d) {
    const int tb = (d.n + 255) / 256, tb2 = (d.ld / 2 + 255) / 256;
    launch_k(k_bc_partial, dim3(tb2, std::max(1, std::min(d.nrb_max, d.nsm * 8 / tb2))), 256, 0, d.st, d.n, d.ld, d.Dl,
             d.partial, d.err);
    launch_k(k_bc_finish, tb, 256, 0, d.st, d.n, d.ld, d.partial, d.bc_hi, d.bc_lo, d.err);
}

}  // namespace bcg
