// k_batch.cu -- many graphs, one launch per phase.
//
// A batch applies, to each of G graphs, its own list of updates; round r applies the
// r-th update of every graph that has one.  Within a round the phases of an update
// (k_update.cu: Algorithm 4 and the rank-1 pass of Lemma 2 / 4, both directions;
// k_accum.cu: DAG rebuild, Kahn levels, Eq. 4, BC update) run phase by phase over all
// graphs at once: each phase is one persistent kernel whose work is the concatenation
// of every graph's work for that phase, so a 64-vertex graph and a 2048-vertex graph
// share the GPU instead of each getting its own launches.  A task index is mapped to
// its graph by binary search over per-graph prefix offsets; offsets of work that is
// known only on the device (rows that changed) are computed by a one-CTA plan kernel
// just before the phase.  Every per-element, per-item and per-source body is the same
// device function the single-graph kernels call (bc_device.cuh), so a graph's result
// in a batch is bit-identical to its result alone.  The whole multi-round sequence is
// captured once into a CUDA graph and replayed with one graph launch per batch.
#include "bc_batch.cuh"
#include "bc_device.cuh"

namespace bcg {

// ---------------------------------------------------------------- E* writes

__global__ void kb_estar(BatchArgs b, int r) {
    const int64_t o0 = b.eop_off[r], o1 = b.eop_off[r + 1];
    for (int64_t j = o0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < o1;
         j += (int64_t)gridDim.x * blockDim.x) {
        const BatchEOp op = b.eops[j];
        const Dev& d = b.devs[op.g];
        dev_estar_write(op.op, d.e_arc, d.e_w64, d.e_len);
    }
}

// ---------------------------------------------------------------- per-vertex passes

// kind 0: Algorithm 4 forward (IN edges, per source); 1: OUT row test (per source);
// 2: Algorithm 4 on the reverse graph (per target); 3: write row v.
template <typename DT>
__global__ void kb_vertex_pass(BatchArgs b, int r, int kind) {
    const int G = b.G;
    const int64_t* off = b.voff + ((int64_t)r * 4 + kind) * (G + 1);
    const int64_t total = off[G];
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < total;
         j += (int64_t)gridDim.x * blockDim.x) {
        const int g = graph_of(off, G, j);
        const int x = (int)(j - off[g]);
        const Dev& d = b.devs[g];
        if (*d.err) continue;
        const BatchUpd u = b.upd[(int64_t)r * G + g];
        const VEdge* e = b.entries + u.first;
        const DT* D = (const DT*)d.D;
        switch (kind) {
            case 0:
                if (dev_alg4_in<DT>(x, d.ld, D, d.S, u.v, e, u.k, d.directed, (DT*)d.fD, d.fS, d.fM, d.err)) {
                    d.changed[x] = 1u;
                    d.rows[atomicAdd(d.counts, 1)] = x;
                    d.acc_rows[atomicAdd(d.counts + 1, 1)] = x;
                }
                break;
            case 1:
                if (dev_rows_out<DT>(x, d.ld, D, d.S, u.v, e, u.k, d.directed, (DT*)d.fD, d.fS, d.fM, d.err)) {
                    d.rows2[atomicAdd(d.counts + 2, 1)] = x;
                    if (atomicExch(d.changed + x, 1u) == 0u) d.acc_rows[atomicAdd(d.counts + 1, 1)] = x;
                }
                break;
            case 2:
                if (dev_alg4_out<DT>(x, d.ld, D, d.S, u.v, e, u.k, d.directed, (DT*)d.cD, d.cS, d.cM, d.err) &&
                    atomicExch(d.changed + u.v, 1u) == 0u)
                    d.acc_rows[atomicAdd(d.counts + 1, 1)] = u.v;
                break;
            default:
                if (d.pair_on) {
                    // row v is never written before this in an update: its changes are first changes
                    PairRec rec = make_pair_rec(d);
                    rec.first = 1;
                    const size_t i = (size_t)u.v * d.ld + x;
                    if (D[i] != ((const DT*)d.cD)[x] || d.S[i] != d.cS[x])
                        record_change<DT>(rec, u.v, x, D[i], d.S[i]);
                }
                dev_write_row<DT>(x, d.ld, (DT*)d.D, d.S, u.v, (const DT*)d.cD, d.cS, d.err);
        }
    }
}

// ---------------------------------------------------------------- plans

// Per-graph work known only on the device, as exclusive prefix offsets over graphs:
// kind 0: scan items of the phase rows (rows x column chunks); 2: sources to
// re-accumulate; 3: changed rows (and the walks' counters back to zero); 4: column-test weight (and its piece counter back to
// zero).  One CTA.
__global__ void __launch_bounds__(1024) kb_plan(BatchArgs b, int r, int kind, int phase_active, int64_t* out,
                                                int scan_unroll) {
    __shared__ int64_t wsum[32];
    __shared__ int64_t s_total, s_base;
    const int G = b.G, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    for (int g0 = 0; g0 < G; g0 += 1024) {
        const int g = g0 + threadIdx.x;
        int64_t v = 0;
        if (g < G) {
            const Dev& d = b.devs[g];
            const BatchUpd u = b.upd[(int64_t)r * G + g];
            const bool on = (phase_active == 0) ? (u.kin != 0) : (phase_active == 1) ? (u.kout != 0) : (u.present != 0);
            if (on && *d.err == 0) {
                if (kind == 0) {
                    const int cw = kScanThreads * (d.dbytes == 4 ? 4 : 2) * scan_unroll;
                    const int rows = d.counts[phase_active == 0 ? 0 : 2];
                    v = (int64_t)rows * ((d.ld + cw - 1) / cw);
                    atomicAdd(reinterpret_cast<unsigned long long*>(d.stats + 6), (unsigned long long)rows);
                } else if (kind == 2) {
                    v = acc_list_count(d);
                } else if (kind == 3) {
                    v = d.counts[1];
                } else if (d.pair_on && !update_walks(d, u.k)) {
                    v = d.pair_w[d.counts[5]];
                }
            }
        }
        int64_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            const int64_t x = wsum[lane];
            int64_t ix = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t y = __shfl_up_sync(0xffffffffu, ix, o);
                if (lane >= o) ix += y;
            }
            wsum[lane] = ix - x;
            if (lane == 31) s_total = ix;
        }
        __syncthreads();
        if (g < G) out[g] = s_base + wsum[wid] + incl - v;
        __syncthreads();
        if (threadIdx.x == 0) s_base += s_total;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[G] = s_base;
        if (kind == 4) *b.pctr = 0;
        if (kind == 3)
            for (int k = 0; k < 8; ++k) b.wctl[k] = 0;
    }
}

// ---------------------------------------------------------------- rank-1 pass

template <typename DT>
__device__ __forceinline__ ScanArgs<DT> batch_scan_args(const Dev& d, const BatchUpd& u, int phase) {
    ScanArgs<DT> a;
    a.ld = d.ld;
    a.D = (DT*)d.D;
    a.S = d.S;
    a.rows = d.rows;
    a.count = d.counts;
    a.fD = (const DT*)d.fD;
    a.fS = d.fS;
    a.fM = d.fM;
    a.err = d.err;
    a.stats = d.stats;
    a.tie_rows = 0;
    a.tie_cols = 0;
    a.rec = d.pair_on ? make_pair_rec(d) : PairRec{};
    a.rows2 = nullptr;
    a.count2 = nullptr;
    a.cD2 = nullptr;
    a.cS2 = a.cM2 = nullptr;
    if (phase == 0) {
        a.cD = (const DT*)d.D + (size_t)u.v * d.ld;
        a.cS = d.S + (size_t)u.v * d.ld;
        a.cM = a.cS;
        a.skip_row = -1;
        a.rec.first = 1;   // the IN phase is the first pass of an update that writes pairs
    } else {
        a.cD = (const DT*)d.cD;
        a.cS = d.cS;
        a.cM = d.cM;
        a.rows = d.rows2;
        a.count = d.counts + 2;
        a.skip_row = u.v;
    }
    return a;
}

// U: vectors per thread per item (the item's chunk width); sched 0: a contiguous block of
// items per CTA, 1: items dealt out in turn.
template <typename DT, int U>
__global__ void __launch_bounds__(kScanThreads, 4) kb_scan(BatchArgs b, int r, int phase, const int64_t* off,
                                                           int sched) {
    const int G = b.G;
    const int64_t total = off[G];
    const int64_t per = (total + gridDim.x - 1) / gridDim.x;
    const int64_t it0 = sched ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * per;
    const int64_t it1 = sched ? total : min(total, it0 + per);
    const int64_t step = sched ? (int64_t)gridDim.x : 1;
    constexpr int VN = Vec<DT>::N;
    constexpr int CW = kScanThreads * VN * U;
    int cg = -1, cur = -1, s = -1, nchunks = 1;
    int64_t rd = Inf<DT>::v;
    uint64_t rs = 0, rm = 0;
    int n_changed = 0, n_ties = 0;
    ScanArgs<DT> a{};
    for (int64_t j = it0; j < it1; j += step) {
        int g = cg;
        if (g < 0 || j >= off[g + 1] || j < off[g]) {
            // flush the counters of the previous graph before moving on
            if (cg >= 0) {
                scan_stats(a.stats, n_changed, n_ties);
                n_changed = n_ties = 0;
            }
            g = graph_of(off, G, j);
            cg = g;
            cur = -1;
            const Dev& d = b.devs[g];
            a = batch_scan_args<DT>(d, b.upd[(int64_t)r * G + g], phase);
            nchunks = (d.ld + CW - 1) / CW;
        }
        const int64_t item = j - off[g];
        const int i = (int)(item / nchunks);
        const int c = (int)(item - (int64_t)i * nchunks);
        if (i != cur) {
            cur = i;
            s = a.rows[i];
            rd = (s == a.skip_row) ? Inf<DT>::v : (int64_t)a.fD[s];
            rs = a.fS[s];
            rm = a.fM[s];
        }
        if (rd == Inf<DT>::v) continue;
        dev_scan_item<DT, U>(a, s, rd, rs, rm, c, n_changed, n_ties);
    }
    if (cg >= 0) scan_stats(a.stats, n_changed, n_ties);
    else scan_stats(b.devs[0].stats, 0, 0);
}

// ---------------------------------------------------------------- accumulation

// One source per CTA of T threads (128, 256 or 512: a tile the autotuner picks), held to
// 64 registers so that 1024 threads share an SM.
template <typename DT, int T, bool SM>
__global__ void __launch_bounds__(T, 1024 / T) kb_accum(BatchArgs b, int r, const int64_t* off) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ AccShared sh;
    const int G = b.G;
    const int64_t total = off[G];
    const AccMem m = acc_mem<SM>(b.lay, smem, b.ws + (size_t)blockIdx.x * b.ws_stride);
    for (int64_t j = blockIdx.x; j < total; j += gridDim.x) {
        const int g = graph_of(off, G, j);
        const Dev& d = b.devs[g];
        if (block_err(d.err)) continue;
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
        a.rows = acc_list(d);
        a.count = d.pair_on ? d.counts + 3 : d.counts + 1;
        a.ws = b.ws;
        a.ws_stride = b.ws_stride;
        a.err = d.err;
        a.bcfix = d.bcfix;
        a.lay = b.lay;
        dev_accum_source<DT, false, T, SM>(a, a.rows[j - off[g]], m, sh);
    }
}

// ---------------------------------------------------------------- launches

static inline int nb(int64_t x, int t) { return (int)std::max<int64_t>(1, (x + t - 1) / t); }

template <typename DT>
static void batch_scan(const BatchArgs& b, const BatchLaunch& L, int r, int phase, cudaStream_t st) {
    const int grid = L.nsm * L.scan_ctas;
    switch (L.scan_unroll) {
        case 1: kb_scan<DT, 1><<<grid, kScanThreads, 0, st>>>(b, r, phase, b.plan_scan, L.scan_sched); break;
        case 2: kb_scan<DT, 2><<<grid, kScanThreads, 0, st>>>(b, r, phase, b.plan_scan, L.scan_sched); break;
        case 8: kb_scan<DT, 8><<<grid, kScanThreads, 0, st>>>(b, r, phase, b.plan_scan, L.scan_sched); break;
        default: kb_scan<DT, 4><<<grid, kScanThreads, 0, st>>>(b, r, phase, b.plan_scan, L.scan_sched); break;
    }
}

template <typename DT, int T>
static void batch_accum(const BatchArgs& b, const BatchLaunch& L, int r, cudaStream_t st) {
    if (acc_all_smem(b.lay)) kb_accum<DT, T, true><<<L.acc_grid, T, b.lay.smem, st>>>(b, r, b.plan_acc);
    else kb_accum<DT, T, false><<<L.acc_grid, T, b.lay.smem, st>>>(b, r, b.plan_acc);
}

template <typename DT, int T>
static int batch_accum_occupancy(const AccLayout& l) {
    int per_sm = 1;
    auto occ = [&](auto kern) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kAccSmemMax);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, T, l.smem);
    };
    if (acc_all_smem(l)) occ(kb_accum<DT, T, true>);
    else occ(kb_accum<DT, T, false>);
    return std::max(per_sm, 1);
}

template <typename DT>
static void round_launches(const BatchArgs& b, const BatchLaunch& L, int r, cudaStream_t st) {
    const int nsm = L.nsm;
    kb_estar<<<nb(L.max_eops, 256), 256, 0, st>>>(b, r);
    // IN phase
    kb_vertex_pass<DT><<<nsm * L.vpass_ctas, 256, 0, st>>>(b, r, 0);
    kb_plan<<<1, 1024, 0, st>>>(b, r, 0, 0, b.plan_scan, L.scan_unroll);
    batch_scan<DT>(b, L, r, 0, st);
    // OUT phase (graphs without out-edges in this round have no work)
    kb_vertex_pass<DT><<<nsm * L.vpass_ctas, 256, 0, st>>>(b, r, 2);
    kb_vertex_pass<DT><<<nsm * L.vpass_ctas, 256, 0, st>>>(b, r, 1);
    kb_plan<<<1, 1024, 0, st>>>(b, r, 0, 1, b.plan_scan, L.scan_unroll);
    batch_scan<DT>(b, L, r, 1, st);
    kb_vertex_pass<DT><<<nsm * L.vpass_ctas, 256, 0, st>>>(b, r, 3);
    // the changed rows re-accumulated; in graphs with pair corrections only those over the
    // target cap, and the others corrected pair by pair after
    kb_plan<<<1, 1024, 0, st>>>(b, r, 3, 2, b.plan_pr, L.scan_unroll);
    if (L.pairs & 1) batch_pair_plan(b, L, r, sizeof(DT), st);
    if (L.pairs & 2) batch_walk_class(b, L, r, st);
    kb_plan<<<1, 1024, 0, st>>>(b, r, 2, 2, b.plan_acc, L.scan_unroll);
    // (disjoint dependency rows, the rest of the state only read: a branch each of the
    // captured graph.  A call of 8 rounds so and in one branch: 96 graphs of n < 2048 4.41 and
    // 4.70 ms, 512 graphs 22.8 and 23.4, 24 graphs of n < 4000 with vertex updates 3.36 and 3.91)
    cudaEventRecord(L.fork, st);
    cudaStreamWaitEvent(L.side, L.fork, 0);
    if (L.acc_threads == 128) batch_accum<DT, 128>(b, L, r, L.side);
    else if (L.acc_threads == 256) batch_accum<DT, 256>(b, L, r, L.side);
    else batch_accum<DT, 512>(b, L, r, L.side);
    cudaEventRecord(L.join, L.side);
    if (L.pairs & 1) batch_pair_launches(b, L, r, sizeof(DT), st);
    if (L.pairs & 2) batch_walk_launches(b, L, r, sizeof(DT), st);
    cudaStreamWaitEvent(st, L.join, 0);
    batch_round_end(b, L, r, st);
}

// (round_launches, and the kernels of batch_pair_plan, batch_pair_launches, batch_walk_class,
// batch_walk_launches and batch_round_end in it.)
int batch_round_kernels(const BatchLaunch& L) { return 14 + (L.pairs & 1 ? 4 : 0) + (L.pairs & 2 ? 4 : 0); }

void batch_plan(const BatchArgs& b, int r, int kind, int phase_active, int64_t* out, int scan_unroll,
                cudaStream_t st) {
    kb_plan<<<1, 1024, 0, st>>>(b, r, kind, phase_active, out, scan_unroll);
}

// One layout for all graphs of the batch, sized for the largest.
void batch_config(BatchLaunch& L, int dbytes, int n_max, int64_t cap_max) {
    L.lay = acc_layout(n_max, cap_max, false);
    if (L.acc_threads != 128 && L.acc_threads != 256 && L.acc_threads != 512) L.acc_threads = 256;
    auto occ = [&](auto dt) {
        using DT = decltype(dt);
        if (L.acc_threads == 128) return batch_accum_occupancy<DT, 128>(L.lay);
        if (L.acc_threads == 256) return batch_accum_occupancy<DT, 256>(L.lay);
        return batch_accum_occupancy<DT, 512>(L.lay);
    };
    int per_sm = dbytes == 4 ? occ(int32_t{}) : occ(int64_t{});
    if (L.acc_per_sm > 0) per_sm = std::min(per_sm, L.acc_per_sm);
    L.acc_grid = L.nsm * per_sm;
    L.ws_stride = (L.lay.ws + 3) / 4;
}

__global__ void kb_errors(BatchArgs b) {
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < b.G; g += gridDim.x * blockDim.x) b.errs[g] = *b.devs[g].err;
}

void batch_launch_rounds(const BatchArgs& b, const BatchLaunch& L, int rounds, int dbytes, cudaStream_t st) {
    for (int r = 0; r < rounds; ++r) {
        if (dbytes == 4) round_launches<int32_t>(b, L, r, st);
        else round_launches<int64_t>(b, L, r, st);
    }
    kb_errors<<<nb(b.G, 256), 256, 0, st>>>(b);
}

}  // namespace bcg
