// k_noalloc.cu -- static betweenness of a small graph without any device allocation.
//
// Some callers cannot call cudaMalloc: a process whose device memory is owned by a
// framework's caching allocator or a serving runtime that reserves HBM up front and
// forbids further allocation (cudaMalloc may synchronise the device and stall other
// streams), or code that must not allocate once it has started.  For them
// bc_static_scores_noalloc runs the same static computation as bc_init_static --
// all-pairs distances, path counts, Algorithm 1 per source, BC as column sums -- on a
// graph the caller already holds in device memory, and writes the scores to a device
// buffer the caller provides.  Its scratch (the n x n state, packed arcs, work space)
// is one file-scope __device__ array of kScratchBytes, present on every GPU that loads
// the library until the process exits; it caps the graph at kMaxN vertices and
// kMaxArcs arcs.  Every arc of the graph is used as the superset of E* (any superset
// gives the same DAGs), so no host round trip is needed.
#include <mutex>

#include "bcgpu.h"
#include "bc_internal.cuh"

namespace bcg {

namespace {

constexpr int32_t kMaxN = 512;
constexpr int64_t kMaxArcs = 32768;
constexpr int kMaxDevices = 64;

// Byte offsets into the scratch array (every piece 256-byte aligned).
constexpr size_t al(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr size_t kOffD = 0;
constexpr size_t kOffS = kOffD + al((size_t)kMaxN * kMaxN * 8);
constexpr size_t kOffDl = kOffS + al((size_t)kMaxN * kMaxN * 8);
constexpr size_t kOffHi = kOffDl + al((size_t)kMaxN * kMaxN * sizeof(ff));
constexpr size_t kOffLo = kOffHi + al((size_t)kMaxN * 8);
constexpr size_t kSlots = (size_t)kMaxArcs;
static_assert(kSlots % kGroupSlots == 0, "whole groups of slots");
constexpr size_t kOffArc = kOffLo + al((size_t)kMaxN * 8);
constexpr size_t kOffW64 = kOffArc + al(kSlots * sizeof(Arc));
constexpr size_t kOffLen = kOffW64 + al(kSlots * 8);
constexpr size_t kOffPart = kOffLen + al((size_t)kMaxN * 4);
constexpr size_t kOffErr = kOffPart + al((size_t)((kMaxN + kRowsPerBlock - 1) / kRowsPerBlock) * kMaxN * sizeof(ff));
constexpr size_t kOffCnt = kOffErr + 256;
constexpr size_t kOffStats = kOffCnt + 256;
constexpr size_t kOffWs = kOffStats + 256;
constexpr size_t kWsBytes = (size_t)4 << 20;
constexpr size_t kScratchBytes = kOffWs + kWsBytes;

}  // namespace

// The scratch itself.  Host code must not use this name as an address: it is only a
// host-side stand-in for the symbol; the device address comes from
// cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

namespace {

std::mutex g_mu;
unsigned char* g_addr[kMaxDevices] = {};

// Device address of the scratch on the current device, looked up once per device.
cudaError_t scratch_address(unsigned char** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess) return e;
        g_addr[dev] = static_cast<unsigned char*>(p);
    }
    *out = g_addr[dev];
    return cudaSuccess;
}

// Pack the caller's CSR into the slot format of the accumulation (every arc a slot),
// and check each arc: endpoints in range, no self-loop, weight in [1, INF-1].  The offsets
// cover every slot (0 first, the number of arcs last, none smaller than the one before):
// the search goes over all of them, and one left out would hold an earlier call's arc.
// The slots past the arcs, up to a whole group, are empty.  A thread per slot, its tail found
// in the offsets by bisection: a thread per vertex took 34 us for BA n = 512 (8150 arcs) and
// 76 us for the complete graph of 181 (32580), this takes 2.8 and 2.6.
template <typename DT>
__global__ void k_pack_graph(int n, int64_t arcs, unsigned long long* count, const int32_t* off, const int32_t* dst, const int64_t* w,
                             Arc* arc, int64_t* w64, int32_t* len, int32_t* err) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        *count = (unsigned long long)arcs;
        if (off[0] != 0 || off[n] != arcs) set_err(err, ERRF_ARG_DEVICE);
    }
    if (i < n) {
        const int32_t a = off[i], b = off[i + 1];
        const bool ok = a >= 0 && b >= a && b <= arcs;
        len[i] = ok ? b - a : 0;
        if (!ok) set_err(err, ERRF_ARG_DEVICE);
    }
    if (i < arcs) {
        const int32_t b = dst[i];
        const int64_t x = w[i];
        int lo = 0, hi = n;   // the last vertex below hi whose arcs start at or before i, or 0
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (off[mid] <= i) lo = mid;
            else hi = mid;
        }
        if (b < 0 || b >= n || b == lo || x < 1 || x >= Inf<DT>::v) set_err(err, ERRF_ARG_DEVICE);
        arc[i] = make_arc(lo, b, x);
        if (sizeof(DT) == 8) w64[i] = x;
    } else if (i < group_slots(arcs)) {
        arc[i] = empty_arc();
    }
}

__global__ void k_scores_out(int n, const double* hi, const double* lo, double f, double* out, const int32_t* err) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n || *err) return;
    out[t] = (hi[t] + lo[t]) * f;
}

}  // namespace
}  // namespace bcg

using namespace bcg;

extern "C" int bc_static_scores_noalloc(int32_t n, int64_t arcs, const int32_t* d_off, const int32_t* d_dst,
                                        const int64_t* d_w, uint32_t flags, double* d_scores, void* cuda_stream) {
    const bool dir = (flags & BC_DIRECTED) != 0, und = (flags & BC_UNDIRECTED) != 0;
    const bool i32 = (flags & BC_DIST_I32) != 0, i64 = (flags & BC_DIST_I64) != 0;
    if (dir == und || i32 == i64) return BC_ERR_ARG;
    if (n < 1 || n > kMaxN || arcs < 0 || arcs > kMaxArcs) return BC_ERR_ARG;
    if (!d_off || !d_scores || (arcs > 0 && (!d_dst || !d_w))) return BC_ERR_ARG;
    unsigned char* base = nullptr;
    if (scratch_address(&base) != cudaSuccess) return BC_ERR_CUDA;
    Dev d{};
    d.n = n;
    d.ld = row_pitch(n);
    d.dbytes = i32 ? 4 : 8;
    d.directed = dir ? 1 : 0;
    d.st = (cudaStream_t)cuda_stream;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&d.nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return BC_ERR_CUDA;
    d.D = base + kOffD;
    d.S = reinterpret_cast<uint64_t*>(base + kOffS);
    d.Dl = reinterpret_cast<ff*>(base + kOffDl);
    d.bc_hi = reinterpret_cast<double*>(base + kOffHi);
    d.bc_lo = reinterpret_cast<double*>(base + kOffLo);
    d.g_arcs = arcs;
    d.e_off = const_cast<int32_t*>(d_off);
    d.e_len = reinterpret_cast<int32_t*>(base + kOffLen);
    d.e_arc = reinterpret_cast<Arc*>(base + kOffArc);
    d.e_w64 = i64 ? reinterpret_cast<int64_t*>(base + kOffW64) : nullptr;
    d.e_cap = d.e_used = arcs;
    d.g_arc = d.e_arc;
    d.g_w64 = d.e_w64;
    d.g_off = d.e_off;
    d.err = reinterpret_cast<int32_t*>(base + kOffErr);
    d.counts = reinterpret_cast<int32_t*>(base + kOffCnt);
    d.stats = reinterpret_cast<int64_t*>(base + kOffStats);
    d.g_count = reinterpret_cast<unsigned long long*>(base + kOffStats + 128);
    d.partial = reinterpret_cast<ff*>(base + kOffPart);
    d.nrb_max = (n + kRowsPerBlock - 1) / kRowsPerBlock;
    accum_config(d);
    if ((size_t)d.acc_ctas * (size_t)d.ws_stride * sizeof(int32_t) > kWsBytes) return BC_ERR_ARG;   // not for n <= kMaxN
    d.ws = reinterpret_cast<int32_t*>(base + kOffWs);
    // the error word and counters start at zero on every call (the scratch keeps the
    // previous call's contents)
    if (cudaMemsetAsync(d.err, 0, 256 * 3, d.st) != cudaSuccess) return BC_ERR_CUDA;
    const int blocks = (int)((std::max<int64_t>(n, group_slots(arcs)) + 255) / 256);
    if (d.dbytes == 4)
        k_pack_graph<int32_t><<<blocks, 256, 0, d.st>>>(n, arcs, d.g_count, d_off, d_dst, d_w, d.e_arc, d.e_w64, d.e_len, d.err);
    else
        k_pack_graph<int64_t><<<blocks, 256, 0, d.st>>>(n, arcs, d.g_count, d_off, d_dst, d_w, d.e_arc, d.e_w64, d.e_len, d.err);
    launch_sssp(d, 0, true);
    launch_accum(d, 1);
    launch_bc_static(d);
    k_scores_out<<<(n + 255) / 256, 256, 0, d.st>>>(n, d.bc_hi, d.bc_lo, dir ? 1.0 : 0.5, d_scores, d.err);
    if (cudaGetLastError() != cudaSuccess) return BC_ERR_CUDA;
    int32_t h_err = 0;
    if (cudaMemcpyAsync(&h_err, d.err, sizeof(int32_t), cudaMemcpyDeviceToHost, d.st) != cudaSuccess ||
        cudaStreamSynchronize(d.st) != cudaSuccess)
        return BC_ERR_CUDA;
    if (h_err & ERRF_ARG_DEVICE) return BC_ERR_ARG;
    if (h_err & ERRF_OVERFLOW) return BC_ERR_OVERFLOW;
    if (h_err & ERRF_DIST) return BC_ERR_DIST_OVERFLOW;
    if (h_err & ERRF_TIMEOUT) return BC_ERR_TIMEOUT;
    return BC_OK;
}
