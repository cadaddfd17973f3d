// kernels.cu -- sm_103a kernels of the phase-space library.
//
// ps_map_kernel evaluates the compiled instruction list of a channel (the
// paper's compute graph, Sec. 3.1 / Fig. compute_graph) for one event per
// thread.  All instructions of an event run back to back in that thread: the
// values live in a per-thread slot file in shared memory (slot s of thread t at
// smem[s * block + t], conflict-free), the byte-code, immediates and VEGAS grid
// of the channel are staged in shared memory once per channel change, and only
// the declared outputs (SoA, coalesced) and one partial-sum record per tile of
// `block` events reach global memory.  Tiles of all channels are distributed
// over a persistent grid; tile -> channel is a scan of at most 32 prefix sums
// held in the kernel parameters.
//
// Every branch inside an op depends only on the op's immediates (warp-uniform)
// or is resolved by selects, so the warps of a channel never diverge.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <string>

#include "map_device.cuh"
#include "ps_internal.h"

namespace ps {

static unsigned long long g_launches = 0;


// The interpreter's policy: a channel change stages its byte-code, immediates and VEGAS grid in
// shared memory; an event runs the byte-code on the thread's column of the slot file.
template <bool kMix>
struct InterpPolicy {
    static constexpr bool kTwoJoins = false;  // map_tiles
    const LaunchParams& lp;
    dev::Frame f;
    int32_t* s_code;
    double* s_imm;
    float* s_immf;
    double* s_grid;
    int out_pc;
    __device__ __forceinline__ void stage(int c, const ChannelLaunch& C) {
        const int B = lp.block, tid = threadIdx.x;
        for (int i = tid; i < C.code_len; i += B) s_code[i] = lp.code[C.code_off + i];
        for (int i = tid; i < C.imm_len; i += B) s_imm[i] = lp.imm[C.imm_off + i];
        if (kMix)
            for (int i = tid; i < C.imm_len; i += B) s_immf[i] = static_cast<float>(lp.imm[C.imm_off + i]);
        double* g = s_grid + kTrigDoubles;  // the grid after the azimuth table
        if (kMix) {
            dev::stage_grid(reinterpret_cast<float*>(g), lp.grid + C.grid_off, C.vdims, C.vbins, tid, B);
        } else {
            dev::stage_trig(s_grid, tid, B);
            dev::stage_grid(g, lp.grid + C.grid_off, C.vdims, C.vbins, tid, B);
        }
        __syncthreads();
        out_pc = dev::find_output(s_code, C.code_len);
    }
    __device__ __forceinline__ double event(int c, const ChannelLaunch& C, int64_t ev, int64_t local, bool active) {
        dev::load_inputs<kMix>(f, lp, c, C.n_random, ev, local, active);
        double* g = s_grid + kTrigDoubles;
        if (kMix) dev::run_code_mixed(s_code, out_pc, f, reinterpret_cast<float*>(g), C.vbins, lp.status + 1, active);
        else dev::run_code(s_code, out_pc, f, g, C.vbins, lp.status + 1, active);
        return dev::store_outputs<kMix>(f, s_code + out_pc + 3, s_code[out_pc + 1], lp, C, local, active);
    }
};

template <bool kMix>
__global__ void __launch_bounds__(256) ps_map_kernel(const __grid_constant__ LaunchParams lp) {
    extern __shared__ __align__(16) double smem[];
    const int B = lp.block;
    double* s_imm = smem;
    double* s_grid = s_imm + lp.smem_imm;
    double* s_slots = s_grid + lp.smem_grid;
    double* s_red = s_slots + static_cast<size_t>(lp.smem_slots) * B;
    int32_t* s_code = reinterpret_cast<int32_t*>(s_red + 4 * (B / 32));
    float* s_immf = reinterpret_cast<float*>(s_code + lp.smem_code_ints);  // mixed mode: float immediates
    InterpPolicy<kMix> pol{lp, dev::Frame{s_slots + threadIdx.x, s_imm, B, s_immf}, s_code, s_imm, s_immf, s_grid, 0};
    dev::map_tiles(lp, pol, s_red);
}

// One cluster of eight CTAs per channel sums the channel's tile partials in a fixed order (deterministic: slice by
// rank, thread and unroll step, then fixed trees, the ranks' sums in rank order through distributed shared
// memory); in streaming mode the launch's sums are added to the statistics of the earlier launches.  What bounds it
// is latency, and the FP64 adds of the trees, which one SM issues at one per 16 cycles (so few threads, and the
// maxima on the integer ALU).  One CTA of 1024 threads took 17 us for 782 tiles and 23 us for 7813; 6.5 and 11 us now.
constexpr int kReduceThreads = 128;
constexpr int kReduceUnroll = 4;
constexpr int kReduceRanks = 8;

struct TileSum {
    double n, s, s2;
    unsigned long long m;  // the maximum: +0 and above order like their bits
};
__device__ __forceinline__ void add(TileSum& a, const TileSum& b) {
    a.n += b.n;
    a.s += b.s;
    a.s2 += b.s2;
    a.m = max(a.m, b.m);
}

__global__ void __cluster_dims__(kReduceRanks, 1, 1) __launch_bounds__(kReduceThreads)
    ps_reduce_kernel(const __grid_constant__ LaunchParams lp, double* stats) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int c = blockIdx.x / kReduceRanks, rank = static_cast<int>(cluster.block_rank());
    const ChannelLaunch& C = lp.ch[c];
    const int64_t t0 = C.tile_begin;
    const int64_t t1 = (c + 1 < lp.n_ch) ? lp.ch[c + 1].tile_begin : lp.n_tiles;
    const int64_t len = (t1 - t0 + kReduceRanks - 1) / kReduceRanks;
    const int64_t b0 = min(t1, t0 + rank * len), b1 = min(t1, b0 + len);
    TileSum a[kReduceUnroll];
#pragma unroll
    for (int u = 0; u < kReduceUnroll; ++u) a[u] = {0.0, 0.0, 0.0, 0ULL};
    for (int64_t t = b0 + threadIdx.x; t < b1; t += kReduceUnroll * kReduceThreads) {
        double2 lo[kReduceUnroll], hi[kReduceUnroll];
#pragma unroll
        for (int u = 0; u < kReduceUnroll; ++u) {  // the loads first, then the sums
            const int64_t tu = t + u * kReduceThreads;
            const double2* tp = reinterpret_cast<const double2*>(lp.tile_partials + 4 * tu);
            lo[u] = tu < b1 ? tp[0] : make_double2(0.0, 0.0);
            hi[u] = tu < b1 ? tp[1] : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int u = 0; u < kReduceUnroll; ++u)
            if (t + u * kReduceThreads < b1)
                add(a[u], {lo[u].x, lo[u].y, hi[u].x, static_cast<unsigned long long>(__double_as_longlong(hi[u].y))});
    }
    add(a[0], a[1]);
    add(a[2], a[3]);
    add(a[0], a[2]);
    TileSum v = a[0];
    // a fixed tree within each warp, then the warps of the CTA, then the ranks
    for (int s = 16; s > 0; s >>= 1) {
        TileSum o;
        o.n = __shfl_down_sync(0xffffffffu, v.n, s);
        o.s = __shfl_down_sync(0xffffffffu, v.s, s);
        o.s2 = __shfl_down_sync(0xffffffffu, v.s2, s);
        o.m = __shfl_down_sync(0xffffffffu, v.m, s);
        add(v, o);
    }
    __shared__ TileSum red[kReduceThreads / 32], ranks[kReduceRanks];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    cluster.sync();  // rank 0 has started: its shared memory can be written
    if (threadIdx.x == 0) {
        for (int k = 1; k < kReduceThreads / 32; ++k) add(v, red[k]);
        *cluster.map_shared_rank(&ranks[rank], 0) = v;
    }
    cluster.sync();
    if (rank != 0 || threadIdx.x != 0) return;
    for (int k = 1; k < kReduceRanks; ++k) add(v, ranks[k]);
    const double vmax = __longlong_as_double(static_cast<long long>(v.m));
    double* o = stats + 5 * c;
    if (lp.stats_mode && *lp.stats_mode != 0) {  // streaming: add this launch to the running sums
        o[0] += static_cast<double>(C.n_events);
        o[1] += v.n;
        o[2] += v.s;
        o[3] += v.s2;
        o[4] = fmax(o[4], vmax);
    } else {
        o[0] = static_cast<double>(C.n_events);
        o[1] = v.n;
        o[2] = v.s;
        o[3] = v.s2;
        o[4] = vmax;
    }
}

// ---------------------------------------------------------------- VEGAS training histogram
// The importance sums of VEGAS training, sum of w^2 per (dimension, bin of the unmapped r), for
// every channel of a launch, added in a fixed order so that an adaptation is reproducible bit for
// bit and does not depend on how tiles were scheduled.  A CTA takes one chunk of a channel's events
// (kHistChunks equal slices) and one dimension.  Every thread owns a histogram in shared memory ([bin][thread]: no
// two threads of a warp meet in a bank) and adds the w^2 (from the stored weights) of events t, t + T, t + 2T ...
// of the chunk in that order; the threads' rows are then added in an order fixed by the entry, and the second
// kernel adds a channel's chunks in chunk order.
// Bound: one FP64 add per event and dimension (15 us per 1e6 events x 8), and the latency of a thread's
// read-modify-write chain: 32 KB a CTA at 64 bins keep seven CTAs on an SM.  1e6 events x 8 x 64 bins: 1229 us when
// every thread of 128 CTAs compared every event with its own entries, 88 us with two dimensions to a CTA (three on an
// SM, two waves), 37 us now.
constexpr int kHistThreads = 64;
constexpr int kHistSmem = kHistThreads * 256 * 8;  // the largest grid, 256 bins

// kBits: Philox points and a power of two of bins, so that the bin is the leading bits of r.  A template and not
// a branch: the general bin's product and conversion would be evaluated for every event and selected away.
template <bool kBits>
__device__ __forceinline__ void hist_chunk(const LaunchParams& lp, const ChannelLaunch& C, double* part, int stride,
                                           double* acc) {
    constexpr int T = kHistThreads;
    const int c = blockIdx.z, j = blockIdx.y, k = blockIdx.x, tid = threadIdx.x;
    const int bins = C.vbins;
    for (int i = 0; i < bins; ++i) acc[i * T + tid] = 0.0;
    const int64_t len = (C.n_events + kHistChunks - 1) / kHistChunks;
    const int64_t e0 = min(C.n_events, k * len), e1 = min(C.n_events, e0 + len);
    const bool odd = j & 1;
    const int bits = __ffs(bins) - 1;
    constexpr int kU = 4;                     // events in flight per thread
    auto weight = [&](int64_t e) { return e < e1 ? lp.w[C.col_off + e] : 0.0; };
    double w[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) w[u] = weight(e0 + tid + u * T);
    for (int64_t base = e0 + tid; base < e1; base += kU * T) {
        double w2[kU];
        int b[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            w2[u] = w[u] * w[u];
            w[u] = weight(base + (kU + u) * T);  // the next round's
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t e = min(base + u * T, e1 - 1), ev = C.ev_offset + e;
            uint4 o = make_uint4(0u, 0u, 0u, 0u);
            if (kBits || lp.r == nullptr)
                o = rng::philox4x32_10(make_uint4(static_cast<uint32_t>(ev), static_cast<uint32_t>(ev >> 32),
                                                              static_cast<uint32_t>(c), static_cast<uint32_t>(j >> 1)),
                                                   static_cast<uint32_t>(lp.seed), static_cast<uint32_t>(lp.seed >> 32));
            const uint32_t lead = odd ? o.w : o.y;
            if constexpr (kBits) {
                b[u] = static_cast<int>(__funnelshift_l(lead, 0u, bits));
            } else {
                const double r = lp.r != nullptr ? lp.r[j * lp.ld_r + e] : rng::unit_from_bits(lead, odd ? o.z : o.x);
                b[u] = min(max(static_cast<int>(r * bins), 0), bins - 1);
            }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (base + u * T < e1) acc[b[u] * T + tid] += w2[u];
    }
    __syncthreads();
    double* o = part + (static_cast<int64_t>(c) * kHistChunks + k) * stride + j * bins;
    for (int i = tid; i < bins; i += T) {
        double s = 0.0;  // the rows in the order i, i + 1, ... (mod T): the threads read different banks
#pragma unroll 8
        for (int q = 0; q < T; ++q) s += acc[i * T + ((i + q) & (T - 1))];
        o[i] = s;
    }
}

__global__ void __launch_bounds__(kHistThreads) ps_hist_partial_kernel(const __grid_constant__ LaunchParams lp, double* part,
                                                                       int stride) {
    extern __shared__ __align__(16) double acc[];
    const ChannelLaunch& C = lp.ch[blockIdx.z];
    if (static_cast<int>(blockIdx.y) >= C.vdims) return;
    if (lp.r == nullptr && (C.vbins & (C.vbins - 1)) == 0) hist_chunk<true>(lp, C, part, stride, acc);
    else hist_chunk<false>(lp, C, part, stride, acc);
}

__global__ void __launch_bounds__(kHistReduce) ps_hist_reduce_kernel(const __grid_constant__ LaunchParams lp,
                                                                     const double* part, int stride) {
    const int c = blockIdx.y;
    const ChannelLaunch& C = lp.ch[c];
    const int idx = blockIdx.x * kHistReduce + threadIdx.x;
    if (idx >= C.vdims * C.vbins) return;
    const double* q = part + static_cast<int64_t>(c) * kHistChunks * stride + idx;
    double s = 0.0;
    for (int k0 = 0; k0 < kHistChunks; k0 += 16) {
        double v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = q[static_cast<int64_t>(k0 + k) * stride];  // the loads first
#pragma unroll
        for (int k = 0; k < 16; ++k) s += v[k];
    }
    lp.hist[C.hist_off + idx] += s;
}

size_t smem_bytes_for(const LaunchParams& lp) {
    size_t doubles = static_cast<size_t>(lp.smem_imm) + lp.smem_grid + static_cast<size_t>(lp.smem_slots) * lp.block +
                     4 * (lp.block / 32);
    return doubles * sizeof(double) + static_cast<size_t>(lp.smem_code_ints) * sizeof(int32_t) +
           (lp.mixed ? static_cast<size_t>(lp.smem_imm) * sizeof(float) : 0);
}

static int cuda_fail(cudaError_t e, const char* what, std::string* err) {
    *err = std::string(what) + ": " + cudaGetErrorString(e);
    return PS_ERR_CUDA;
}

int max_ctas_per_sm(int block, size_t smem, int mixed, int* out, std::string* err) {
    const void* fn = mixed ? reinterpret_cast<const void*>(ps_map_kernel<true>)
                           : reinterpret_cast<const void*>(ps_map_kernel<false>);
    // The dynamic shared-memory limit is a per-kernel, per-device setting shared by every program:
    // it only ever grows, so a program created later with a smaller slot file cannot lower the
    // limit below what an earlier program launches with.
    static std::mutex mu;
    static int limit[kMaxDevices][2] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice", err);
    if (dev < 0 || dev >= kMaxDevices) {
        *err = "device index beyond the library's limit";
        return PS_ERR_INVALID_ARGUMENT;
    }
    {
        std::lock_guard<std::mutex> lock(mu);
        int& cur = limit[dev][mixed ? 1 : 0];
        if (static_cast<int>(smem) > cur) {
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
            if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute", err);
            cur = static_cast<int>(smem);
        }
    }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, fn, block, smem);
    if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor", err);
    return PS_OK;
}

int launch_map(const LaunchParams& lp, int grid_ctas, size_t smem, void* stream, std::string* err) {
    if (lp.n_tiles == 0) return PS_OK;
    if (lp.mixed) ps_map_kernel<true><<<grid_ctas, lp.block, smem, static_cast<cudaStream_t>(stream)>>>(lp);
    else ps_map_kernel<false><<<grid_ctas, lp.block, smem, static_cast<cudaStream_t>(stream)>>>(lp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "ps_map_kernel launch", err);
    __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
    return PS_OK;
}

int launch_reduce(const LaunchParams& lp, double* stats, void* stream, std::string* err) {
    ps_reduce_kernel<<<lp.n_ch * kReduceRanks, kReduceThreads, 0, static_cast<cudaStream_t>(stream)>>>(lp, stats);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "ps_reduce_kernel launch", err);
    __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
    return PS_OK;
}

int launch_hist(const LaunchParams& lp, double* part, int stride, void* stream, std::string* err) {
    if (lp.hist == nullptr || stride <= 0) return PS_OK;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    int dims = 0, bins = 0;
    for (int c = 0; c < lp.n_ch; ++c) {
        if (lp.ch[c].vdims == 0) continue;
        dims = std::max(dims, static_cast<int>(lp.ch[c].vdims));
        bins = std::max(bins, static_cast<int>(lp.ch[c].vbins));
    }
    if (dims == 0) return PS_OK;
    cudaError_t e = cudaSuccess;
    {
        // the dynamic shared memory above the default is granted once per device
        static std::mutex mu;
        static bool granted[kMaxDevices] = {};
        std::lock_guard<std::mutex> lock(mu);
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess && dev >= 0 && dev < kMaxDevices && !granted[dev]) {
            e = cudaFuncSetAttribute(ps_hist_partial_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kHistSmem);
            granted[dev] = e == cudaSuccess;
        }
        if (e != cudaSuccess) return cuda_fail(e, "ps_hist_partial_kernel shared memory", err);
    }
    ps_hist_partial_kernel<<<dim3(kHistChunks, dims, lp.n_ch), kHistThreads, sizeof(double) * kHistThreads * bins, cs>>>(
        lp, part, stride);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "ps_hist_partial_kernel launch", err);
    ps_hist_reduce_kernel<<<dim3((stride + kHistReduce - 1) / kHistReduce, lp.n_ch), kHistReduce, 0, cs>>>(lp, part, stride);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "ps_hist_reduce_kernel launch", err);
    __atomic_add_fetch(&g_launches, 2ULL, __ATOMIC_RELAXED);
    return PS_OK;
}

bool is_hist_kernel(const void* func) {
    return func == reinterpret_cast<const void*>(ps_hist_partial_kernel) ||
           func == reinterpret_cast<const void*>(ps_hist_reduce_kernel);
}

// Copies the statistics into host-mapped pinned memory: the read-back of ps_stats uses no copy
// engine, so it does not queue behind large device-to-host copies of event records.
__global__ void __launch_bounds__(256) ps_copy_kernel(double* dst, const double* src, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = src[i];
}

int launch_copy(double* dst, const double* src, int n, void* stream, std::string* err) {
    if (n <= 0) return PS_OK;
    ps_copy_kernel<<<(n + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(dst, src, n);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "ps_copy_kernel launch", err);
    __atomic_add_fetch(&g_launches, 1ULL, __ATOMIC_RELAXED);
    return PS_OK;
}

unsigned long long launch_count() { return __atomic_load_n(&g_launches, __ATOMIC_RELAXED); }
void count_launches(int n) { __atomic_add_fetch(&g_launches, static_cast<unsigned long long>(n), __ATOMIC_RELAXED); }
bool is_reduce_kernel(const void* func) { return func == reinterpret_cast<const void*>(ps_reduce_kernel); }

// ---------------------------------------------------------------- mixed-form helpers
// Elementwise application of one device helper of the map kernels (ps_mixed_helpers).
template <int kKind, class In, class Out>
__global__ void __launch_bounds__(256) ps_mixed_helper_kernel(const In* in, Out* out, int64_t n) {
    for (int64_t i = blockIdx.x * 256LL + threadIdx.x; i < n; i += static_cast<int64_t>(gridDim.x) * 256) {
        if constexpr (kKind == PS_MIXED_F2D) out[i] = dev::mx::f2d(in[i]);
        else if constexpr (kKind == PS_MIXED_D2F) out[i] = dev::mx::d2f(in[i]);
        else if constexpr (kKind == PS_MIXED_SQRT64) out[i] = dev::mx::sqrt64(in[i]);
        else if constexpr (kKind == PS_MIXED_TAN_QUARTER) out[i] = dev::tan_quarter(in[i]);
        else out[i] = dev::mx::rcp64(in[i]);
    }
}

// The FP64 azimuth (ps_mixed_helpers, PS_MIXED_SINCOS_TURN): each CTA stages its table first.
__global__ void __launch_bounds__(256) ps_turn_kernel(const double* in, double* out, int64_t n) {
    __shared__ double t[kTrigDoubles];
    dev::stage_trig(t, threadIdx.x, 256);
    __syncthreads();
    for (int64_t i = blockIdx.x * 256LL + threadIdx.x; i < n; i += static_cast<int64_t>(gridDim.x) * 256) {
        double s, c;
        dev::sincos_turn(in[i], t, s, c);
        out[2 * i] = c;
        out[2 * i + 1] = s;
    }
}

// ---------------------------------------------------------------- allocation-free scratch
// Fixed scratch for ps_generate_noalloc: kNoallocTiles per-tile partial-sum records (4 doubles
// each, 4 MiB) in a file-scope device array.  Every device that loads the library holds it until
// the process exits.  Host code must not hand the symbol itself to a kernel (on the host it is
// only a stand-in); its device address is fetched once per device with cudaGetSymbolAddress.
static __device__ __align__(256) double g_noalloc_scratch[static_cast<size_t>(kNoallocTiles) * 4];

namespace {
std::mutex g_noalloc_mutex;
void* g_noalloc_ptr[kMaxDevices] = {};
}  // namespace

int noalloc_scratch(int device, void** ptr, size_t* bytes, std::string* err) {
    if (device < 0 || device >= kMaxDevices) {
        *err = "device index beyond the library's limit";
        return PS_ERR_INVALID_ARGUMENT;
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (g_noalloc_ptr[device] == nullptr) {
        // set-up: the calling thread has `device` current (the caller guarantees it)
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(noalloc scratch)", err);
        g_noalloc_ptr[device] = p;
    }
    *ptr = g_noalloc_ptr[device];
    *bytes = sizeof(g_noalloc_scratch);
    return PS_OK;
}

}  // namespace ps

extern "C" int ps_mixed_helpers(int kind, const void* in, void* out, int64_t n, void* stream) {
    using namespace ps;
    if (n < 0 || (n > 0 && (in == nullptr || out == nullptr))) return PS_ERR_INVALID_ARGUMENT;
    if (kind < PS_MIXED_F2D || kind > PS_MIXED_TAN_QUARTER) return PS_ERR_INVALID_ARGUMENT;
    if (n == 0) return PS_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, 152LL * 16);
    const int g = static_cast<int>(blocks);
    switch (kind) {
        case PS_MIXED_F2D:
            ps_mixed_helper_kernel<PS_MIXED_F2D><<<g, 256, 0, s>>>(static_cast<const float*>(in), static_cast<double*>(out), n);
            break;
        case PS_MIXED_D2F:
            ps_mixed_helper_kernel<PS_MIXED_D2F><<<g, 256, 0, s>>>(static_cast<const double*>(in), static_cast<float*>(out), n);
            break;
        case PS_MIXED_SQRT64:
            ps_mixed_helper_kernel<PS_MIXED_SQRT64><<<g, 256, 0, s>>>(static_cast<const double*>(in), static_cast<double*>(out), n);
            break;
        case PS_MIXED_RCP64:
            ps_mixed_helper_kernel<PS_MIXED_RCP64><<<g, 256, 0, s>>>(static_cast<const double*>(in), static_cast<double*>(out), n);
            break;
        case PS_MIXED_TAN_QUARTER:
            ps_mixed_helper_kernel<PS_MIXED_TAN_QUARTER><<<g, 256, 0, s>>>(static_cast<const double*>(in), static_cast<double*>(out), n);
            break;
        default:
            ps_turn_kernel<<<g, 256, 0, s>>>(static_cast<const double*>(in), static_cast<double*>(out), n);
            break;
    }
    if (cudaGetLastError() != cudaSuccess) return PS_ERR_CUDA;
    count_launches(1);
    return PS_OK;
}
