// unweight.cu -- event unweighting on the GPU (Sec. "Unweighting and file output").
//
// Maximum weight with a bounded over-weight share: w_max(eps) is the smallest t >= 0 with
//     sum_b max(0, w_b - t) <= eps * sum_b w_b.
// The excess is continuous and decreasing in t.  Non-negative doubles order like their bit
// patterns, so the root is located on them, in three stages:
//   - one pass over the weights (k_partials) takes their sum, maximum and a histogram of counts by exponent and
//     two fraction bits (of one weight in eight of a long list: counting all of them in shared memory costs as
//     much as reading them twice).  A bucket's weights are at least its lower edge, so the counts bound the
//     excess at every edge from below: the highest edge T0 whose bound exceeds 1.5 eps S is taken to lie below
//     the root (the first radix pass sees whether it does, and starts again from 0 in all weights if not);
//   - a second pass (k_gather) lists the weights >= T0, the tail that decides the root (1% of the weights of a
//     2->4 sample at eps = 1e-3).  A tail longer than the workspace's list is searched in the weights themselves;
//   - a radix search over the bits of t in [T0, max], up to 256 buckets a pass (k_pass): count and sum of the
//     weights per bucket, and the last block to finish keeps the bucket in which the excess crosses eps S (the
//     excess at a bucket's lower edge T follows from the counts and sums of all weights >= T).  The search
//     stops when the kept bucket holds no weight (or is one bit pattern wide); then no weight lies strictly
//     between the root and the bucket's upper edge, and w_max = (A - eps S) / K in closed form, A and K the
//     sum and count of the weights above.  At most 8 passes (9 with a new start); those after the last return at
//     once.
// What bounds it: one read of the weights from HBM and one from L2, and the FP64 pipe in the first (one add per
// weight, 19 us per 1e7; the maximum and the tests are integer).  1e7 weights, eps = 1e-3: 685 us as eight
// passes over all weights with per-block histograms combined by one block, 140 us now; where the tail outgrows the
// list, eps = 1e-2: 771 -> 216 us, 0.6: 760 -> 532 us (852 with one load in flight a thread and two blocks an SM).
//
// The bucket sums are exact integers: a weight m 2^(e-1075) (53-bit significand m, exponent
// field e) enters its bucket as m 2^(e-E) in units of 2^(E-1075), E the exponent field of the
// bucket's largest bit pattern, accumulated in two 64-bit limbs of 32 bits.  Integer addition does not
// depend on order, so the result is reproducible bit for bit; the truncation of the
// low bits of weights below the bucket's top binade costs at most one unit of 2^(E-1075) per
// weight (relative 2^-48 of a bucket sum spanning up to 16 binades).  The total sum and the
// maximum are per-block partials over a fixed grid, combined in block order.
//
// Accept/reject: event b is kept iff u_b w_max < w_b, u_b the first uniform of the generator's
// Philox point of event (event_offset + b) in stream 0x556E7700; kept events carry max(w_b, w_max)
// and are written in increasing event order: one pass decides (one bit per event and the block counts), one
// scan, and one pass writes from the bits.  The decision is taken in FP32 with bounds on both sides and in
// FP64 only where they leave it open (1e-6 of the events): in FP64 alone the product and the comparison bound
// the pass.  1e7 weights, 41% kept: 156 us (two FP64 passes over the weights) -> 78 us, now bound by Philox (70% of the
// issue slots in the deciding pass).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <string>

#include "philox.cuh"
#include "ps.h"

namespace ps {
void count_launches(int n);
namespace uw {

constexpr int kGrid = 512;          // blocks of the reductions and histograms (fixed: reproducible sums)
constexpr int kThreads = 256;
constexpr int kBuckets = 256;
constexpr int kPasses = 9;
// Lists from this length on are counted by a sample, one weight in kUnroll: counted in full, 5e6 weights take as long
// and 1e7 at eps = 1e-2 286 us instead of 215; sampled from 2^18 on, 3e5 wide (sigma 1.5) weights at 1e-2, whose first edge
// a sample of 4e4 misses, take 101 us instead of 78.
constexpr int64_t kSampleFrom = 1 << 20;
constexpr int kUnroll = 8;          // loads in flight per thread
constexpr int kCoarseShift = 50;    // the counting histogram: exponent and two fraction bits
constexpr int kCoarse = 1 << (63 - kCoarseShift);
constexpr int kPassGrid = 304;       // two blocks per SM, and twice as many from kSampleFrom weights on
constexpr int kPassUnroll = 4;      // loads in flight per thread of a radix pass
// Weights of the tail list, at most 8 MiB of the workspace.  2^18: 3e7 log-normal weights at eps = 1e-3 430 us instead
// of 252; 2^22, 32 MiB: 1e7 at 1e-2 181 us instead of 215, the others the same.
constexpr int64_t kListMax = 1 << 20;
constexpr int kSelPerThread = 8;    // events per thread in the select kernels
constexpr int kSelBlock = kThreads * kSelPerThread;
constexpr uint32_t kStream = 0x556E7700u;

struct State {
    unsigned long long lo, hi;          // current bit range of the root, [lo, hi)
    int shift;                          // the bucket digit of the next pass: bits shift .. shift+7
    int compact;                        // the weights >= the first lo are listed
    int guess;                          // the first lo is taken from the counts, and not yet confirmed
    double S, target, wmax;
    double carry_sum;                   // sum and count of the weights >= hi
    unsigned long long carry_cnt;
    unsigned long long invalid;
    double t;                           // the result once done
    int done;
    unsigned long long n_list;          // weights for the list (it holds no more than its length of them)
    unsigned int ticket;                // blocks of the running kernel that have finished
};

// finite and non-negative, decided on the bit pattern (sign clear, exponent field not all ones)
// (on the high word: a 64-bit pattern test becomes a floating-point class test on the FP64 pipe)
__device__ __forceinline__ bool valid_bits(unsigned long long u) { return static_cast<unsigned>(u >> 32) < 0x7FF00000u; }
__device__ __forceinline__ bool valid(double w) {
    return static_cast<unsigned>(__double2hiint(w)) < 0x7FF00000u;
}

// exponent field of the largest bit pattern of bucket j (the bucket's fixed-point unit)
__device__ __forceinline__ int bucket_exp(unsigned long long lo, unsigned long long step, unsigned long long hi, int j) {
    unsigned long long top = lo + static_cast<unsigned long long>(j + 1) * step;  // wraps to 0 only at 2^64
    if (top == 0 || top > hi) top = hi;
    return static_cast<int>((top - 1) >> 52);
}

// significand of a non-negative finite double scaled to units of 2^(E-1075)
// (subnormals have the unit of exponent field 1; a bucket of subnormals only uses that unit)
__device__ __forceinline__ unsigned long long fixed_units(unsigned long long u, int E) {
    const int e = static_cast<int>(u >> 52);
    const unsigned long long m = (u & 0xFFFFFFFFFFFFFULL) | (e > 0 ? (1ULL << 52) : 0ULL);
    const int sh = (E > 0 ? E : 1) - (e > 0 ? e : 1);
    return sh >= 64 ? 0ULL : (m >> sh);
}

// Whether this block is the last of the grid to get here, its own and the others' writes before it visible.
__device__ __forceinline__ bool last_block(unsigned int* ticket, bool* flag) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) *flag = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (*flag) __threadfence();
    return *flag;
}

// zero the counters that the kernels below add into
__global__ void __launch_bounds__(256) k_zero(State* st, unsigned int* coarse, unsigned long long* sums) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < kCoarse) coarse[i] = 0;
    if (i < 3 * kBuckets) sums[i] = 0;
    if (i == 0) {
        State s{};
        *st = s;
    }
}

// Per-block partials of sum, max and the number of invalid (negative or non-finite) weights, and the counts by
// leading bits; the last block combines the partials in a fixed-order tree and sets the first range.
__global__ void __launch_bounds__(kThreads) k_partials(const double* w, int64_t n, double eps, double* part,
                                                       unsigned int* coarse, unsigned int list_max, State* st) {
    __shared__ double ss[kGrid], sm[kGrid], sb[kGrid];
    __shared__ unsigned int sc[kCoarse + kCoarse / 32];
    __shared__ bool is_last;
    const int tid = threadIdx.x;
    for (int i = tid; i < kCoarse; i += kThreads) sc[i] = 0;
    __syncthreads();
    const int64_t chunk = (n + kGrid - 1) / kGrid;
    const int64_t b0 = blockIdx.x * chunk, b1 = min(n, b0 + chunk);
    double s = 0.0;
    unsigned long long m = 0;  // the maximum as bits: +0 and above order like them
    unsigned int bad = 0;
    for (int64_t base = b0 + tid; base < b1; base += kUnroll * kThreads) {
        unsigned long long u[kUnroll];
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) {
            const int64_t i = base + k * kThreads;
            u[k] = i < b1 ? static_cast<unsigned long long>(__double_as_longlong(w[i])) : 0ULL;
        }
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) {
            const bool in = base + k * kThreads < b1;
            if (in && valid_bits(u[k])) {
                s += __longlong_as_double(static_cast<long long>(u[k]));
                m = max(m, u[k]);
                if (k == 0 || n < kSampleFrom) atomicAdd(&sc[u[k] >> kCoarseShift], 1u);
            } else if (in) {
                ++bad;
            }
        }
    }
    ss[tid] = s;
    sm[tid] = __longlong_as_double(static_cast<long long>(m));
    sb[tid] = static_cast<double>(bad);
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (tid < o) {
            ss[tid] += ss[tid + o];
            sm[tid] = fmax(sm[tid], sm[tid + o]);
            sb[tid] += sb[tid + o];
        }
        __syncthreads();
    }
    if (tid == 0) {
        part[3 * blockIdx.x] = ss[0];
        part[3 * blockIdx.x + 1] = sm[0];
        part[3 * blockIdx.x + 2] = sb[0];
    }
    for (int i = tid; i < kCoarse; i += kThreads)
        if (sc[i]) atomicAdd(&coarse[i], sc[i]);
    if (!last_block(&st->ticket, &is_last)) return;

    for (int i = tid; i < kGrid; i += kThreads) {
        ss[i] = __ldcg(part + 3 * i);
        sm[i] = __ldcg(part + 3 * i + 1);
        sb[i] = __ldcg(part + 3 * i + 2);
    }
    __syncthreads();
    for (int o = kGrid / 2; o > 0; o >>= 1) {
        for (int i = tid; i < o; i += kThreads) {
            ss[i] += ss[i + o];
            sm[i] = fmax(sm[i], sm[i + o]);
            sb[i] += sb[i + o];
        }
        __syncthreads();
    }
    const double S = ss[0], wmax = sm[0], n_bad = sb[0], target = eps * S;
    __syncthreads();  // ss and sm are used again below
    // The excess at lower edge j is at least sum_{k >= j} cnt_k (edge_k - edge_j) = A_j - K_j edge_j (A, K the
    // suffix sums of cnt_k edge_k and cnt_k).  Each thread takes the suffix over its slice of buckets, the
    // slices above are added, and the highest edge above the target wins.
    const double scale = n < kSampleFrom ? 1.0 : static_cast<double>(kUnroll);
    constexpr int kPer = kCoarse / kThreads;
    double* sa = ss;
    unsigned long long* sk = reinterpret_cast<unsigned long long*>(sm);
    __shared__ int best;
    auto edge = [](int j) { return __longlong_as_double(static_cast<long long>(j) << kCoarseShift); };
    // (one word of padding per 32: a thread walks its slice of 32 buckets, and unpadded the lanes of a warp shared one bank)
    auto at = [](int j) { return j + (j >> 5); };
    for (int i = tid; i < kCoarse; i += kThreads) sc[at(i)] = __ldcg(coarse + i);
    if (tid == 0) best = 0;
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5;
    double A = 0.0;
    unsigned long long K = 0;
    for (int j = kPer - 1; j >= 0; --j)
        if (const unsigned int c = sc[at(tid * kPer + j)]) {
            A += static_cast<double>(c) * edge(tid * kPer + j);
            K += c;
        }
    const double A0 = A;
    const unsigned long long K0 = K;
    for (int o = 1; o < 32; o <<= 1) {  // suffix sums: within the warp, then the warps above
        const double a = __shfl_down_sync(0xffffffffu, A, o);
        const unsigned long long k = __shfl_down_sync(0xffffffffu, K, o);
        if (lane + o < 32) {
            A += a;
            K += k;
        }
    }
    if (lane == 0) {
        sa[warp] = A;
        sk[warp] = K;
    }
    __syncthreads();
    for (int k = kThreads / 32 - 1; k > warp; --k) {
        A += sa[k];
        K += sk[k];
    }
    // (the bound needs no more than a few digits: subtracting the own slice again costs roundings only)
    A -= A0;
    K -= K0;
    const unsigned long long K_above = K;
    for (int j = kPer - 1; j >= 0; --j) {
        const int b = tid * kPer + j;
        const unsigned int c = sc[at(b)];
        if (c == 0) continue;
        const double T = edge(b);
        A += static_cast<double>(c) * T;
        K += c;
        // (1.5: with 1.05 a sampled edge lies above the root more often, 2e6 wide weights at eps = 1e-2 143 us instead of
        // 87; with 3 the tails are longer, 1e7 log-normal ones at 1e-3 158 us instead of 140)
        if (scale * (A - T * static_cast<double>(K)) > 1.5 * target) {
            atomicMax(&best, b);
            break;
        }
    }
    __syncthreads();
    // weights at or above the chosen edge
    if (tid == best / kPer) {
        K = K_above;
        for (int j = kPer - 1; j >= best % kPer; --j) K += sc[at(tid * kPer + j)];
        State x{};
        x.S = S;
        x.wmax = wmax;
        x.invalid = static_cast<unsigned long long>(n_bad);
        x.target = target;
        x.lo = static_cast<unsigned long long>(best) << kCoarseShift;
        x.hi = static_cast<unsigned long long>(__double_as_longlong(wmax)) + 1;
        x.shift = max(0, 56 - __clzll(static_cast<long long>(x.hi - x.lo)));  // at most 256 buckets cover the range
        x.compact = scale * static_cast<double>(K) <= 0.75 * list_max;  // a quarter for the sample's error
        x.guess = 1;
        if (S == 0.0 || x.target >= S) {  // nothing to keep above: every weight is below w_max = 0
            x.t = 0.0;
            x.done = 1;
        } else if (!(eps > 0.0)) {
            x.t = wmax;
            x.done = 1;
        }
        *st = x;  // ticket 0 again
    }
}

// the weights >= the first lower edge into the list (their order does not matter: the sums are exact), staged in
// shared memory: one addition to the list's length per block and kUnroll kThreads weights
__global__ void __launch_bounds__(kThreads) k_gather(const double* w, int64_t n, State* st, unsigned long long* list,
                                                     unsigned int list_max) {
    __shared__ unsigned long long buf[kUnroll * kThreads];
    __shared__ unsigned int cnt;
    __shared__ unsigned long long at;
    if (st->done || !st->compact) return;
    const unsigned long long lo = st->lo;
    const int tid = threadIdx.x, lane = tid & 31;
    constexpr int kSpan = kUnroll * kThreads;
    if (tid == 0) cnt = 0;
    __syncthreads();
    for (int64_t base = blockIdx.x * static_cast<int64_t>(kSpan); base < n; base += static_cast<int64_t>(gridDim.x) * kSpan) {
        unsigned long long u[kUnroll];
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) {
            const int64_t i = base + k * kThreads + tid;
            u[k] = i < n ? static_cast<unsigned long long>(__double_as_longlong(w[i])) : ~0ULL;
        }
#pragma unroll
        for (int k = 0; k < kUnroll; ++k) {
            const bool in = valid_bits(u[k]) && u[k] >= lo;
            const unsigned mask = __ballot_sync(0xffffffffu, in);
            if (mask == 0) continue;
            unsigned p = 0;
            if (lane == 0) p = atomicAdd(&cnt, static_cast<unsigned>(__popc(mask)));
            p = __shfl_sync(0xffffffffu, p, 0) + __popc(mask & ((1u << lane) - 1u));
            if (in) buf[p] = u[k];
        }
        __syncthreads();
        if (tid == 0) at = cnt ? atomicAdd(&st->n_list, static_cast<unsigned long long>(cnt)) : 0;
        __syncthreads();
        const unsigned m = cnt;
        const unsigned long long a = at;
        for (unsigned i = tid; i < m; i += kThreads)
            if (a + i < list_max) list[a + i] = buf[i];
        __syncthreads();
        if (tid == 0) cnt = 0;
        __syncthreads();
    }
}

// One radix pass: count and exact sum per bucket of [lo, hi) over the list or the weights, added into sums[]
// (limbs of 32 bits and counts), and the last block chooses the bucket holding the root.
__global__ void __launch_bounds__(kThreads) k_pass(const double* w, int64_t n, const unsigned long long* list,
                                                   unsigned int list_max, State* st, unsigned long long* sums) {
    // warp-private histograms: no contention between warps on a crowded bucket
    __shared__ unsigned long long s0[kThreads / 32][kBuckets], s1[kThreads / 32][kBuckets];
    __shared__ unsigned int sc[kThreads / 32][kBuckets];
    __shared__ int sexp[kBuckets];
    __shared__ bool is_last;
    if (st->done) return;
    const unsigned long long lo = st->lo, hi = st->hi;
    const int shift = st->shift;
    const unsigned long long step = 1ULL << shift;
    const int64_t total = st->compact ? static_cast<int64_t>(min(st->n_list, static_cast<unsigned long long>(list_max))) : n;
    const unsigned long long* src = st->compact ? list : reinterpret_cast<const unsigned long long*>(w);
    const int64_t chunk = (total + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = blockIdx.x * chunk, b1 = min(total, b0 + chunk);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (b0 < b1) {
        sexp[tid] = bucket_exp(lo, step, hi, tid);
        for (int j = tid; j < (kThreads / 32) * kBuckets; j += kThreads) {
            s0[j / kBuckets][j % kBuckets] = 0;
            s1[j / kBuckets][j % kBuckets] = 0;
            sc[j / kBuckets][j % kBuckets] = 0;
        }
        __syncthreads();
        for (int64_t base = b0; base < b1; base += kPassUnroll * kThreads) {  // block-uniform trip count (warp collectives)
            unsigned long long us[kPassUnroll];
#pragma unroll
            for (int k = 0; k < kPassUnroll; ++k) {
                const int64_t i = base + k * kThreads + tid;
                us[k] = i < b1 ? __ldcg(src + i) : ~0ULL;
            }
#pragma unroll
            for (int k = 0; k < kPassUnroll; ++k) {
                const unsigned long long u = us[k];
                const bool in = valid_bits(u) && u >= lo && u < hi;
                if (__ballot_sync(0xffffffffu, in) == 0) continue;
                const int bk = in ? static_cast<int>((u - lo) >> shift) : -1;
                const unsigned long long v = in ? fixed_units(u, sexp[bk]) : 0ULL;
                // lanes of one bucket combine first: exact 21-bit limb sums, one leader per bucket
                const unsigned grp = __match_any_sync(0xffffffffu, bk);
                const unsigned l0 = __reduce_add_sync(grp, static_cast<unsigned>(v & 0x1FFFFF));
                const unsigned l1 = __reduce_add_sync(grp, static_cast<unsigned>((v >> 21) & 0x1FFFFF));
                const unsigned l2 = __reduce_add_sync(grp, static_cast<unsigned>(v >> 42));
                if (in && lane == __ffs(grp) - 1) {
                    // l0 + l1 2^21 + l2 2^42 in limbs of 32 bits (l2 below 2^16)
                    const unsigned long long t = static_cast<unsigned long long>(l0) + (static_cast<unsigned long long>(l1) << 21);
                    // one leader per bucket in this warp and the histogram private to the warp: plain
                    // read-modify-write, no atomics
                    s0[warp][bk] += t & 0xFFFFFFFFULL;
                    s1[warp][bk] += (t >> 32) + (static_cast<unsigned long long>(l2) << 10);
                    sc[warp][bk] += static_cast<unsigned>(__popc(grp));
                }
                __syncwarp();
            }
        }
        __syncthreads();
        unsigned long long t0 = 0, t1 = 0, c = 0;
        for (int k = 0; k < kThreads / 32; ++k) {
            t0 += s0[k][tid];
            t1 += s1[k][tid];
            c += sc[k][tid];
        }
        if (c) {
            atomicAdd(&sums[tid], t0);
            atomicAdd(&sums[kBuckets + tid], t1);
            atomicAdd(&sums[2 * kBuckets + tid], c);
        }
    }
    if (!last_block(&st->ticket, &is_last)) return;

    // suffix sums over the buckets (256 threads: shuffles within a warp, then the warps above), in a fixed order
    double* ws = reinterpret_cast<double*>(s0[0]);
    unsigned long long* wc = s1[0];
    double* cs = reinterpret_cast<double*>(s0[1]);
    unsigned long long* cc = s1[1];
    __shared__ int best;
    State x = *st;
    double v;
    unsigned long long c;
    {
        const unsigned long long l = __ldcg(sums + tid), h = __ldcg(sums + kBuckets + tid);
        c = __ldcg(sums + 2 * kBuckets + tid);
        // the value (h 2^32 + l) 2^(E - 1075), as high and low 64-bit words
        const unsigned long long low = l + (h << 32), high = (h >> 32) + (low < l ? 1ULL : 0ULL);
        const int E = bucket_exp(lo, step, hi, tid);
        v = ldexp(static_cast<double>(high) * 18446744073709551616.0 + static_cast<double>(low), (E > 0 ? E : 1) - 1075);
        sums[tid] = sums[kBuckets + tid] = sums[2 * kBuckets + tid] = 0;  // for the next pass
    }
    const unsigned long long own = c;
    for (int o = 1; o < 32; o <<= 1) {
        const double a = __shfl_down_sync(0xffffffffu, v, o);
        const unsigned long long b = __shfl_down_sync(0xffffffffu, c, o);
        if (lane + o < 32) {
            v += a;
            c += b;
        }
    }
    if (tid == 0) best = 0;
    if (lane == 0) {
        ws[warp] = v;
        wc[warp] = c;
    }
    __syncthreads();
    double above = x.carry_sum;
    unsigned long long above_c = x.carry_cnt;
    for (int k = kThreads / 32 - 1; k > warp; --k) {
        above += ws[k];
        above_c += wc[k];
    }
    v += above;
    c += above_c;
    cs[tid] = v;
    cc[tid] = c;
    const unsigned long long edge = lo + static_cast<unsigned long long>(tid) * step;
    if (edge < hi && v - __longlong_as_double(static_cast<long long>(edge)) * static_cast<double>(c) > x.target)
        atomicMax(&best, tid);
    __syncthreads();
    const int sel = best;  // no crossing within rounding: the lowest bucket
    if (tid != sel) return;
    x.ticket = 0;
    if (x.guess) {
        // the guessed edge (its own excess not above the target) or the list (cut short, also from 0 on: the sample sees
        // few weights where it meets invalid ones) was wrong: from 0, in all weights
        x.guess = 0;
        const double T = __longlong_as_double(static_cast<long long>(lo));
        const bool cut = x.compact && x.n_list > list_max;
        if (cut || (lo > 0 && !(cs[0] - T * static_cast<double>(cc[0]) > x.target))) {
            x.compact = 0;
            x.lo = 0;
            x.shift = max(0, 56 - __clzll(static_cast<long long>(x.hi)));
            *st = x;
            return;
        }
    }
    // the carry of the next pass: weights >= the kept bucket's upper edge
    const double cum_s = sel + 1 < kBuckets ? cs[sel + 1] : x.carry_sum;
    const unsigned long long cum_c = sel + 1 < kBuckets ? cc[sel + 1] : x.carry_cnt;
    const unsigned long long new_lo = x.lo + static_cast<unsigned long long>(sel) * step;
    unsigned long long new_hi = new_lo + step;
    if (new_hi > x.hi) new_hi = x.hi;
    x.lo = new_lo;
    x.hi = new_hi;
    x.carry_sum = cum_s;
    x.carry_cnt = cum_c;
    if (own == 0 || step == 1) {
        // no weight strictly inside (lo, hi): excess(t) = A - t K on [lo, hi]
        double t = cum_c > 0 ? (cum_s - x.target) / static_cast<double>(cum_c) : 0.0;
        const double tlo = __longlong_as_double(static_cast<long long>(x.lo));
        const double thi = __longlong_as_double(static_cast<long long>(x.hi));
        x.t = fmin(fmax(t, tlo), thi);
        x.done = 1;
    }
    x.shift = max(0, shift - 8);
    *st = x;
}

__global__ void k_result(State* st, double* result) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    State x = *st;
    if (!x.done) {  // every pass narrowed the range: lo is the root to the last bit
        x.t = __longlong_as_double(static_cast<long long>(x.lo));
        x.done = 1;
        *st = x;
    }
    result[0] = x.t;
    result[1] = x.S;
    result[2] = x.wmax;
    result[3] = static_cast<double>(x.carry_cnt);
    result[4] = static_cast<double>(x.invalid);
}

// u t < w, u the event's uniform.  t = tf 2^te, tf in [1, 2): in FP32 on w 2^-te, u between its leading 24 bits
// and the next multiple of 2^-24, each bound moved by 2^-20 for the roundings; FP64 where they leave it open.
struct Threshold {
    double t;
    float tf;
    int te;  // exponent field of t, or -1: always FP64 (zero, subnormal or extreme thresholds)
};
__device__ __forceinline__ Threshold threshold(double t) {
    const unsigned hi = static_cast<unsigned>(__double2hiint(t)), lo = static_cast<unsigned>(__double2loint(t));
    const int e = static_cast<int>(hi >> 20);
    return {t, __uint_as_float(0x3F800000u | (__funnelshift_l(lo, hi, 3) & 0x7FFFFFu)), e >= 128 && e < 1920 ? e : -1};
}
__device__ __forceinline__ bool keep(double w, const Threshold& T, uint64_t seed, uint64_t ev) {
    if (!valid(w)) return false;
    const uint4 o = rng::philox4x32_10(make_uint4(static_cast<uint32_t>(ev), static_cast<uint32_t>(ev >> 32), kStream, 0u),
                                       static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32));
    const unsigned hi = static_cast<unsigned>(__double2hiint(w)), lo = static_cast<unsigned>(__double2loint(w));
    const int e = static_cast<int>(hi >> 20) - T.te + 127;  // exponent field of w 2^-te as a float
    if (T.te > 0 && e > 27 && e < 227) {
        const float wf = __uint_as_float((static_cast<unsigned>(e) << 23) | (__funnelshift_l(lo, hi, 3) & 0x7FFFFFu));
        const float u0 = static_cast<float>(o.y >> 8) * 0x1p-24f;
        if (u0 * T.tf > wf * (1.0f + 0x1p-20f)) return false;
        if ((u0 + 0x1p-24f) * T.tf * (1.0f + 0x1p-20f) < wf) return true;
    }
    return rng::unit_from_bits(o.y, o.x) * T.t < w;
}

// One bit per event (word i of bits[]: events 32 i .. 32 i + 31) and the number kept of each block.
__global__ void __launch_bounds__(kThreads) k_count(const double* w, int64_t n, const double* tmax, uint64_t seed,
                                                    uint64_t ev0, unsigned int* bits, long long* counts) {
    __shared__ int sc[kThreads / 32];
    const Threshold T = threshold(*tmax);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t e0 = blockIdx.x * static_cast<int64_t>(kSelBlock) + threadIdx.x;
    double v[kSelPerThread];
#pragma unroll
    for (int k = 0; k < kSelPerThread; ++k) {
        const int64_t e = e0 + k * kThreads;
        v[k] = e < n ? w[e] : -1.0;  // an invalid weight is never kept
    }
    int c = 0;
#pragma unroll
    for (int k = 0; k < kSelPerThread; ++k) {
        const int64_t e = e0 + k * kThreads;
        const unsigned m = __ballot_sync(0xffffffffu, keep(v[k], T, seed, ev0 + static_cast<uint64_t>(e)));
        if (lane == 0) bits[e >> 5] = m;
        c += __popc(m);
    }
    if (lane == 0) sc[warp] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long s = 0;
        for (int k = 0; k < kThreads / 32; ++k) s += sc[k];
        counts[blockIdx.x] = s;
    }
}

// exclusive scan of the block counts (one block), total into n_out
__global__ void __launch_bounds__(1024) k_scan(const long long* counts, int64_t nb, long long* offsets,
                                               int64_t* n_out) {
    __shared__ long long s[1024];
    const int64_t per = (nb + 1023) / 1024;
    const int64_t a = threadIdx.x * per, b = min(nb, a + per);
    long long loc = 0;
    for (int64_t i = a; i < b; ++i) loc += counts[i];
    s[threadIdx.x] = loc;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        long long v = threadIdx.x >= o ? s[threadIdx.x - o] : 0;
        __syncthreads();
        s[threadIdx.x] += v;
        __syncthreads();
    }
    long long run = s[threadIdx.x] - loc;  // exclusive prefix of this thread's segment
    for (int64_t i = a; i < b; ++i) {
        offsets[i] = run;
        run += counts[i];
    }
    if (threadIdx.x == 1023) *n_out = s[1023];
}

// The kept events of a block in order, from its bits: word k of warp r is word 8 k + r of the block.
__global__ void __launch_bounds__(kThreads) k_write(const double* w, const double* tmax, const unsigned int* bits,
                                                    const long long* offsets, int64_t* idx, double* wout) {
    constexpr int kWords = kSelBlock / 32;
    __shared__ unsigned int sm[kWords];
    __shared__ int sp[kWords];
    // max(w, t) on the bits: a kept w is not negative (and no event is kept at a NaN t)
    const long long tb = __double_as_longlong(*tmax);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < kWords) {
        sm[tid] = bits[blockIdx.x * static_cast<int64_t>(kWords) + tid];
        sp[tid] = __popc(sm[tid]);
    }
    __syncthreads();
    if (warp == 0) {  // exclusive prefix over the words, two per lane
        const int a = sp[2 * lane], b = sp[2 * lane + 1];
        int run = a + b;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += v;
        }
        sp[2 * lane] = run - a - b;
        sp[2 * lane + 1] = run - b;
    }
    __syncthreads();
    const long long off = offsets[blockIdx.x];
#pragma unroll
    for (int k = 0; k < kSelPerThread; ++k) {
        const int word = k * (kThreads / 32) + warp;
        const unsigned m = sm[word];
        if (m >> lane & 1u) {
            const int64_t e = blockIdx.x * static_cast<int64_t>(kSelBlock) + word * 32 + lane;
            const long long pos = off + sp[word] + __popc(m & ((1u << lane) - 1u));
            idx[pos] = e;
            wout[pos] = __longlong_as_double(max(__double_as_longlong(w[e]), tb));
        }
    }
}

}  // namespace uw
}  // namespace ps

using namespace ps::uw;

namespace {
thread_local std::string u_err;
int ufail(int code, const std::string& m) {
    u_err = m;
    return code;
}
int ucheck(cudaError_t e, const char* what) {
    if (e == cudaSuccess) return PS_OK;
    return ufail(PS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}
constexpr size_t kStateBytes = 256;
constexpr size_t kPartBytes = sizeof(double) * 3 * kGrid;
constexpr size_t kCoarseBytes = sizeof(unsigned int) * kCoarse;
constexpr size_t kSumBytes = sizeof(unsigned long long) * 3 * kBuckets;
size_t align256(size_t x) { return (x + 255) / 256 * 256; }
int64_t sel_blocks(int64_t n) { return (n + kSelBlock - 1) / kSelBlock; }
int64_t list_len(int64_t n) { return std::max<int64_t>(1, std::min<int64_t>(n, kListMax)); }
size_t max_bytes(int64_t n) {
    return kStateBytes + align256(kPartBytes) + kCoarseBytes + align256(kSumBytes) +
           align256(sizeof(unsigned long long) * static_cast<size_t>(list_len(n)));
}
}  // namespace

extern "C" {

const char* ps_unweight_last_error(void) { return u_err.c_str(); }

int ps_unweight_workspace_size(int64_t n, size_t* bytes) {
    if (n < 0 || !bytes) return ufail(PS_ERR_INVALID_ARGUMENT, "ps_unweight_workspace_size: bad arguments");
    const size_t nb = static_cast<size_t>(std::max<int64_t>(1, sel_blocks(n)));
    const size_t sel = align256(sizeof(long long) * nb) * 2 + align256(nb * (kSelBlock / 8));
    *bytes = max_bytes(n) + sel;
    return PS_OK;
}

int ps_unweight_max(const double* w, int64_t n, double eps, double* result, void* workspace, size_t ws_bytes,
                    void* stream) {
    size_t need = 0;
    if (!result || n < 0 || (n > 0 && !w) || !(eps >= 0.0) || !workspace ||
        ps_unweight_workspace_size(n, &need) != PS_OK || ws_bytes < need ||
        (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
        return ufail(PS_ERR_INVALID_ARGUMENT, "ps_unweight_max: bad arguments or workspace");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char* base = static_cast<char*>(workspace);
    State* state = reinterpret_cast<State*>(base);
    char* at = base + kStateBytes;
    double* part = reinterpret_cast<double*>(at);
    at += align256(kPartBytes);
    unsigned int* coarse = reinterpret_cast<unsigned int*>(at);
    at += kCoarseBytes;
    unsigned long long* sums = reinterpret_cast<unsigned long long*>(at);
    at += align256(kSumBytes);
    unsigned long long* list = reinterpret_cast<unsigned long long*>(at);
    k_zero<<<(kCoarse + 255) / 256, 256, 0, st>>>(state, coarse, sums);
    const unsigned int cap = static_cast<unsigned int>(list_len(n));
    k_partials<<<kGrid, kThreads, 0, st>>>(w, n, eps, part, coarse, cap, state);
    int launches = 3;
    // eps = 0 is the maximum itself, which k_partials has: no search (1e5 weights: 70 us with the search's launches, 65 before
    // there was a list, 28 now)
    if (eps > 0.0) {
        k_gather<<<kGrid, kThreads, 0, st>>>(w, n, state, list, cap);
        // A long list's tail may outgrow the workspace: the passes then read all weights, with four blocks an SM (1e7
        // weights, eps = 0.6: 776 us with two, 532 with four).  A short one's extra blocks only take tickets (1000: 81 and 83 us).
        const int grid = n < kSampleFrom ? kPassGrid : 2 * kPassGrid;
        for (int p = 0; p < kPasses; ++p) k_pass<<<grid, kThreads, 0, st>>>(w, n, list, cap, state, sums);
        launches += 1 + kPasses;
    }
    k_result<<<1, 32, 0, st>>>(state, result);
    ps::count_launches(launches);
    return ucheck(cudaGetLastError(), "ps_unweight_max");
}

int ps_unweight_select(const double* w, int64_t n, const double* w_max, uint64_t seed, uint64_t event_offset,
                       int64_t* idx, double* w_out, int64_t* n_accepted, void* workspace, size_t ws_bytes,
                       void* stream) {
    size_t need = 0;
    if (n < 0 || (n > 0 && (!w || !idx || !w_out)) || !w_max || !n_accepted || !workspace ||
        ps_unweight_workspace_size(n, &need) != PS_OK || ws_bytes < need ||
        (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
        return ufail(PS_ERR_INVALID_ARGUMENT, "ps_unweight_select: bad arguments or workspace");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int64_t nb = sel_blocks(n);
    if (nb == 0) return ucheck(cudaMemsetAsync(n_accepted, 0, sizeof(int64_t), st), "ps_unweight_select");
    char* base = static_cast<char*>(workspace) + max_bytes(n);
    const size_t cb = align256(sizeof(long long) * nb);
    long long* counts = reinterpret_cast<long long*>(base);
    long long* offsets = reinterpret_cast<long long*>(base + cb);
    unsigned int* bits = reinterpret_cast<unsigned int*>(base + 2 * cb);
    k_count<<<static_cast<unsigned>(nb), kThreads, 0, st>>>(w, n, w_max, seed, event_offset, bits, counts);
    k_scan<<<1, 1024, 0, st>>>(counts, nb, offsets, n_accepted);
    k_write<<<static_cast<unsigned>(nb), kThreads, 0, st>>>(w, w_max, bits, offsets, idx, w_out);
    ps::count_launches(3);
    return ucheck(cudaGetLastError(), "ps_unweight_select");
}

}  // extern "C"
