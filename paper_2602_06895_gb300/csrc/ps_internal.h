// ps_internal.h -- structures shared by the host compiler (graph.cpp) and the
// device interpreter (kernels.cu) of the GB300 phase-space library.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include "launch_params.h"
#include "ps.h"

namespace ps {

constexpr int kMaxOutMomenta = 24;
constexpr int kNoallocTiles = 131072;  // tiles of the allocation-free entry point's fixed scratch
constexpr int kMaxDevices = 64;
// VEGAS training histogram (kernels.cu): chunks per channel, threads that add them, and the largest
// grid it takes (dimensions x bins <= kHistMaxEntries, bins <= 256)
// (Fixed, since the order of the sums depends on it.  A chunk costs a CTA of 64 threads a dimension, seven on an SM: 112
// chunks of 8 dimensions are one wave.  1e6 events x 8 dimensions, kernels and sum: 64 chunks 56 us, 112 49, 128 66, 224
// 66; x 1 dimension 55, 39, 39, 34; 1000 events x 8: 20, 24, 30, 39.)
constexpr int kHistChunks = 112;
constexpr int kHistReduce = 64;
constexpr int kHistMaxEntries = 4096;
constexpr int kHistMaxDims = 64;

// ---------------------------------------------------------------- graph IR
struct Arg {
    int kind;  // PS_ARG_VALUE / PS_ARG_IMM
    int id;
    double imm;
};

struct Instr {
    int op;
    std::vector<Arg> args;
    std::vector<int> outs;  // value ids
};

struct Graph {
    int n_random = 0;
    std::vector<int> type;  // value id -> PS_TYPE_*
    std::vector<Instr> code;
    std::vector<int> out_ids, out_roles;
    bool outputs_set = false;
};

// ---------------------------------------------------------------- compiled channel
// Byte-code: per instruction [op, n_args, n_out, args..., outs...]; an argument >= 0 is a
// slot index (momenta occupy 4 consecutive slots), < 0 encodes immediate ~arg.  The code
// ends with [kOpOutput, n, 0, (role, slot) x n].
struct Compiled {
    std::vector<int32_t> code;
    std::vector<double> imm;
    int n_slots = 0;
    int n_random = 0;
    int vegas_dims = 0;  // dims of the VEGAS op (0 if none)
    int n_momenta_out = 0;
    bool has_x1 = false, has_x2 = false, has_alpha = false;
};

// derive: constants of the channel (map_nu's logarithm of a constant range) go along as extra arguments
int compile_graph(const Graph& g, Compiled* out, std::string* err, bool derive);

// ---------------------------------------------------------------- inverse map plan
// Everything the inverse kernel needs about one channel, flattened on the host from its
// ps_channel_desc (the same layout, bounds recipe and propagators as the forward builder).
constexpr int kInvNodes = 32, kInvLegs = 10, kInvIds = 512, kInvProps = 40;
struct InvNode {
    int32_t kind, nch, leaf;
    int32_t child[kInvLegs];
    uint32_t mask;       // leaf-index bit mask of the subtree
    double mass, M, G, nu;
};
struct InvPlan {
    int32_t n, n_nodes, hadronic, lab_frame, kappa, n_sorder, n_pre, d, vdims, vbins;
    double S, sqrt_s, a, shat_M, shat_G, shat_nu, t_nu, ts_nu, mleaf;
    int32_t sorder[kInvNodes], pre[kInvNodes];
    int32_t d_shat, d_x, d_s[kInvNodes], d_ts[kInvLegs + 1], d_tt[kInvLegs + 1], d_tphi[kInvLegs + 1];
    int32_t d_dphi[kInvNodes], d_dth[kInvNodes];
    int32_t order[kInvLegs + 2], side[kInvLegs + 1];
    // s-order step i: m_min = lo_c + sum sqrt(s_id) over ids[lo_beg[i] .. off_beg[i]),
    // m_max = m_top - (off_c + sum sqrt(s_id) over ids[off_beg[i] .. lo_beg[i+1])),
    // m_top = sqrt(s_top) (sqrt_s for the root at fixed energy)
    double lo_c[kInvNodes], off_c[kInvNodes];
    int32_t top[kInvNodes], lo_beg[kInvNodes + 1], off_beg[kInvNodes + 1];
    int32_t ids[kInvIds];
    // propagators of the channel's SDE weight P(p): kind 0 s-channel (mask, M, G), 1 t-channel
    int32_t n_prop, pkind[kInvProps];
    uint32_t pmask[kInvProps];
    double pM[kInvProps], pG[kInvProps];
    InvNode node[kInvNodes];
};
int build_inverse_plan(const ps_channel_desc* d, InvPlan* plan, std::string* err);

// kernels.cu
int launch_map(const LaunchParams& lp, int grid_ctas, size_t smem_bytes, void* stream, std::string* err);
int launch_reduce(const LaunchParams& lp, double* stats_dev, void* stream, std::string* err);
int launch_copy(double* dst, const double* src, int n, void* stream, std::string* err);
// The VEGAS training histogram of a launch whose weights are stored (lp.hist non-null): partial
// sums per (channel, chunk) into part [n_ch][kHistChunks][stride], then added in a fixed order.
int launch_hist(const LaunchParams& lp, double* part, int stride, void* stream, std::string* err);
bool is_hist_kernel(const void* func);
void count_launches(int n);

// Compiled programs (jit.cpp): the CUDA source of a program, NVRTC to a cubin (host only), the
// cached kernel on the current device, its occupancy and its launch.
// min_blocks > 0: the kernel is compiled so that that many CTAs of `block` threads fit on an SM
// (launch bounds; the split form's channel units get the matching register cap).
std::string jit_source(const std::vector<Compiled>& ch, int block, int min_blocks, bool mixed, int tiles);
// Tiles a CTA of a compiled program runs side by side: several for a split mixed program that is asked to fit four CTAs
// or more on an SM, as long as two CTAs and 256 threads remain.  Such a program's code is straight-line and long (24
// 2->8 channels: ~10^4 instructions an event each), instruction fetch bounds it, and neighbouring tiles, mostly of one
// channel, share what they fetch: 128 threads x 4 CTAs took 5.1 ms per 2^22 2->8 events, 2 x 128 threads x 2 CTAs, with
// the same registers and warps, 4.22 ms (64 x 8: 7.6 and 4.20 ms; 9728 events: 80 and 74 us).  A program in one unit
// gains nothing (six 2->5 channels, 128 x 4: 6e6 events 4.23 ms with two tiles, 4.19 with one, 38912 events 79 and 65 us).
// Two CTAs of 128 threads, 8 warps an SM, gain nothing either (2->8: 6.12 and 6.20 ms).
// The CTAs an SM is to hold: those requested; when none are, for a split mixed program, as many as hold 512 threads
// at 128 registers (2->8 at 128 threads: 6.25 ms with the registers the compiler takes, 4.29 ms with 128).  A
// program in one unit does better with the compiler's own choice (2->5: 4.09 ms against 4.32 ms capped; three 2->8
// channels, 2^21 events: 2.12 against 2.29 ms).
int jit_min_blocks(size_t n_ch, bool mixed, int block, int ctas_per_sm);
int jit_cta_tiles(size_t n_ch, bool mixed, int block, int min_blocks, int smem_grid);
int jit_compile(const std::string& src, std::vector<char>* cubin, std::string* log, bool relocatable, int max_regs);
// Programs of more channels than these are compiled one unit per channel, in parallel, and linked: one
// unit of all channels compiles in time that grows faster than the channel count.  FP64 units are
// longer (six 2->5 channels: 14.5 s as one unit, 2.3 s as six, the kernel 5% slower), mixed ones shorter.
constexpr int kJitInlineChannels = 2, kJitInlineMixed = 6;
std::vector<std::string> jit_sources_split(const std::vector<Compiled>& ch, int block, int min_blocks, bool mixed,
                                           int tiles);
// The program's kernel as one executable cubin: a single unit, or the split units linked.
int jit_build(const std::vector<Compiled>& ch, int block, int min_blocks, bool mixed, int tiles,
              std::vector<char>* cubin, std::string* log);
int jit_prepare(const std::vector<Compiled>& ch, int block, int min_blocks, bool mixed, int tiles, int device, void** fn,
                std::string* err);
int jit_occupancy(void* fn, int block, size_t smem, int* per_sm);
int jit_launch(void* fn, const LaunchParams& lp, int grid, size_t smem, void* stream, std::string* err);
// Whether a captured kernel node runs the compiled kernel fn.
bool jit_node_runs(void* node, void* fn);
// Point an instantiated graph's compiled-kernel node at new launch parameters.
int jit_node_set(void* exec, void* node, void* fn, const LaunchParams& lp, int grid, size_t smem, std::string* err);
size_t smem_bytes_for(const LaunchParams& lp);
int max_ctas_per_sm(int block, size_t smem_bytes, int mixed, int* out, std::string* err);
// Device address and size of the fixed scratch of ps_generate_noalloc on `device` (which must be
// current); the first call on a device looks the address up.
int noalloc_scratch(int device, void** ptr, size_t* bytes, std::string* err);

// inverse.cu
int launch_inverse(const InvPlan& plan, int64_t batch, const double* mom, int64_t ld_m, const double* x1,
                   const double* x2, const double* grid, double* r, int64_t ld_r, double* P, void* stream,
                   std::string* err);
int launch_global_weights(int n_ch, int64_t batch, const double* J, int64_t ld_j, const double* P, int64_t ld_p,
                          const double* alpha, const double* x1, const double* x2, double pdf_a, double pdf_b,
                          const double* f, double* w, void* stream, std::string* err);

}  // namespace ps
