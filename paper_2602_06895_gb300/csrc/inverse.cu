// inverse.cu -- the inverse channel map on the GPU (every mapping of Sec. 2 is invertible; the
// round trip of Sec. 4.1) and the global multichannel weight of Kleiss and Pittau (Eq.
// multi-channel-standard).
//
// ps_inverse_kernel recovers, for one event per thread and in FP64, the random numbers r of a
// channel from the lab-frame momenta [p_a, p_b, p_1..p_n] and (x1, x2):
//   - the longitudinal beam boost is undone on the light cone;
//   - every node's invariant comes from its leaves in the collinear-safe chord form
//       (sum p_i)^2 = sum m_i^2 + sum_{i<k} [2 (m_i^2 |p_k|^2 + m_k^2 |p_i|^2 + m_i^2 m_k^2)
//                      / (E_i E_k + |p_i||p_k|) + |p_i||p_k| |n_i - n_k|^2];
//   - shat, x1 x2, the s-channel invariants (with the forward's recursive bounds), the t-chain
//     invariants, |t| of every 2->2 block and its azimuth about p_A in the block rest frame, and
//     the decay angles in each parent's rest frame are passed through the inverse invariant maps;
//   - the VEGAS grid is inverted last.
// The same kernel evaluates the channel's SDE propagator product P(p) from the lab momenta.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <string>

#include "kin.cuh"
#include "ps_internal.h"

namespace ps {
namespace inv {

using dev::kPi;
using dev::P4;

constexpr int kMaxLeg = kMaxOutMomenta + 2;

namespace fast = dev::fast;

// Both inverse maps: where rounding has collapsed the range to a point every r maps to it, and 0 is
// returned (the quotients below would be 0/0 or infinite); for a NaN x or NaN bounds, NaN as from the quotients.
// (comparisons on the bits here and below: the FP64 pipe that bounds the kernel would execute them)
__device__ __forceinline__ bool nan_bits(double v) { return (dev::dbits(v) & 0x7FFFFFFFFFFFFFFFLL) > dev::kInfBits; }
__device__ __forceinline__ bool empty_range(double x, double xmin, double xmax) {  // x_max <= x_min for bounds >= 0
    return dev::dbits(xmax) <= dev::dbits(xmin) && !nan_bits(x) && !nan_bits(xmin) && !nan_bits(xmax);
}

// inverse power-law map (anchored as the forward map; by roots where 1/(1 - nu) is an integer, as there: 31 FP64
// instructions where the logarithms and exponentials take 47 and CUDA's took 130)
__device__ __forceinline__ double inv_nu(double x, double m, double nu, double xmin, double xmax, double a) {
    const double m2 = dev::pos_bits(m) ? m * m : -a;
    const double lo = xmin - m2, hi = xmax - m2;
    if (empty_range(x, xmin, xmax)) return 0.0;
    const double p = fast::div(xmax - xmin, lo), q = fast::div(x - xmin, lo);
    if (dev::dbits(nu) == dev::dbits(1.0)) return fast::div(fast::log1p(q), fast::log1p(p));
    const double w = 1.0 - nu;
    if (dev::dbits(nu) < dev::dbits(1.0)) {
        const fast::WholePower k = fast::whole_power(w, false);
        if (k.ok && fast::root_arg(p) && fast::root_arg(q)) return fast::div(fast::power_root(q, k), fast::power_root(p, k));
        return fast::div(fast::expm1(w * fast::log1p(q)), fast::expm1(w * fast::log1p(p)));
    }
    return 1.0 - fast::div(fast::expm1(w * fast::log(fast::div(x - m2, hi))), fast::expm1(-w * fast::log1p(p)));
}

// inverse Breit-Wigner map: the angle measured from the nearer end of the range.  With CUDA's functions: far above a
// narrow resonance r is within 1e-8 of 1, one ulp of it moves the density there by 1e-8, and this is the rounding
// that earlier densities were computed with.
__device__ __forceinline__ double inv_bw(double x, double M, double G, double xmin, double xmax) {
    const double mg = M * G, m2 = M * M;
    const double a = (xmin - m2) / mg, b = (xmax - m2) / mg;
    if (empty_range(x, xmin, xmax)) return 0.0;
    const double D = atan2((xmax - xmin) / mg, fma(a, b, 1.0));
    const double t = (x - m2) / mg;
    if (x - xmin <= xmax - x) return atan2((x - xmin) / mg, fma(a, t, 1.0)) / D;
    return 1.0 - atan2((xmax - x) / mg, fma(b, t, 1.0)) / D;
}

__device__ __forceinline__ double inv_invariant(double x, double M, double G, double nu, double xmin, double xmax,
                                                double a) {
    return dev::pos_bits(G) ? inv_bw(x, M, G, xmin, xmax) : inv_nu(x, M, nu, xmin, xmax, a);
}

// p into the rest frame of q of mass m (1/m given).  Quotients and not products with reciprocals here and in the
// kernel: their extra rounding raised the error of the densities by 13%, at 5% of the kernel's time.
__device__ __forceinline__ P4 to_rest(const P4& p, const P4& q, double m, double inv_m) {
    const double qp = q.x * p.x + q.y * p.y + q.z * p.z;
    const double c = fma(-p.e, inv_m, fast::div(qp, m * (q.e + m)));
    return {(q.e * p.e - qp) * inv_m, p.x + q.x * c, p.y + q.y * c, p.z + q.z * c};
}

__device__ __forceinline__ double unit_phi(double y, double x) {
    const double ph = fast::atan2(fabs(y), x) * (0.5 / kPi);
    return dev::dbits(y) < 0 && !dev::is_zero(y) ? 1.0 - ph : ph;
}

__device__ __forceinline__ double vegas_inv(double rp, const double* e, int N) {
    int lo = 0, hi = N;  // e[lo] <= rp < e[lo + 1]
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (e[mid] <= rp) lo = mid;
        else hi = mid;
    }
    return (static_cast<double>(lo) + (rp - e[lo]) / (e[lo + 1] - e[lo])) / static_cast<double>(N);
}

__global__ void __launch_bounds__(128) ps_inverse_kernel(const __grid_constant__ InvPlan P, int64_t batch,
                                                          const double* mom, int64_t ldm, const double* x1in,
                                                          const double* x2in, const double* grid, double* r,
                                                          int64_t ldr, double* Pout) {
    const int64_t b = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (b >= batch) return;
    const int n = P.n;
    P4 q[kMaxLeg];
    for (int i = 0; i < n + 2; ++i)
        q[i] = {mom[(4 * i) * ldm + b], mom[(4 * i + 1) * ldm + b], mom[(4 * i + 2) * ldm + b],
                mom[(4 * i + 3) * ldm + b]};
    const double x1 = P.hadronic ? x1in[b] : 1.0, x2 = P.hadronic ? x2in[b] : 1.0;

    // SDE propagator product from the lab momenta (q_k = p_a - legs for t-channel propagators)
    if (Pout) {
        double den = 1.0, prod = 1.0;
        for (int k = 0; k < P.n_prop; ++k) {
            P4 s = P.pkind[k] == 1 ? q[0] : P4{0.0, 0.0, 0.0, 0.0};
            const double sg = P.pkind[k] == 1 ? -1.0 : 1.0;
            for (int i = 0; i < n; ++i)
                if (P.pmask[k] & (1u << i)) s = {s.e + sg * q[2 + i].e, s.x + sg * q[2 + i].x, s.y + sg * q[2 + i].y,
                                                 s.z + sg * q[2 + i].z};
            const double dd = dev::p4_sq(s) - P.pM[k] * P.pM[k], mg = P.pM[k] * P.pG[k];
            den *= P.pkind[k] == 1 ? dd * dd : fma(dd, dd, mg * mg);
            if (den > 1e200) {  // keep the running product in range
                prod = fast::slow_div(prod, den);
                den = 1.0;
            }
        }
        Pout[b] = fast::div(prod, den);
    }

    // partonic frame (light-cone form of the inverse longitudinal boost)
    if (P.hadronic && P.lab_frame) {
        const double rho = fast::sqrt(fast::div(x1, x2));
        for (int i = 0; i < n + 2; ++i) {
            const double plus = fast::div(q[i].e + q[i].z, rho), minus = rho * (q[i].e - q[i].z);
            q[i].e = 0.5 * (plus + minus);
            q[i].z = 0.5 * (plus - minus);
        }
    }

    // node momenta, and the invariants of the non-root decay nodes (the root's is shat; leaves
    // carry their masses): the leaf directions are needed only if such a node exists
    double ap[kMaxLeg], nx[kMaxLeg], ny[kMaxLeg], nz[kMaxLeg], ml[kMaxLeg];
    bool any_decay = false;
    for (int j = 1; j < P.n_nodes; ++j) any_decay |= P.node[j].kind == PS_NODE_DECAY;
    for (int j = 0; j < P.n_nodes; ++j)
        if (P.node[j].kind == PS_NODE_LEAF) {
            const int i = P.node[j].leaf;
            ml[i] = P.node[j].mass;
            if (any_decay) {
                const P4 p = q[2 + i];
                const double a = fast::sqrt(p.x * p.x + p.y * p.y + p.z * p.z);
                ap[i] = a;
                nx[i] = fast::div(p.x, a);
                ny[i] = fast::div(p.y, a);
                nz[i] = fast::div(p.z, a);
            }
        }
    P4 pn[kInvNodes];
    double s[kInvNodes];
    for (int j = 1; j < P.n_nodes; ++j) {
        const InvNode& nd = P.node[j];
        if (nd.kind == PS_NODE_LEAF) {
            pn[j] = q[2 + nd.leaf];
            s[j] = nd.mass * nd.mass;
            continue;
        }
        const uint32_t mask = nd.mask;
        P4 acc{0.0, 0.0, 0.0, 0.0};
        double s2 = 0.0;
        for (int i = 0; i < n; ++i) {
            if (!(mask & (1u << i))) continue;
            acc = dev::p4_add(acc, q[2 + i]);
            s2 += ml[i] * ml[i];
            for (int k = i + 1; k < n; ++k) {
                if (!(mask & (1u << k))) continue;
                const double dx = nx[i] - nx[k], dy = ny[i] - ny[k], dz = nz[i] - nz[k];
                const double mi2 = ml[i] * ml[i], mk2 = ml[k] * ml[k];
                s2 += ap[i] * ap[k] * (dx * dx + dy * dy + dz * dz);
                if (!(dev::is_zero(mi2) && dev::is_zero(mk2)))
                    s2 += fast::div(2.0 * (mi2 * ap[k] * ap[k] + mk2 * ap[i] * ap[i] + mi2 * mk2),
                                    q[2 + i].e * q[2 + k].e + ap[i] * ap[k]);
            }
        }
        pn[j] = acc;
        s[j] = s2;
    }
    double root[kInvNodes];  // sqrt(s) of the decay nodes
    auto leg_mass = [&](int j) { return P.node[j].kind == PS_NODE_LEAF ? P.node[j].mass : root[j]; };

    double shat;
    if (P.hadronic) {
        shat = x1 * x2 * P.S;
        r[P.d_shat * ldr + b] = inv_invariant(shat, P.shat_M, P.shat_G, P.shat_nu, P.mleaf * P.mleaf, P.S, P.a);
        r[P.d_x * ldr + b] = fast::div(fast::log(x1), fast::log(fast::div(shat, P.S)));
    } else {
        shat = P.sqrt_s * P.sqrt_s;
    }
    s[0] = shat;
    for (int j = 0; j < P.n_nodes; ++j)
        if (j == 0 || P.node[j].kind == PS_NODE_DECAY) root[j] = fast::sqrt(s[j]);

    // s-channel invariants with the forward's bounds
    for (int i = 0; i < P.n_sorder; ++i) {
        const int j = P.sorder[i];
        double mlo = P.lo_c[i];
        for (int k = P.lo_beg[i]; k < P.off_beg[i]; ++k) mlo += root[P.ids[k]];
        double off = P.off_c[i];
        for (int k = P.off_beg[i]; k < P.lo_beg[i + 1]; ++k) off += root[P.ids[k]];
        const int top = P.top[i];
        const double mtop = (top == 0 && !P.hadronic) ? P.sqrt_s : root[top];
        const double mhi = dev::fmax_bits(mtop - off, mlo);
        const InvNode& nd = P.node[j];
        r[P.d_s[j] * ldr + b] = inv_invariant(s[j], nd.M, nd.G, nd.nu, mlo * mlo, mhi * mhi, P.a);
    }

    // t-chain (legs taken inwards from side A or B)
    const int kappa = P.kappa;
    if (kappa > 0) {
        const InvNode& root = P.node[0];
        double sts[kInvLegs + 1], rts[kInvLegs + 1], irs[kInvLegs + 1];  // the block invariants, roots and their reciprocals
        sts[0] = shat;
        rts[0] = fast::sqrt_rcp(shat, irs[0]);
        int l2 = 0, r2 = kappa;
        for (int i = 1; i < kappa; ++i) {
            if (P.side[i] == 0) ++l2;
            else --r2;
            P4 c{0.0, 0.0, 0.0, 0.0};
            double msum = 0.0;
            for (int k = l2; k <= r2; ++k) {
                c = dev::p4_add(c, pn[root.child[k]]);
                msum += leg_mass(root.child[k]);
            }
            sts[i] = dev::p4_sq(c);
            const double mi = leg_mass(root.child[P.order[i]]);
            rts[i] = fast::sqrt_rcp(sts[i], irs[i]);
            const double mx = dev::fmax_bits(rts[i - 1] - mi, 0.0);
            const double smin = msum * msum;
            r[P.d_ts[i] * ldr + b] = inv_nu(sts[i], 0.0, P.ts_nu, smin, dev::fmax_bits(mx * mx, smin), P.a);
        }
        const double e0 = 0.5 * rts[0];
        P4 pA{e0, 0.0, 0.0, e0}, pB{e0, 0.0, 0.0, -e0};
        double mA2 = 0.0, mB2 = 0.0, scur = shat;
        for (int i = 1; i <= kappa; ++i) {
            double m1, m2;
            P4 q1, q2;
            if (i == kappa) {
                const int la = root.child[P.order[kappa]], lb = root.child[P.order[kappa + 1]];
                m1 = leg_mass(la);
                m2 = leg_mass(lb);
                q1 = pn[la];
                q2 = pn[lb];
            } else if (P.side[i] == 0) {
                const int l1 = root.child[P.order[i]];
                m1 = leg_mass(l1);
                m2 = rts[i];
                q1 = pn[l1];
                q2 = dev::p4_sub(dev::p4_add(pA, pB), q1);
            } else {
                const int l1 = root.child[P.order[i]];
                m1 = rts[i];
                m2 = leg_mass(l1);
                q2 = pn[l1];
                q1 = dev::p4_sub(dev::p4_add(pA, pB), q2);
            }
            const double tabs = -dev::p4_sq(dev::p4_sub(pA, q1));
            const dev::TRange tr = dev::t_range_fast(scur, mA2, mB2, m1, m2);
            const double tlo = dev::fmax_bits(tr.lo, 0.0), thi = dev::fmax_bits(tr.hi, tlo);
            r[P.d_tt[i] * ldr + b] = inv_nu(tabs, 0.0, P.t_nu, tlo, thi, P.a);
            // azimuth of q1 about the direction of pA in the block rest frame
            const P4 p0 = dev::p4_add(pA, pB);
            const P4 pAs = to_rest(pA, p0, rts[i - 1], irs[i - 1]), q1s = to_rest(q1, p0, rts[i - 1], irs[i - 1]);
            const double pt = fast::sqrt(pAs.x * pAs.x + pAs.y * pAs.y);
            const double pp = fast::sqrt(pt * pt + pAs.z * pAs.z);
            const double cA = fast::div(pAs.z, pp), sA = fast::div(pt, pp);
            const bool off_axis = dev::pos_bits(pt);
            const double cpA = off_axis ? fast::div(pAs.x, pt) : 1.0, spA = off_axis ? fast::div(pAs.y, pt) : 0.0;
            const double v1 = cpA * q1s.x + spA * q1s.y;
            const double v2 = -spA * q1s.x + cpA * q1s.y;
            r[P.d_tphi[i] * ldr + b] = unit_phi(v2, cA * v1 - sA * q1s.z);
            if (i < kappa) {
                if (P.side[i] == 0) {
                    pA = dev::p4_sub(pA, q1);
                    mA2 = -tabs;
                } else {
                    pB = dev::p4_sub(pB, q2);
                    mB2 = -tabs;
                }
                scur = sts[i];
            }
        }
    }

    // decay angles in each parent's rest frame (the root decays at rest)
    for (int i = 0; i < P.n_pre; ++i) {
        const int j = P.pre[i];
        const int c1 = P.node[j].child[0];
        const P4 qq = j == 0 ? pn[c1] : to_rest(pn[c1], pn[j], root[j], fast::rcp(root[j]));
        const double pt2 = qq.x * qq.x + qq.y * qq.y;
        const double pa = fast::sqrt(pt2 + qq.z * qq.z);
        // r_theta = (1 + cos theta)/2 in the sin^2(theta/2) form near the poles
        const double h = 0.5 * fast::div(pt2, pa * (pa + fabs(qq.z)));
        const double rth = dev::dbits(qq.z) >= 0 || dev::is_zero(qq.z) ? 1.0 - h : h;
        r[P.d_dth[j] * ldr + b] = rth;
        r[P.d_dphi[j] * ldr + b] = unit_phi(qq.y, qq.x);
    }

    for (int j = 0; j < P.vdims; ++j) r[j * ldr + b] = vegas_inv(r[j * ldr + b], grid + j * (P.vbins + 1), P.vbins);
}

struct GlobalArgs {
    int32_t n_ch;
    double alpha[kMaxChannels];
};

// (x1 x2)^pa ((1 - x1)(1 - x2))^pb: one exponential of the sum of the logarithms as pairs, and for pb = 1, 2, 3
// products (38 FP64 instructions where four powers take 330; relative error below 4e-16 either way).  Outside
// 0 < x < 1 and for infinite or NaN exponents: the powers.
__device__ __forceinline__ double pdf_pair(double x1, double x2, double pa, double pb) {
    auto inside = [](double x) { return fast::hi32(x) - 0x00100000u < 0x3FE00000u; };  // positive, normal, below 1
    if (!(inside(x1) && inside(x2) && fabs(pa) < 1e3 && fabs(pb) < 1e3))
        return pow(x1, pa) * pow(1.0 - x1, pb) * pow(x2, pa) * pow(1.0 - x2, pb);
    double h1, l1, h2, l2;
    fast::log_pair(x1, h1, l1);
    fast::log_pair(x2, h2, l2);
    const double f = fast::exp_of(pa, h1 + h2, l1 + l2);
    const double y1 = 1.0 - x1, y2 = 1.0 - x2;
    if (pb == 3.0) return f * (y1 * y1 * y1) * (y2 * y2 * y2);
    if (pb == 2.0) return f * (y1 * y1) * (y2 * y2);
    if (pb == 1.0) return f * y1 * y2;
    if (pb == 0.0) return f;
    fast::log_pair(y1, h1, l1);
    fast::log_pair(y2, h2, l2);
    return f * fast::exp_of(pb, h1 + h2, l1 + l2);
}

// w = f / sum_j alpha_j g_j with g_j = 1 / J_j (J_j = 0: outside channel j, no density); f is
// the given integrand, or pdf(x1) pdf(x2) sum_j P_j (the SDE propagator sum) when f is null.
__global__ void ps_global_weight_kernel(const __grid_constant__ GlobalArgs A, int64_t batch, const double* J,
                                        int64_t ldj, const double* Pp, int64_t ldp, const double* x1,
                                        const double* x2, double pa, double pb, const double* f, double* w) {
    const int64_t b = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (b >= batch) return;
    double g = 0.0;
    for (int j = 0; j < A.n_ch; ++j) {
        const double Jj = J[j * ldj + b];
        if (dev::pos_bits(Jj)) g += fast::div(A.alpha[j], Jj);
    }
    double fv;
    if (f) {
        fv = f[b];
    } else {
        double ps = 0.0;
        for (int j = 0; j < A.n_ch; ++j) ps += Pp[j * ldp + b];
        fv = ps;
        if (x1) fv *= pdf_pair(x1[b], x2[b], pa, pb);
    }
    w[b] = g > 0.0 ? fast::div(fv, g) : 0.0;
}

}  // namespace inv

void count_launches(int n);

int launch_inverse(const InvPlan& plan, int64_t batch, const double* mom, int64_t ld_m, const double* x1,
                   const double* x2, const double* grid, double* r, int64_t ld_r, double* P, void* stream,
                   std::string* err) {
    if (batch <= 0) return PS_OK;
    const unsigned blocks = static_cast<unsigned>((batch + 127) / 128);
    inv::ps_inverse_kernel<<<blocks, 128, 0, static_cast<cudaStream_t>(stream)>>>(plan, batch, mom, ld_m, x1, x2,
                                                                                   grid, r, ld_r, P);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        *err = std::string("ps_inverse_kernel: ") + cudaGetErrorString(e);
        return PS_ERR_CUDA;
    }
    return PS_OK;
}

int launch_global_weights(int n_ch, int64_t batch, const double* J, int64_t ld_j, const double* P, int64_t ld_p,
                          const double* alpha, const double* x1, const double* x2, double pdf_a, double pdf_b,
                          const double* f, double* w, void* stream, std::string* err) {
    if (batch <= 0) return PS_OK;
    inv::GlobalArgs A{};
    A.n_ch = n_ch;
    for (int j = 0; j < n_ch; ++j) A.alpha[j] = alpha[j];
    const unsigned blocks = static_cast<unsigned>((batch + 255) / 256);
    inv::ps_global_weight_kernel<<<blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(A, batch, J, ld_j, P, ld_p, x1,
                                                                                        x2, pdf_a, pdf_b, f, w);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        *err = std::string("ps_global_weight_kernel: ") + cudaGetErrorString(e);
        return PS_ERR_CUDA;
    }
    return PS_OK;
}

}  // namespace ps
