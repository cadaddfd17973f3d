// kin.cuh -- FP64 kinematic helpers shared by the forward interpreter (kernels.cu) and the
// inverse map (inverse.cu): four-momenta, the Kallen function, pure boosts and the t range of
// a 2->2 block.
#pragma once
#include <cmath>
#include <cstdint>

#include "fp64_fast.cuh"

namespace ps {
namespace dev {

constexpr double kPi = 3.141592653589793238462643383279502884;

// Decisions on doubles taken on their bit patterns in the integer ALU, which leaves the FP64
// pipe (1/64 of the FP32 rate) to arithmetic: IEEE doubles of one sign order like their bit
// patterns read as signed integers.
constexpr long long kInfBits = 0x7FF0000000000000LL;
__device__ __forceinline__ long long dbits(double v) { return __double_as_longlong(v); }
// isfinite(v)
__device__ __forceinline__ bool finite_bits(double v) { return (dbits(v) & kInfBits) != kInfBits; }
// The same, and v = +-0, on the words: the compiler recognises a test of the 64-bit pattern as a floating-point
// class test or a comparison, which the FP64 pipe executes (25 and more per event).
__device__ __forceinline__ bool is_finite(double v) { return (__double2hiint(v) & 0x7FF00000) != 0x7FF00000; }
__device__ __forceinline__ bool is_zero(double v) { return ((__double2hiint(v) << 1) | __double2loint(v)) == 0; }
// 0 < v <= 1 (false for NaN)
__device__ __forceinline__ bool in_unit_bits(double v) {
    const long long b = dbits(v);
    return b > 0 && b <= 0x3FF0000000000000LL;
}
// v > 0 (false for NaN and -0)
__device__ __forceinline__ bool pos_bits(double v) {
    const long long b = dbits(v);
    return b > 0 && b <= kInfBits;
}
// a >= b for b >= +0 (false for NaN a)
__device__ __forceinline__ bool ge_pos_bits(double a, double b) {
    const long long x = dbits(a);
    return x >= dbits(b) && x <= kInfBits;
}
// v < -c and v > c for a constant c > 0 and finite v
__device__ __forceinline__ bool below_neg_bits(double v, double c) {
    const long long b = dbits(v);
    return b < 0 && (b & 0x7FFFFFFFFFFFFFFFLL) > dbits(c);
}
__device__ __forceinline__ bool above_pos_bits(double v, double c) { return dbits(v) > dbits(c); }
// an integer 0 <= v < 2^31 held in a double (byte-code immediates), decoded from its bits:
// v = 1.m 2^e gives (1m) >> (52 - e)
__device__ __forceinline__ int small_int(double v) {
    const unsigned long long b = static_cast<unsigned long long>(dbits(v));
    const int e = static_cast<int>((b >> 52) & 0x7FF) - 1023;
    if (e < 0) return 0;
    return static_cast<int>(((b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL) >> (52 - e));
}
// floor(y) for y >= 0 as the conversion to int gives it (saturating at 2^31 - 1; NaN and
// negative y give 0), from the bits: y = 1.m 2^e gives (1m) >> (52 - e)
__device__ __forceinline__ int floor_small(double y) {
    const long long b = dbits(y);
    const int e = static_cast<int>(b >> 52) - 1023;  // b < 0 (negative y) gives e < 0
    if (e < 0) return 0;
    if (e > 30) return b > kInfBits ? 0 : 0x7FFFFFFF;
    return static_cast<int>(((static_cast<unsigned long long>(b) & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL) >> (52 - e));
}
// the double of an int 0 <= k < 2^31, from the bits
__device__ __forceinline__ double small_to_double(int k) {
    if (k <= 0) return 0.0;
    const int msb = 31 - __clz(k);
    const unsigned long long m = (static_cast<unsigned long long>(k) << (52 - msb)) & 0xFFFFFFFFFFFFFULL;
    return __longlong_as_double(static_cast<long long>((static_cast<unsigned long long>(1023 + msb) << 52) | m));
}
// y - k for 0 <= k <= floor(y) < 2^31, y >= 0, exactly, from the bits: the fraction below the binary point where k is
// the floor; another k (a clamped bin) is subtracted as a double
__device__ __forceinline__ double sub_small(double y, int k) {
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(y)), lo = static_cast<uint32_t>(__double2loint(y));
    const int e = static_cast<int>(hi >> 20) - 1023;  // negative y, NaN: out of the range below
    if (k == 0) return y;
    const unsigned long long m = ((static_cast<unsigned long long>((hi & 0xFFFFFu) | 0x100000u) << 32) | lo) << 11;
    const int es = e & 31;
    const unsigned long long f = m << (es + 1);  // the fraction, in units of 2^-64
    const int lz = __clzll(static_cast<long long>(f));
    double v = f == 0 ? 0.0
                      : __longlong_as_double(static_cast<long long>(((f << (lz & 63)) >> 11) +
                                                                          (static_cast<unsigned long long>(1021 - lz) << 52)));
    const bool ok = e >= 0 && e < 31 && static_cast<int>(static_cast<uint32_t>(m >> 32) >> (31 - es)) == k;
    if (__builtin_expect(!ok, 0)) v = fast::slow_sub(y, small_to_double(k));
    return v;
}
// fmax(a, b) on the bit patterns: doubles order like the integers b ^ (0x7FF..F if negative);
// a NaN operand gives the other one
__device__ __forceinline__ double fmax_bits(double a, double b) {
    const long long x = dbits(a), y = dbits(b);
    const bool nan_a = (x & 0x7FFFFFFFFFFFFFFFLL) > kInfBits, nan_b = (y & 0x7FFFFFFFFFFFFFFFLL) > kInfBits;
    const long long kx = x ^ ((x >> 63) & 0x7FFFFFFFFFFFFFFFLL), ky = y ^ ((y >> 63) & 0x7FFFFFFFFFFFFFFFLL);
    return nan_a ? b : (nan_b ? a : (kx >= ky ? a : b));
}
// fmin(fmax(x, lo), hi) for 0 <= lo <= hi: NaN and values below lo give lo, +inf gives hi
__device__ __forceinline__ double clamp_nonneg(double x, double lo, double hi) {
    const long long b = dbits(x);
    if (b < dbits(lo) || b > kInfBits) return lo;
    return b > dbits(hi) ? hi : x;
}

struct P4 {
    double e, x, y, z;
};

__device__ __forceinline__ P4 p4_add(P4 a, P4 b) { return {a.e + b.e, a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ P4 p4_sub(P4 a, P4 b) { return {a.e - b.e, a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ double p4_sq(P4 a) { return a.e * a.e - a.x * a.x - a.y * a.y - a.z * a.z; }

__device__ __forceinline__ bool zero_bits(double v) { return (dbits(v) << 1) == 0; }       // +-0
__device__ __forceinline__ bool nonneg_bits(double v) { return dbits(v) >= 0 || zero_bits(v); }
__device__ __forceinline__ bool nonpos_bits(double v) { return dbits(v) <= 0; }            // includes -0
// lambda(x, m1^2, m2^2) from the masses m1, m2 >= 0 themselves: the factorised form of kallen_in with
// sqrt(m^2) replaced by m.  For a double m the correctly rounded sqrt of fl(m^2) is m exactly (its
// error is below half an ulp of m), so no square root is taken.  Its root: x itself for two massless legs.
__device__ __forceinline__ double kallen_out(double x, double m1, double m2) {
    double l;
    if (is_zero(m1) && is_zero(m2)) {
        l = __dmul_rn(x, x);
    } else {
        const double hi = __dadd_rn(m1, m2), lo = __dadd_rn(m1, -m2);
        l = __dmul_rn(fma(-hi, hi, x), fma(-lo, lo, x));
    }
    return pos_bits(l) ? l : 0.0;
}
__device__ __forceinline__ double sqrt_kallen_out(double x, double m1, double m2) {
    if (is_zero(m1) && is_zero(m2)) return x;
    const double l = kallen_out(x, m1, m2);
    return pos_bits(l) ? fast::sqrt(l) : 0.0;
}

// Pure boosts out of the rest frame of q (mass mq) sharing their reciprocals: 1/mq and
// 1/(mq (E_q + mq)) are taken once per frame, for every momentum boosted with it.
struct BoostFrame {
    double e, x, y, z;  // q
    double inv_m, k;    // 1/mq, 1/(mq (E_q + mq))
};
__device__ __forceinline__ BoostFrame boost_frame(const P4& q, double mq, double inv_m) {
    return {q.e, q.x, q.y, q.z, inv_m, fast::rcp(mq * (q.e + mq))};
}
// The back-to-back daughters q1 = (e1, v) and q2 = (e2, -v) of a two-body decay, boosted out of
// the same frame: q2 . b = -(q1 . b) exactly, so the dot product is formed once.
__device__ __forceinline__ void boost_out_pair(const P4& q1, double e2, const BoostFrame& b, P4& p1, P4& p2) {
    const double qp = b.x * q1.x + b.y * q1.y + b.z * q1.z;
    const double c1 = fma(qp, b.k, q1.e * b.inv_m), c2 = fma(-qp, b.k, e2 * b.inv_m);
    p1 = {(b.e * q1.e + qp) * b.inv_m, q1.x + b.x * c1, q1.y + b.y * c1, q1.z + b.z * c1};
    p2 = {(b.e * e2 - qp) * b.inv_m, b.x * c2 - q1.x, b.y * c2 - q1.y, b.z * c2 - q1.z};
}
__device__ __forceinline__ P4 boost_in(const P4& p, const BoostFrame& b) {
    double qp = b.x * p.x + b.y * p.y + b.z * p.z;
    double c = fma(qp, b.k, -p.e * b.inv_m);
    return {(b.e * p.e - qp) * b.inv_m, p.x + b.x * c, p.y + b.y * c, p.z + b.z * c};
}

// Sums and products with a term that may be the constant zero of a compiled channel (massless legs):
// x + 0 and x * 0 do not fold under IEEE rules, a select on the bits of a constant does.
__device__ __forceinline__ double add_z(double a, double b) { return is_zero(b) ? a : (is_zero(a) ? b : __dadd_rn(a, b)); }
__device__ __forceinline__ double sub_z(double a, double b) { return is_zero(b) ? a : (is_zero(a) ? -b : __dadd_rn(a, -b)); }
__device__ __forceinline__ double mul_z(double a, double b) { return is_zero(a) || is_zero(b) ? 0.0 : __dmul_rn(a, b); }

// Kallen lambda(x, y, z) = (x - y - z)^2 - 4 y z (x >= 0) of the incoming legs of a 2->2 block, without cancellation
// and with every rounding spelled out:
//   y, z >= 0: (x - (sqrt y + sqrt z)^2)(x - (sqrt y - sqrt z)^2)
//   y, z <= 0: x^2 + 2x(|y| + |z|) + (|y| - |z|)^2  (space-like legs of a t-chain)
//   mixed:     (x - y - z)^2 - 4 y z                (-4yz >= 0)
// clamped at zero.  The branches are taken on the bit patterns (integer ALU); y = z = 0 (two massless legs)
// is x^2.
__device__ __forceinline__ double kallen_in(double x, double y, double z) {
    double l;
    if (is_zero(y) && is_zero(z)) {
        l = __dmul_rn(x, x);
    } else if (nonneg_bits(y) && nonneg_bits(z)) {
        const double ry = fast::sqrt(y), rz = fast::sqrt(z);
        const double hi = __dadd_rn(ry, rz), lo = __dadd_rn(ry, -rz);
        l = __dmul_rn(fma(-hi, hi, x), fma(-lo, lo, x));
    } else if (nonpos_bits(y) && nonpos_bits(z)) {
        const double d = sub_z(z, y), t = add_z(y, z);  // (x - t)^2 - 4 y z = x (x - 2 t) + d^2, t <= 0
        l = fma(d, d, __dmul_rn(x, fma(-2.0, t, x)));
    } else {
        const double d = __dadd_rn(__dadd_rn(x, -y), -z);
        l = fma(d, d, __dmul_rn(__dmul_rn(-4.0, y), z));
    }
    return pos_bits(l) ? l : 0.0;
}

// t range of a 2->2 block (Eq. t_invariant_theta): t = A + B cos(theta); the root of larger
// magnitude directly, the other from t+ t- =
//   (m1^2 - mA^2)(m2^2 - mB^2) + (m1^2 mB^2 - m2^2 mA^2)(m1^2 - m2^2 - mA^2 + mB^2)/s.
// With it goes what the block itself needs: the Kallen functions of
// the incoming and outgoing legs and B.  Every rounding is spelled out (no contraction is left to the
// compiler): the |t| map and the block evaluate it separately, and the distance |t| - |t|_min must be
// taken from the very bound that |t| was built on.
struct TRange {
    double lo, hi, B, lam_in, lam_out;  // |t|_min, |t|_max
    double e1, e2;                      // s + m1^2 - m2^2, s - m1^2 + m2^2
};
__device__ __forceinline__ TRange t_range_fast(double s, double mA2, double mB2, double m1, double m2) {
    TRange r;
    const double m12 = __dmul_rn(m1, m1), m22 = __dmul_rn(m2, m2);
    const double inv_s = fast::rcp(s), inv2s = fast::half(inv_s);
    r.e1 = sub_z(add_z(s, m12), m22);
    r.e2 = sub_z(add_z(s, m22), m12);
    const double A = fma(-__dmul_rn(sub_z(add_z(s, mA2), mB2), r.e1), inv2s, add_z(mA2, m12));
    r.lam_in = kallen_in(s, mA2, mB2);
    r.lam_out = kallen_out(s, m1, m2);
    const double l = __dmul_rn(r.lam_in, r.lam_out);
    r.B = pos_bits(l) ? __dmul_rn(fast::sqrt(l), inv2s) : 0.0;
    const double cross = mul_z(sub_z(mul_z(m12, mB2), mul_z(m22, mA2)), add_z(sub_z(sub_z(m12, m22), mA2), mB2));
    const double prod = fma(cross, inv_s, mul_z(sub_z(m12, mA2), sub_z(m22, mB2)));
    const bool a_nonpos = nonpos_bits(A);
    const double big = __dadd_rn(A, a_nonpos ? -r.B : r.B);
    const double small = is_zero(big) ? 0.0 : fast::div(prod, big);
    r.lo = -(a_nonpos ? small : big);
    r.hi = -(a_nonpos ? big : small);
    return r;
}

}  // namespace dev
}  // namespace ps
