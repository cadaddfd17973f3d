// fp64_fast.cuh -- FP64 division, roots and elementary functions that spend few FP64 instructions.
//
// The FP64 pipe takes a warp instruction every 64 cycles of a scheduler (2 lanes per cycle and SM),
// the integer and FP32 pipes one in 1-2 cycles, and the phase-space kernels run the FP64 pipe at its
// ceiling while the others idle.  So each function here
//   - takes its seed (reciprocal, root) in FP32, refined to about 43 bits as an unevaluated pair of
//     floats, and assembles the pair into a double's bits on the integer ALU;
//   - reduces its argument with a table index found in FP32, and evaluates in FP32 the terms of its
//     polynomial that lie 2^-29 or more below the result;
//   - scales by powers of two on the exponent field;
// and leaves to the FP64 pipe only the operations that carry the result's last bits.
// FP64 instructions per call here, and of CUDA's function (measured by ps_fp64_probe's kinds):
//   rcp 2 (5), div 3 (8), sqrt 2 (8), rsqrt 4 (9), exp 7 (15), expm1 9 (25), log 9 (28),
//   log1p 13 (30), atan2 11 (34).
// Every function takes its short form on the range its comment names; zeros, subnormals,
// infinities, NaN and extreme exponents go to CUDA's function, in one out-of-line copy.  The short form
// comes first and unconditionally (a value that is not used out of its range; table indices are in
// bounds for every input), so that two calls on the same argument are one to the compiler.
#pragma once
#include "fp64_tables.h"

namespace ps {
namespace dev {
namespace fast {

constexpr int kMaxPower = 6;

// CUDA's functions for the arguments outside the short forms' ranges: out of line, so that the
// kernels' straight code does not carry them.
static __device__ __noinline__ double slow_div(double a, double b) { return a / b; }
static __device__ __noinline__ double slow_mul(double a, double b) { return a * b; }
static __device__ __noinline__ double slow_sub(double a, double b) { return a - b; }
static __device__ __noinline__ double slow_sqrt(double x) { return ::sqrt(x); }
static __device__ __noinline__ double slow_rsqrt(double x) { return ::rsqrt(x); }
static __device__ __noinline__ double slow_exp(double x) { return ::exp(x); }
// exp(v + w) for a correction w of a few ulps of v: e + e w
static __device__ __noinline__ double slow_exp(double v, double w) {
    const double e = ::exp(v);
    return ::isfinite(e) && ::isfinite(w) ? ::fma(e, w, e) : e;
}
static __device__ __noinline__ double slow_expm1(double x) { return ::expm1(x); }
static __device__ __noinline__ double slow_log(double x) { return ::log(x); }
static __device__ __noinline__ double slow_log1p(double x) { return ::log1p(x); }
static __device__ __noinline__ double slow_atan2(double y, double x) { return ::atan2(y, x); }

__device__ __forceinline__ uint32_t hi32(double x) { return static_cast<uint32_t>(__double2hiint(x)); }
__device__ __forceinline__ uint32_t lo32(double x) { return static_cast<uint32_t>(__double2loint(x)); }
__device__ __forceinline__ double from32(uint32_t hi, uint32_t lo) {
    return __hiloint2double(static_cast<int>(hi), static_cast<int>(lo));
}
// the exponent field lies in [64, 1984): the value and the products formed with its reciprocal or
// root are normal numbers
__device__ __forceinline__ bool mid_range(double x) { return ((hi32(x) >> 20) & 0x7FFu) - 64u < 1920u; }

// FP32 approximations of the hardware (about 1 ulp), for arguments in [1, 4)
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// a float normal as a double, and a double truncated to a float (0 below the float normals; the
// caller keeps |x| below 2^127)
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x);
    return from32((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u), u << 29);
}
__device__ __forceinline__ float narrow(double x) {
    const uint32_t hi = hi32(x), e = (hi >> 20) & 0x7FFu;
    const uint32_t m = __funnelshift_l(lo32(x), hi, 3) & 0x7FFFFFu;
    return e < 897u ? 0.0f : __uint_as_float((hi & 0x80000000u) | ((e - 896u) << 23) | m);
}
// any float below 2^127 as a double, 0 for |x| < 2^-100
__device__ __forceinline__ double widen_or_zero(float x) { return fabsf(x) < 0x1p-100f ? 0.0 : widen(x); }
// an integer-valued float |k| < 2^23 as a double
__device__ __forceinline__ double widen_int(float k) { return k == 0.0f ? 0.0 : widen(k); }
// x 2^k on the exponent field; k and the result's exponent as the callers' ranges allow
__device__ __forceinline__ double scale2(double x, int k) { return from32(hi32(x) + (static_cast<uint32_t>(k) << 20), lo32(x)); }
// x 2^k for |k| < 60, on the exponent field (a plain product as the alternative would be evaluated for every
// x and selected, and a predicated one still takes the FP64 pipe's time: 5% of the 2->4 program)
__device__ __forceinline__ double mul2(double x, int k) {
    double v = scale2(x, k);
    if (__builtin_expect(!mid_range(x), 0)) v = slow_mul(x, scale2(1.0, k));
    return v;
}
__device__ __forceinline__ double half(double x) { return mul2(x, -1); }
__device__ __forceinline__ double twice(double x) { return mul2(x, 1); }

// The fraction 1.f of a double as the float of its top 23 bits and (times 2^23) the rest.
__device__ __forceinline__ float frac_hi(double x) {
    return __uint_as_float(0x3F800000u | (__funnelshift_l(lo32(x), hi32(x), 3) & 0x7FFFFFu));
}
__device__ __forceinline__ float frac_lo(double x) {
    return __uint_as_float(0x3F800000u | ((lo32(x) & 0x1FFFFFFFu) >> 6)) - 1.0f;
}
// The double of s + n 2^-43 (s a float in [1/2, 1]) or of s + n 2^-42 (s in [1, 2]), its exponent
// field raised by `e` (and a sign, in bit 31 of `e`): 2^10 units of the last place each.
__device__ __forceinline__ double join(float s, int n, uint32_t e) {
    const uint32_t u = __float_as_uint(s);
    const unsigned long long b = (static_cast<unsigned long long>((u >> 3) + 0x38000000u + e) << 32) | (u << 29);
    return __longlong_as_double(static_cast<long long>(b) + (static_cast<long long>(n) << 10));
}
// round(x) of |x| < 2^22 as an int
__device__ __forceinline__ int round_int(float x) { return __float_as_int(x + 12582912.0f) - 0x4B400000; }

// 1/x to a relative 2^-42 (mid_range(x)): r = 1/m of the leading float m, corrected by the residual
// 1 - r (m + the rest), which is exact up to its last bits.
__device__ __forceinline__ double rcp_seed(double x) {
    const float m = frac_hi(x), l = frac_lo(x);
    const float r = fminf(fmaxf(rcp_approx(m), 0.5f), 1.0f);
    const float e = fmaf(-l * 0x1p-23f, r, fmaf(-m, r, 1.0f));
    const uint32_t hi = hi32(x);
    return join(r, round_int(r * e * 0x1p43f), (hi & 0x80000000u) - ((hi & 0x7FF00000u) - 0x3FF00000u));
}

// 1/x and a/b: a seed and one Newton step, the quotient corrected by its exact remainder.  Half an
// ulp plus 2^-30 of one; the correctly rounded value otherwise.
__device__ __forceinline__ double rcp(double x) {
    const double s = rcp_seed(x);
    double r = fma(s, fma(-x, s, 1.0), s);
    if (__builtin_expect(!mid_range(x), 0)) r = slow_div(1.0, x);
    return r;
}
__device__ __forceinline__ double div(double a, double b) {
    // b and a/b in the middle of the range (or a zero, whose quotient is its product with the seed: the remainder's
    // sum would lose the sign of -0)
    const uint32_t ea = (hi32(a) >> 20) & 0x7FFu, eb = (hi32(b) >> 20) & 0x7FFu;
    const bool zero = (hi32(a) << 1 | lo32(a)) == 0u;
    const bool ok = eb - 64u < 1920u && ((ea - 64u < 1920u && ea - eb + 900u < 1800u) || zero);
    const double r = rcp_seed(b), q = __dmul_rn(a, r);
    double v = fma(fma(-b, q, a), r, q);
    if (zero) v = q;
    if (__builtin_expect(!ok, 0)) v = slow_div(a, b);
    return v;
}

// Seeds of the square root of x = m 4^k, m in [1, 4): the root s of the leading float, corrected by
// the residual (m + the rest) - s^2, and 1/sqrt(x) as a float with its exponent.
struct RootSeed {
    double s;   // sqrt(x) to a relative 2^-42
    double h;   // 1/(2 sqrt(x)) to float accuracy
    float y, c, f;  // 1/sqrt(m), the correction of the root f of m
    uint32_t e;     // -k in the exponent field
};
__device__ __forceinline__ RootSeed root_seed(double x) {
    const uint32_t hi = hi32(x);
    const uint32_t odd = (~hi >> 20) & 1u;  // the exponent E (field - 1023) is odd: m = 2 * 1.f
    const float sc = odd ? 2.0f : 1.0f;
    const float m = frac_hi(x) * sc, l = frac_lo(x) * (sc * 0x1p-23f);
    const uint32_t k2 = (hi - 0x3FF00000u - (odd << 20)) & 0xFFE00000u;  // 2 k, in the place of the exponent
    const uint32_t kf = static_cast<uint32_t>(static_cast<int32_t>(k2) >> 1);
    RootSeed r;
    r.y = rsqrt_approx(m);
    r.f = fminf(fmaxf(m * r.y, 1.0f), 2.0f);
    const float t = fmaf(-r.f, r.f, m) + l;
    r.c = 0.5f * r.y * t;
    r.s = join(r.f, round_int(r.c * 0x1p42f), kf);
    r.e = 0u - kf;
    r.h = from32((__float_as_uint(r.y) >> 3) + 0x38000000u - 0x00100000u + r.e, __float_as_uint(r.y) << 29);
    return r;
}
// 1/sqrt(x) to a relative 2^-42 from the seeds: y corrected by 1 - y (f + c)
__device__ __forceinline__ double inv_root_seed(const RootSeed& r) {
    const float y = fminf(fmaxf(r.y, 0.5f), 1.0f);
    const float e = fmaf(-r.c, y, fmaf(-r.f, y, 1.0f));
    return join(y, round_int(y * e * 0x1p43f), r.e);
}
__device__ __forceinline__ bool root_range(double x) { return (hi32(x) >> 20) - 64u < 1920u; }  // positive, mid range

// sqrt(x): the seed corrected by its exact residual x - s^2 (half an ulp plus 2^-12 of one at most)
__device__ __forceinline__ double sqrt(double x) {
    const RootSeed r = root_seed(x);
    double s = fma(fma(-r.s, r.s, x), r.h, r.s);
    if (__builtin_expect(!root_range(x), 0)) s = slow_sqrt(x);
    return s;
}
// 1/sqrt(x): the seed cut to 26 bits, so that its square is exact and e = 1 - x y^2 carries one
// rounding; then y (1 + e/2 + 3 e^2/8), the last term (below 2^-49) in FP32
__device__ __forceinline__ double rsqrt(double x) {
    const double s = inv_root_seed(root_seed(x));
    const double y = from32(hi32(s), lo32(s) & 0xF8000000u);
    const double e = fma(-x, __dmul_rn(y, y), 1.0);
    const float ef = narrow(e), t = 0.75f * ef * ef;
    double v = fma(scale2(y, -1), __dadd_rn(e, widen_or_zero(t)), y);
    if (__builtin_expect(!root_range(x), 0)) v = slow_rsqrt(x);
    return v;
}
// sqrt(x) and 1/sqrt(x), the reciprocal that of the rounded root
__device__ __forceinline__ double sqrt_rcp(double x, double& inv) {
    const RootSeed r = root_seed(x);
    double s = fma(fma(-r.s, r.s, x), r.h, r.s);
    const double y = inv_root_seed(r);
    inv = fma(y, fma(-s, y, 1.0), y);
    if (__builtin_expect(!root_range(x), 0)) {
        s = slow_sqrt(x);
        inv = slow_div(1.0, s);
    }
    return s;
}

// ---------------------------------------------------------------- exponentials
// v = (256 q + j) ln2/256 + r, |r| <= ln2/512: exp(v) = 2^q 2^(j/256) (1 + p), p = exp(r) - 1, and
// T = 2^q 2^(j/256) as a pair (the low part keeps the table's rounding out of the result).
struct ExpParts {
    double t, l, r;
    float rf;
};
__device__ __forceinline__ ExpParts exp_parts(double v) {  // |v| < 600
    const float kf = narrow(v) * 0x1.715476p+8f + 12582912.0f;  // 256/ln2
    const int k = __float_as_int(kf) - 0x4B400000;
    const double kd = widen_int(kf - 12582912.0f);
    ExpParts e;
    e.r = fma(-kd, kExpStepLo, fma(-kd, kExpStepHi, v));
    e.rf = narrow(e.r);
    const double2 t = __ldg(reinterpret_cast<const double2*>(kExpTab) + (k & 255));
    const int q = k >> 8;
    e.t = scale2(t.x, q);
    e.l = (k & 255) ? scale2(t.y, q) : 0.0;
    return e;
}
__device__ __forceinline__ bool exp_range(double v) { return (hi32(v) & 0x7FFFFFFFu) < 0x4082C000u; }  // |v| < 600
// p = r + r^2 (1/2 + r c), c = 1/6 + r/24 + r^2/120 in FP32 (its error enters at 2^-55 of the result)
__device__ __forceinline__ double exp(double v) {
    const ExpParts e = exp_parts(v);
    const double c = widen(fmaf(e.rf, fmaf(e.rf, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f));
    double x = __dadd_rn(e.t, fma(e.t, fma(__dmul_rn(e.r, e.r), fma(e.r, c, 0.5), e.r), e.l));
    if (__builtin_expect(!exp_range(v), 0)) x = slow_exp(v);
    return x;
}
// exp(v + w) for a correction w of a few ulps of v (the low part of a product)
__device__ __forceinline__ double exp(double v, double w) {
    const ExpParts e = exp_parts(v);
    const double r = __dadd_rn(e.r, w);
    const double c = widen(fmaf(e.rf, fmaf(e.rf, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f));
    double x = __dadd_rn(e.t, fma(e.t, fma(__dmul_rn(r, r), fma(r, c, 0.5), r), e.l));
    if (__builtin_expect(!exp_range(v), 0)) x = slow_exp(v, w);
    return x;
}
// exp(v) - 1: T - 1 is exact where it cancels (T in [1/2, 2]) and 0 for j = q = 0; the result may be
// as small as r, so FP32 begins one term later than in exp
__device__ __forceinline__ double expm1(double v) {
    const ExpParts e = exp_parts(v);
    const double c = widen(fmaf(e.rf, fmaf(e.rf, 1.0f / 720.0f, 1.0f / 120.0f), 1.0f / 24.0f));
    const double p = fma(__dmul_rn(e.r, e.r), fma(e.r, fma(e.r, c, 1.0 / 6.0), 0.5), e.r);
    double x = __dadd_rn(__dadd_rn(e.t, -1.0), fma(e.t, p, e.l));
    if (__builtin_expect(!exp_range(v), 0)) x = slow_expm1(v);
    return x;
}

// ---------------------------------------------------------------- logarithms
// u = m 2^E, m in [1, 2), c the float nearest 1/m on a grid of 256 points: r = m c - 1 (|r| <= 2^-9),
// log u = E ln2 - log c + log1p(r), log1p(r) = r + r^2 (-1/2 + r (1/3 + r g)), g = -1/4 + r/5 - r^2/6
// + r^3/7 in FP32.  E ln2 and -log c have heads on one grid of 2^-41, so their sum is exact; at u near
// 1 it is 0 and r alone is left.  `w` 2^-E is added to m first (log1p's low part).
__device__ __forceinline__ double log_tail(double u, double w, bool with_w) {  // u normal and positive
    const uint32_t hi = hi32(u);
    const int j = static_cast<int>(((hi & 0xFFFFFu) + 0x800u) >> 12);
    const int E = static_cast<int>(hi >> 20) - 1023;
    const double m = from32((hi & 0xFFFFFu) | 0x3FF00000u, lo32(u));
    const double c = widen(__ldg(&kLogInv[j]));
    const double2 t = __ldg(reinterpret_cast<const double2*>(kLogTab) + j);
    const double Ed = widen_int(__int_as_float(0x4B400000 + E) - 12582912.0f);
    double r = fma(m, c, -1.0);
    if (with_w) r = fma(w, c, r);
    const float rf = narrow(r);
    const double g = widen(fmaf(rf, fmaf(rf, fmaf(rf, 1.0f / 7.0f, -1.0f / 6.0f), 0.2f), -0.25f));
    const double p = fma(__dmul_rn(r, r), fma(r, fma(r, g, 1.0 / 3.0), -0.5), r);
    return __dadd_rn(fma(Ed, kLn2Hi, t.x), __dadd_rn(fma(Ed, kLn2Lo, t.y), p));
}
__device__ __forceinline__ double log(double x) {
    double v = log_tail(x, 0.0, false);
    if (__builtin_expect((hi32(x) >> 20) - 1u >= 2046u, 0)) v = slow_log(x);  // zero, subnormal, negative, inf, NaN
    return v;
}
// log(1 + y) for y in [2^-960, 2^900): u = 1 + y rounded, its rounding error w by a two-sum
__device__ __forceinline__ double log1p(double y) {
    const bool big = hi32(y) >= 0x3FF00000u;
    const double a = big ? y : 1.0, b = big ? 1.0 : y;
    const double u = __dadd_rn(a, b), w = __dadd_rn(b, -__dadd_rn(u, -a));
    // w 2^-E
    const double ws = (hi32(w) << 1 | lo32(w)) == 0u ? 0.0 : from32(hi32(w) - ((hi32(u) & 0x7FF00000u) - 0x3FF00000u), lo32(w));
    double v = log_tail(u, ws, true);
    if (__builtin_expect(hi32(y) - 0x03F00000u >= 0x74400000u, 0)) v = slow_log1p(y);  // also 0, negative, inf, NaN
    return v;
}

// ---------------------------------------------------------------- arc tangent
// atan2(y, x) for y >= 0: with (n, d) = (y, |x|) or (|x|, y) so that n <= d, the table point c = k/64
// nearest n/d, t = (n - c d)/(d + c n) = tan(atan(n/d) - atan c), |t| <= 1/127, and
// atan t = t + t^3 (-1/3 + t^2 g), g = 1/5 - t^2/7 + t^4/9 in FP32; the octant's base angle plus or minus
// atan c is a table pair.
__device__ __forceinline__ double atan2(double y, double x) {
    const double ax = __longlong_as_double(__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFLL);
    const bool swap = __double_as_longlong(y) > __double_as_longlong(ax), neg = __double_as_longlong(x) < 0;
    const double n = swap ? ax : y, d = swap ? y : ax;
    const float cf = rintf(fminf(fmaxf(narrow(n) * rcp_approx(narrow(d)) * 64.0f, 0.0f), 64.0f));  // NaN: 0
    const int k = static_cast<int>(cf);
    const double c = widen_int(cf * 0.015625f);
    const double t = div(fma(-c, d, n), fma(c, n, d));
    const int q = neg ? (swap ? 2 : 3) : (swap ? 1 : 0);
    const double2 b = __ldg(reinterpret_cast<const double2*>(kAtanTab) + (65 * q + k));
    const double t2 = __dmul_rn(t, t);
    const float t2f = narrow(t2);
    const double g = widen(fmaf(t2f, fmaf(t2f, 1.0f / 9.0f, -1.0f / 7.0f), 0.2f));
    const double a = fma(__dmul_rn(t, t2), fma(t2, g, -1.0 / 3.0), t);
    double v = __dadd_rn(b.x, __dadd_rn(b.y, (q & 1) ? -a : a));
    // y >= 0 and d a float normal with room (2^-100 .. 2^100): otherwise CUDA's
    if (__builtin_expect(!(hi32(d) - 0x39B00000u < 0x0C800000u && hi32(y) < 0x80000000u), 0)) v = slow_atan2(y, x);
    return v;
}

// atan(a), as atan2 of |a| and 1
__device__ __forceinline__ double atan(double a) {
    const long long b = __double_as_longlong(a), sign = b & static_cast<long long>(0x8000000000000000ULL);
    return __longlong_as_double(__double_as_longlong(atan2(__longlong_as_double(b ^ sign), 1.0)) ^ sign);
}

// ---------------------------------------------------------------- integer powers
// The sums S_k(u) = 1 + u + ... + u^(k-1) = (u^k - 1)/(u - 1), k = n - 1 and n, of u >= 1 (no cancellation)
__device__ __forceinline__ void geometric(double u, int n, double& s_prev, double& s_n) {
    s_prev = 1.0;
    s_n = __dadd_rn(u, 1.0);
#pragma unroll
    for (int k = 3; k <= kMaxPower; ++k)
        if (k <= n) {
            s_prev = s_n;
            s_n = fma(s_n, u, 1.0);
        }
}
// rho = (1 + p)^(1/n) - 1, p in [2^-60, 2^100), n in 2..kMaxPower: the root of rho S_n(1 + rho) = p.  A FP32
// seed (series below 1/16, else exp2 of log2) and one FP32 Newton step bring it to 2^-20 or better; one
// Halley step in FP64, third order, ends it.  11 FP64 instructions.
__device__ __forceinline__ double root1p(double p, int n) {
    const float pf = narrow(p), nf = static_cast<float>(n), in = rcp_approx(nf);
    const float q = pf * in;
    const float small = q * fmaf(-0.5f * (nf - 1.0f) * q, fmaf(-(2.0f * nf - 1.0f) * (1.0f / 3.0f), q, 1.0f), 1.0f);
    float rf = pf < 0.0625f ? small : ex2_approx(lg2_approx(1.0f + pf) * in) - 1.0f;
    const float uf = 1.0f + rf;
    float sp = 1.0f, sn = uf + 1.0f;
#pragma unroll
    for (int k = 3; k <= kMaxPower; ++k)
        if (k <= n) {
            sp = sn;
            sn = fmaf(sn, uf, 1.0f);
        }
    rf = fmaf(-fmaf(rf, sn, -pf), rcp_approx(nf * fmaf(rf, sp, 1.0f)), rf);
    const double r = widen(rf);
    const double u = __dadd_rn(1.0, r);
    double s_prev, s_n;
    geometric(u, n, s_prev, s_n);
    const double f = fma(r, s_n, -p);
    const double d = __dmul_rn(widen(nf), fma(r, s_prev, 1.0));  // the derivative n u^(n-1)
    const double c = __dmul_rn(f, rcp_seed(d));
    const float t = 0.5f * (nf - 1.0f) * narrow(c) * rcp_approx(1.0f + rf);
    return __dadd_rn(r, -fma(c, widen_or_zero(t), c));
}

// The exponent w = 1 - nu of a power law, near 1/n for an integer n: n w = 1 - eta.
struct WholePower {
    int n;
    double nd;  // n
    float eta;
    bool ok;    // 2 <= n <= kMaxPower and |eta| < 1e-13
};
__device__ __forceinline__ WholePower whole_power(double w, bool constant) {  // constant: of a compiled channel, folds
    WholePower p;
    const float wf = constant ? static_cast<float>(w) : narrow(w);
    const float nf = rintf(constant ? 1.0f / wf : rcp_approx(wf));
    const bool near = wf > 0.15f && wf < 0.55f && fabsf(fmaf(-nf, wf, 1.0f)) < 1e-6f;
    p.nd = constant ? static_cast<double>(nf) : widen(near ? nf : 1.0f);
    const double eta = fma(-p.nd, w, 1.0);
    p.eta = constant ? static_cast<float>(eta) : narrow(eta);
    p.n = static_cast<int>(nf);
    p.ok = near && fabsf(p.eta) < 1e-13f;
    return p;
}
__device__ __forceinline__ bool root_arg(double p) { return hi32(p) - 0x3C300000u < 0x0A000000u; }  // [2^-60, 2^100)
// (1 + p)^w - 1, root_arg(p): (1 + p)^-eta to first order moves p by -eta (1 + p) log(1 + p)
__device__ __forceinline__ double power_root(double p, const WholePower& k) {
    const float pf = narrow(p);
    const float dp = k.eta * (1.0f + pf) * (0.693147181f * lg2_approx(1.0f + pf));
    return root1p(k.eta != 0.0f ? __dadd_rn(p, -widen_or_zero(dp)) : p, k.n);
}

// ---------------------------------------------------------------- powers
// log x of a positive normal x as a head on the grid of 2^-41 and a rest (below 2^-8) good to 2^-61
__device__ __forceinline__ void log_pair(double x, double& head, double& rest) {
    const uint32_t hi = hi32(x);
    const int j = static_cast<int>(((hi & 0xFFFFFu) + 0x800u) >> 12);
    const double m = from32((hi & 0xFFFFFu) | 0x3FF00000u, lo32(x));
    const double2 t = __ldg(reinterpret_cast<const double2*>(kLogTab) + j);
    const double Ed = widen_int(__int_as_float(0x4B400000 + static_cast<int>(hi >> 20) - 1023) - 12582912.0f);
    const double r = fma(m, widen(__ldg(&kLogInv[j])), -1.0);
    const float rf = narrow(r);
    const double g = widen(fmaf(rf, fmaf(rf, fmaf(rf, 1.0f / 7.0f, -1.0f / 6.0f), 0.2f), -0.25f));
    head = fma(Ed, kLn2Hi, t.x);
    rest = __dadd_rn(fma(Ed, kLn2Lo, t.y), fma(__dmul_rn(r, r), fma(r, fma(r, g, 1.0 / 3.0), -0.5), r));
}
// exp(a (head + rest)): the product as a pair
__device__ __forceinline__ double exp_of(double a, double head, double rest) {
    const double v = __dmul_rn(a, head), w = fma(a, rest, fma(a, head, -v));
    const double s = __dadd_rn(v, w);
    return exp(s, __dadd_rn(w, -__dadd_rn(s, -v)));
}

}  // namespace fast
}  // namespace dev
}  // namespace ps
