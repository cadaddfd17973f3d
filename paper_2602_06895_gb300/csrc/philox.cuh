// philox.cuh -- Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) for the device code of the
// phase-space library: ten rounds of two 32x32->64 multiplies with the Weyl key schedule.
#pragma once
#include <cstdint>

namespace ps {
namespace rng {

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int i = 0; i < 10; ++i) {
        uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// (k + 1/2) 2^-52 for the top 52 bits k of (hi:lo), exactly: the odd integer 2k + 1 < 2^53 in units of
// 2^-53, its leading bit moved to bit 52 and the exponent set by the integer ALU (no FP64 instruction).
__device__ __forceinline__ double unit_from_bits(uint32_t hi, uint32_t lo) {
    const unsigned long long m = (((static_cast<unsigned long long>(hi) << 32) | lo) >> 11) | 1ULL;
    const int lz = __clzll(static_cast<long long>(m));  // 11..63
    // the leading bit adds one to the exponent field
    return __longlong_as_double(static_cast<long long>((m << (lz - 11)) + (static_cast<unsigned long long>(1032 - lz) << 52)));
}

// The float form of a point coordinate, for the mixed-precision programs: (k + 1/2) 2^-23 for the
// top 23 bits k of hi, exactly: the float 1 + k 2^-23 assembled from bits minus (1 - 2^-24),
// exact by Sterbenz's lemma.  It lies in the same 2^-23 cell as the double form, so every VEGAS
// bin and grid cell agrees with it.
__device__ __forceinline__ float unit_from_bits_f(uint32_t hi) {
    const float one_plus = __int_as_float(0x3F800000u | (hi >> 9));
    return one_plus - 0x1.fffffep-1f;
}

}  // namespace rng
}  // namespace ps
