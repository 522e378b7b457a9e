// Correctly rounded division by 6 for the 3D update (rbgs3d.cu), on the integer pipes.
// __host__ __device__ so that the host test harness checks it against IEEE division.
#pragma once

#include <cmath>
#include <cstdint>

#include "fp64.cuh"

namespace rbgs {

// s / 6 correctly rounded, in about 22 integer operations.  GB300 issues 2 FP64 instructions
// per clock and SM and some 90 integer ones, so the two or three FP64 operations of a
// division by multiplication and correction cost more than this.
//
// s = +-M 2^(E-1075) with the 53-bit significand M, so s / 6 = +-(M / 3) 2^(E-1076).  With
// X = M 2^10 < 2^63, Z = floor(X / 3) has 61 or 62 bits, so at least 8 more than a
// significand.  X / 3 in 32-bit limbs: the high limb gives a quotient and a remainder r < 3;
// (r 2^32 + lo) / 3 = r 0x55555555 + (r + lo) / 3, since 2^32 = 3 0x55555555 + 1, and r + lo
// does not overflow as the low 10 bits of lo are zero.  The quotient is rounded by adding
// half of its last place: a tie would need M / 3 to end on exactly half a place, that is
// M to be 3 times an odd number of 54 or more bits, so there is none, and the fraction that
// the floor dropped cannot turn a value below half into one above.
//
// Biased exponents 0..3 (results in or next to the subnormal range) and 2047 (Inf, NaN: s / 6 =
// s) go through div6_special, on the device behind a vote of the active lanes.  It is integer
// work too, and an opaque move keeps it behind the branch: the compiler moves a division
// instruction there above the vote, and every update then pays for it (20 FP64 instructions in
// all instead of 6).  Zeros are returned as they are.
__host__ __device__ __forceinline__ uint32_t third_u32(uint32_t x) {
#if defined(__CUDA_ARCH__)
    return __umulhi(x, 0xAAAAAAABu) >> 1;
#else
    return (uint32_t)(((uint64_t)x * 0xAAAAAAABull) >> 33);
#endif
}

// Biased exponent 0..3 or 2047.  In units of 2^-1074, s = N = M 2^(max(e, 1) - 1) with M the
// significand, and N / 6 < 2^53, where the encoding counts those units: the bits of s / 6 are
// N / 6 rounded half to even.
__host__ __device__ __forceinline__ uint64_t div6_special(uint64_t u) {
    const uint32_t e = (uint32_t)(u >> 52) & 0x7FFu;
    if (e == 0x7FFu) return u;
    const uint64_t m = (u & 0x000FFFFFFFFFFFFFull) | (e ? 0x0010000000000000ull : 0ull);
    const uint64_t nn = m << (e ? e - 1u : 0u);
    uint64_t q = nn / 6u;
    const uint32_t rem = (uint32_t)(nn - 6u * q);
    if (rem > 3u || (rem == 3u && (q & 1u))) ++q;
    return (u & 0x8000000000000000ull) | q;
}

__host__ __device__ __forceinline__ double div6(double s) {
    const uint64_t u = dbits(s);
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
    const uint32_t e = (hi >> 20) & 0x7FFu;
    const uint32_t xh = (((hi & 0xFFFFFu) | 0x100000u) << 10) | (lo >> 22), xl = lo << 10;
    const uint32_t zh = third_u32(xh), r = xh - 3u * zh;
    const uint32_t zl = r * 0x55555555u + third_u32(xl + r);
    const uint32_t t = (zh >> 29) & 1u;  // 1: Z has 62 bits
    const uint64_t z = ((((uint64_t)zh << 32) | zl) + (128u << t)) >> (8u + t);
    // the significand's hidden bit adds one to the exponent field: e - 3 + t in all
    const uint64_t mag = z + ((uint64_t)((e + t - 4u) << 20) << 32);
    double q = bitsd(mag | ((uint64_t)(hi & 0x80000000u) << 32));
    const bool zero = ((hi << 1) | lo) == 0u;  // on the halves: a 64-bit test becomes an FP64 compare
    if (zero) q = s;
    const bool ok = e - 4u <= 2042u || zero;
#if defined(__CUDA_ARCH__)
    if (__any_sync(__activemask(), !ok))
#endif
    {
        if (!ok) {
            uint64_t v = u;
#if defined(__CUDA_ARCH__)
            asm volatile("mov.b64 %0, %1;" : "=l"(v) : "l"(u));  // keeps the rare path behind the branch
#endif
            q = bitsd(div6_special(v));
        }
    }
    return q;
}

}  // namespace rbgs
