// ratio.cuh -- the crowding distance's quotient (double)gap / (double)range,
// correctly rounded, in integer arithmetic.
//
// The GPU's FP64 pipe is narrow (two lanes' worth a cycle per SM), so the
// division instruction sequence of two objectives for 200 members took most
// of the crowding step; the same IEEE result comes from long division on the
// 53-bit significands in the integer pipe. Each of the three steps estimates
// a radix-2^18 (2^17) digit from single-precision leading parts and corrects
// it by at most one against the exact remainder.
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define MOCD_HD __host__ __device__ __forceinline__
#else
#define MOCD_HD inline
#endif

namespace mocd {

MOCD_HD int leading_zeros64(uint64_t x)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}

// x > 0 as significand * 2^exp with bit 52 of the significand set, rounded to
// nearest, ties to even (what (double)x holds).
MOCD_HD uint64_t significand53(uint64_t x, int &exp)
{
    const int shift = 11 - leading_zeros64(x);  // > 0: x has more than 53 bits
    exp = shift;
    if (shift <= 0) return x << -shift;
    uint64_t s = x >> shift;
    const uint64_t low = x & ((1ull << shift) - 1ull), half = 1ull << (shift - 1);
    s += (low > half || (low == half && (s & 1ull))) ? 1ull : 0ull;
    if (s >> 53) {
        s >>= 1;
        ++exp;
    }
    return s;
}

// One digit: rem < b (b has 53 bits) becomes rem * 2^BITS - digit * b in
// [0, b). The product is taken modulo 2^64, which is enough because the
// remainder before the correction lies in (-b, 2 b).
template <int BITS>
MOCD_HD uint64_t ratio_digit(uint64_t &rem, uint64_t b, float inv)
{
    // Leading 32 bits over leading 32 bits: the estimate's relative error is
    // below 2^-21, the digit's absolute error below 2^-3 before truncation.
    const float est = (float)(uint32_t)(rem >> 21) * inv * (float)(1 << BITS);
    uint64_t d = (uint64_t)(uint32_t)est;
    int64_t r = (int64_t)((rem << BITS) - d * b);
    if (r < 0) {
        r += (int64_t)b;
        --d;
    } else if ((uint64_t)r >= b) {
        r -= (int64_t)b;
        ++d;
    }
    rem = (uint64_t)r;
    return d;
}

// Bit pattern of (double)gap / (double)range rounded to nearest even, for
// 0 <= gap <= range, 0 < range < 2^63. The quotient is 0 or in [2^-63, 1], a
// normal number.
MOCD_HD uint64_t ratio_bits(int64_t gap, int64_t range)
{
    if (gap == 0) return 0;
    int ea, eb;
    uint64_t a = significand53((uint64_t)gap, ea);
    const uint64_t b = significand53((uint64_t)range, eb);
    int e = ea - eb;
    if (a < b) {
        a <<= 1;
        --e;
    }
    // a / b in [1, 2): the leading 1, then 53 more bits (the last one below
    // the significand's end) and the remainder decide the rounding.
    uint64_t rem = a - b;
    const float fb = (float)(uint32_t)(b >> 21);
#ifdef __CUDA_ARCH__
    const float inv = __fdividef(1.0f, fb);
#else
    const float inv = 1.0f / fb;
#endif
    uint64_t q = 1;
    q = (q << 18) + ratio_digit<18>(rem, b, inv);
    q = (q << 18) + ratio_digit<18>(rem, b, inv);
    q = (q << 17) + ratio_digit<17>(rem, b, inv);
    const uint64_t odd = (q >> 1) & 1ull;
    const uint64_t up = (q & 1ull) & ((rem != 0 ? 1ull : 0ull) | odd);
    const uint64_t s = (q >> 1) + up;  // 2^53 carries into the exponent below
    return ((uint64_t)(e + 1023 - 1) << 52) + s;
}

}  // namespace mocd
