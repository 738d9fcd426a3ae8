// soft64.cuh -- correctly rounded binary64 products and quotients on the integer
// pipes, for the FP64 direct sum.  On GB300 one FP64 instruction holds a scheduler's FP64
// unit for 76 cycles a warp (a conversion from FP32 64, a division about 17 such
// operations), an integer instruction for 1 to 2: formed from 32-bit multiplications and
// additions, the same IEEE results cost a fraction, and the FP64 unit is free for the
// sums that stay on it.
//
// A positive normal number is held as N 2^(e - 63): N a 64-bit significand with its top bit
// set, of whose bits the top 53 are used (the rest zero), and e the unbiased exponent.
// Every result below is the nearest such number to the exact one, ties to even, exactly as
// the IEEE operation's (exponents are kept far from overflow and underflow by the
// caller).
#pragma once

#include <stdint.h>

namespace mlens {

struct Soft64 {
    uint64_t n;
    int e;
};

// Nearest 53-bit significand to n, n >= 2^63 (bit 0 may stand for any lower bits: sticky).
__host__ __device__ __forceinline__ Soft64 soft_round(uint64_t n, int e)
{
    // half less one, plus the last kept bit: ties to even.  A carry out leaves the top
    // bit clear (and every kept bit): the significand is then 2^63 and the exponent one more.
    const uint64_t r = n + 0x3ffu + ((n >> 11) & 1u);
    return {(r & ~uint64_t(0x7ff)) | uint64_t(1) << 63, e + 1 - (int)(r >> 63)};
}

// a * b from the top 64 bits of the product of two normalised significands and a sticky
// bit for the rest; e = the exponents' sum.
__host__ __device__ __forceinline__ Soft64 soft_product(uint64_t hi, bool rest, int e)
{
    const uint64_t n = hi | (rest ? 1u : 0u);
    const int top = (int)(n >> 63);
    return soft_round(n << (1 - top), e + top);
}

__host__ __device__ __forceinline__ Soft64 soft_square(Soft64 a)
{
    const unsigned __int128 p = (unsigned __int128)a.n * a.n;
    return soft_product((uint64_t)(p >> 64), (uint64_t)p != 0u, 2 * a.e);
}

// a * m, m a 32-bit significand with its top bit set and exponent em (a float's value)
__host__ __device__ __forceinline__ Soft64 soft_mul32(Soft64 a, uint32_t m, int em)
{
    const uint64_t lo = (uint64_t)(uint32_t)a.n * m;
    const uint64_t hi = (a.n >> 32) * m + (lo >> 32);
    return soft_product(hi, (uint32_t)lo != 0u, a.e + em);
}

// 2^127 / b to within (-5, 0], from a float estimate y of 2^63 / b in [1/2, 1) (relative error
// below 2^-21) and two Newton steps y <- y + y (1 - b y), the first on 32-bit words.
__host__ __device__ __forceinline__ uint64_t soft_reciprocal(uint64_t b, uint32_t y_bits)
{
    const uint32_t r0 = (y_bits << 8) | 0x80000000u;  // y 2^32
    const uint64_t lo = (uint64_t)(uint32_t)b * r0;
    const uint64_t h0 = (b >> 32) * r0 + (lo >> 32);  // b y 2^63
    const int32_t e0 = (int32_t)((int64_t)((uint64_t(1) << 63) - h0) >> 11);
    const uint64_t r1 = ((uint64_t)r0 << 32) + (uint64_t)(((int64_t)(int32_t)(r0 >> 1) * e0) >> 19);
    const uint64_t h1 = (uint64_t)(((unsigned __int128)b * r1) >> 64);
    const int32_t e1 = (int32_t)(int64_t)((uint64_t(1) << 63) - h1);
    return r1 + (uint64_t)(((int64_t)(int32_t)(r1 >> 33) * e1) >> 30) - 3u;
}

// a / b with r = soft_reciprocal(b): q = a r is within (-12, 0] of the quotient in units of
// 2^-63 (normalised), so only a q less than 12 below a rounding midpoint needs the exact
// comparison, the sign of a - midpoint b (never zero: a quotient of two 53-bit significands
// is not a midpoint).
__host__ __device__ __forceinline__ Soft64 soft_div(Soft64 a, Soft64 b, uint64_t r)
{
    const uint64_t q = (uint64_t)(((unsigned __int128)a.n * r) >> 64);
    const int top = (int)(q >> 63);
    uint64_t n = q << (1 - top);
    const int e = a.e - b.e - 1 + top;
    const uint32_t low = (uint32_t)n & 0x7ffu;
    n &= ~uint64_t(0x7ff);
    bool up = low >= 0x400u;
    if (low - (0x400u - 12u) < 12u) {
        const uint64_t mid = (n >> 10) | 1u;  // 54 bits
        up = (int64_t)(((a.n >> 11) << (54 - top)) - mid * (b.n >> 11)) > 0;
    }
    n += up ? 0x800u : 0u;
    return {n | uint64_t(1) << 63, e + 1 - (int)(n >> 63)};  // as in soft_round
}

// A positive normal number's binary64 bits, and back.
__host__ __device__ __forceinline__ Soft64 soft_of(uint64_t bits)
{
    return {bits << 11 | uint64_t(1) << 63, (int)((uint32_t)(bits >> 52) & 0x7ffu) - 1023};
}

__host__ __device__ __forceinline__ uint64_t soft_bits(Soft64 a, uint64_t sign)
{
    return sign | (((uint64_t)(a.e + 1022) << 52) + (a.n >> 11));  // the significand's top bit adds 1 to the exponent field
}

}  // namespace mlens
