// Fixed-point forms of FP64 vectors: a vector scaled by a power of two to integers F
// with ||F||_2 <= 2^bits, so that an inner product of two such vectors is an integer
// below 2^(2 bits) (Cauchy-Schwarz).  Integer and FP32 instructions only.
//
// `s` below is a power of two that an element is multiplied by first (crt.cu balances
// the two halves of a stacked operand with it).
#pragma once

#include <limits.h>
#include <stdint.h>

namespace omm {

// Exponent of a vector that has no fixed-point form here: it holds a NaN or an infinity,
// or nothing above 2^-895 (2^smax times that: smax, the largest shift), where elements in
// FP64's underflow range would count.
constexpr int kUnscaled = INT_MIN;

// Ordered code of an element's exponent: 0 for zero, 1 for a subnormal, kCodeInf for a NaN
// or an infinity, else the biased exponent of v 2^s plus kCodeBias.  The code of a vector is
// the largest of its elements'.
constexpr int kCodeBias = 8192, kCodeInf = 1 << 20;
constexpr int kShiftMax = 2000;   // |s| is at most this

__device__ __forceinline__ int fx_code(uint64_t b /* sign cleared */, int s) {
    const int be = (int)(b >> 52);
    return be == 0x7FF ? kCodeInf : (be != 0 ? be + s + kCodeBias : (b != 0 ? 1 : 0));
}

// (v 2^(s - X))^2 in FP32 for v's magnitude bits b, X = code - kCodeBias - 1022 of the
// vector; zero and subnormal elements (far below the largest of a scaled vector) give 0
__device__ __forceinline__ float fx_square(uint64_t b, int s, int code) {
    const int be = (int)(b >> 52);
    const int e = be + s + kCodeBias - code + 126;
    if (be == 0 || e <= 0) return 0.f;   // below 2^-126 of the largest: nothing of the sum
    const float f = __uint_as_float(((uint32_t)e << 23) | (uint32_t)((b & 0xFFFFFFFFFFFFFull) >> 29));
    return f * f;
}

// Exponent e with v 2^s = F 2^e from the vector's code and S, its sum of fx_square:
// ||v|| <= 2^X sqrt(1.001 S) (the 1.001 covers the FP32 rounding of S), and 2^(bits - 1) <=
// ||F|| (but for that rounding).
__device__ __forceinline__ int fx_exponent(int code, float S, int bits, int smax) {
    if (code == 0) return 0;
    if (code >= kCodeInf || code < kCodeBias + 128 + smax) return kUnscaled;
    const float s = S * 1.001f;
    const int k = (int)((__float_as_uint(s) >> 23) & 0xFF) - 126;   // s < 2^k
    return code - kCodeBias - 1022 + ((k + 1) >> 1) - bits;
}

// F = round(v 2^(s - e)) in two's complement, |F| < 2^79: lo the low 64 bits, hi the rest
struct Fixed {
    uint64_t lo;
    int hi;
};
__device__ __forceinline__ Fixed fx_round(double v, int s, int e) {
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const int be = (int)((b >> 52) & 0x7FF);
    Fixed F{0, 0};
    if (be == 0 || e == kUnscaled) return F;
    const uint64_t mant = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);   // v = mant 2^(be - 1075)
    const int shift = be - 1075 + s - e;
    if (shift >= 0) {
        F.lo = mant << shift;
        F.hi = (int)((mant >> 1) >> (63 - shift));
    } else if (shift > -64) {
        F.lo = (mant + (1ull << (-shift - 1))) >> (-shift);
    }
    if (b >> 63) {
        F.lo = 0ull - F.lo;
        F.hi = ~F.hi + (F.lo == 0 ? 1 : 0);
    }
    return F;
}

// |v| 2^(s - e - bits), at most 1, cut to BF16 (its bits): never above, and 2^-60 instead of
// anything smaller but zero, so that it is zero for a zero alone
__device__ __forceinline__ uint32_t fx_magnitude(double v, int s, int e, int bits) {
    const uint64_t b = (uint64_t)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
    if (b == 0 || e == kUnscaled) return 0u;
    const int be = (int)(b >> 52);
    const int x = be - 1023 + s - e - bits + 127;
    return (be == 0 || x <= 67) ? 67u << 7 : ((uint32_t)x << 7) | (uint32_t)((b >> 45) & 0x7Fu);
}

}  // namespace omm
