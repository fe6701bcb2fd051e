// Fixed-point forms of FP64 vectors: a vector scaled by a power of two to integers F
// with ||F||_2 <= 2^bits, so that an inner product of two such vectors is an integer
// below 2^(2 bits) (Cauchy-Schwarz).  Integer and FP32 instructions only.
#pragma once

#include <limits.h>
#include <stdint.h>

namespace omm {

constexpr int kNonFinite = INT_MIN;   // exponent of a vector that holds a NaN or an infinity

// (a 2^-X)^2 in FP32 for a's magnitude bits b (sign cleared), 2^X > the largest |a|
__device__ __forceinline__ float fx_square(uint64_t b, int X) {
    const int e = (int)(b >> 52) - 1023 - X + 127;
    if (e <= 0) return 0.f;   // below 2^-126 of the largest: nothing of the sum
    const float f = __uint_as_float(((uint32_t)e << 23) | (uint32_t)((b & 0xFFFFFFFFFFFFFull) >> 29));
    return f * f;
}

// Exponent e with a = F 2^e from be, the biased exponent of the largest |a|, and S, the
// sum of (a 2^-X)^2 with X = be - 1022: ||a|| <= 2^X sqrt(1.001 S) (the 1.001 covers
// the FP32 rounding of S).
__device__ __forceinline__ int fx_exponent(int be, float S, int bits) {
    if (be == 0x7FF) return kNonFinite;
    if (be == 0) return 0;
    const float s = S * 1.001f;
    const int k = (int)((__float_as_uint(s) >> 23) & 0xFF) - 126;   // s < 2^k
    return be - 1022 + ((k + 1) >> 1) - bits;
}

// F = round(v 2^-e)
__device__ __forceinline__ int64_t fx_round(double v, int e) {
    const uint64_t b = (uint64_t)__double_as_longlong(v);
    const int be = (int)((b >> 52) & 0x7FF);
    if (be == 0 || e == kNonFinite) return 0;
    const uint64_t mant = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);   // v = mant 2^(be - 1075)
    const int shift = be - 1075 - e;
    int64_t F = 0;
    if (shift >= 0) F = (int64_t)(mant << shift);
    else if (shift > -64) F = (int64_t)((mant + (1ull << (-shift - 1))) >> (-shift));
    return (b >> 63) ? -F : F;
}

}  // namespace omm
