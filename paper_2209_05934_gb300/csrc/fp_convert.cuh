// Double <-> float conversion on the integer pipe.
//
// On GB300 a hardware FP64 -> FP32 conversion issues on the small FP64 unit
// (measured about 0.2 per clock per SM, ten times slower than an FP64 FMA),
// so kernels that convert every element become conversion-bound.  These
// versions take the IEEE-754 bit fields apart with integer instructions.
// d2f rounds to nearest, ties to even, exactly like the hardware conversion
// for every double of magnitude at least 2^-126 (the smallest normal float);
// a smaller magnitude gives a signed zero (the hardware would round to a
// subnormal float, or up to 2^-126), overflow gives a signed infinity, and a
// NaN gives a quiet NaN.  f2d is exact for every float, subnormals included
// (a NaN keeps its payload bits).
#pragma once

#include <stdint.h>

namespace omm {

__device__ __forceinline__ float sw_d2f(double d) {
    const uint64_t b = (uint64_t)__double_as_longlong(d);
    const uint32_t sign = (uint32_t)(b >> 32) & 0x80000000u;
    const int de = (int)((b >> 52) & 0x7FF);                 // biased double exponent
    const int e = de - 1023 + 127;                           // biased float exponent
    const uint64_t m = b & 0xFFFFFFFFFFFFFull;               // 52-bit fraction
    if (de == 0x7FF) return __uint_as_float(sign | 0x7F800000u | (m ? 0x400000u : 0u));  // inf / nan
    if (e <= 0) return __uint_as_float(sign);               // below 2^-126: signed zero
    if (e >= 255) return __uint_as_float(sign | 0x7F800000u);   // overflow: infinity
    uint32_t f = ((uint32_t)e << 23) | (uint32_t)(m >> 29);
    const uint32_t rem = (uint32_t)(m & 0x1FFFFFFFu);       // 29 dropped bits
    if (rem > 0x10000000u || (rem == 0x10000000u && (f & 1u))) f += 1u;   // may carry into the exponent
    return __uint_as_float(sign | f);
}

__device__ __forceinline__ double sw_f2d(float x) {
    const uint32_t u = __float_as_uint(x);
    const uint64_t sign = (uint64_t)(u & 0x80000000u) << 32;
    const uint32_t e = (u >> 23) & 0xFF;
    const uint64_t m = u & 0x7FFFFFu;
    if (e == 0) {
        if (m == 0) return __longlong_as_double((long long)sign);
        // subnormal float: normalise
        // m 2^-149 with the leading one at bit p = 23 - lz: 1.f x 2^(p - 149); shifting
        // by lz puts that one at bit 23, which the 23-bit mask then drops
        const int lz = __clz((int)m) - 8;                      // leading zeros inside the 24-bit field
        const uint64_t mm = (m << lz) & 0x7FFFFFull;
        const uint64_t ed = (uint64_t)(1023 - 126 - lz);
        return __longlong_as_double((long long)(sign | (ed << 52) | (mm << 29)));
    }
    if (e == 255) return __longlong_as_double((long long)(sign | (0x7FFull << 52) | (m << 29)));
    return __longlong_as_double((long long)(sign | ((uint64_t)(e - 127 + 1023) << 52) | (m << 29)));
}

// v * 2^e2 for a 64-bit integer v, rounded to nearest (ties to even); the
// caller keeps the result in the normal range (|v| 2^e2 between 2^-1000 and
// 2^1000).
__device__ __forceinline__ double sw_i64_scaled(int64_t v, int e2) {
    if (v == 0) return 0.0;
    const uint64_t sign = v < 0 ? (1ull << 63) : 0ull;
    const uint64_t a = v < 0 ? (0ull - (uint64_t)v) : (uint64_t)v;
    int p = 63 - __clzll((long long)a);                        // position of the leading one
    uint64_t q;
    if (p <= 52) {
        q = a << (52 - p);
    } else {
        const int sh = p - 52;
        q = a >> sh;
        const uint64_t rem = a & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
        if (rem > half || (rem == half && (q & 1ull))) {
            q += 1ull;
            if (q >> 53) {
                q >>= 1;
                ++p;
            }
        }
    }
    return __longlong_as_double((long long)(sign | ((uint64_t)(1023 + p + e2) << 52) | (q & 0xFFFFFFFFFFFFFull)));
}

// The same for a magnitude and a sign, without branches: the leading one to bit 63,
// then one rounded shift whose carry runs into the exponent.
__device__ __forceinline__ double sw_u64_scaled(uint64_t a, bool neg, int e2) {
    const int lz = __clzll((long long)a);
    const uint64_t n = a << (lz & 63);
    const uint64_t t = n + (0x3FFull + ((n >> 11) & 1ull));    // ties to even
    const uint64_t q = (t >> 11) + (t < n ? 1ull << 53 : 0ull);
    const uint64_t b = ((uint64_t)(1085 - lz + e2) << 52) + q;  // q's leading one adds one to the exponent
    return __longlong_as_double((long long)((a != 0 ? b : 0ull) | ((neg && a != 0) ? 1ull << 63 : 0ull)));
}

// x * 2^e by an exponent add when x and the result are normal; other cases
// (zero, subnormal, overflow, non-finite) go through ldexp.
__device__ __forceinline__ double sw_scale2(double x, int e) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int be = (int)((b >> 52) & 0x7FF);
    const int ne = be + e;
    if (be == 0 || be == 0x7FF || ne <= 0 || ne >= 0x7FF) return ldexp(x, e);
    return __longlong_as_double((long long)((b & ~(0x7FFull << 52)) | ((uint64_t)ne << 52)));
}

// root = sqrt(d) and rcp = 1 / root, both rounded to nearest like the hardware's own, for
// d > 0.  Integer Newton steps (Newton 1669 on s^2 = N and s q = 2^105, each ended by
// the exact remainder in 64-bit wrap-around arithmetic): with d = N 2^(2k - 104), N in
// [2^104, 2^106), the root's significand is the integer nearest to sqrt(N).  From FP32 seeds h and y
// = 1 / sqrt(x) good to 2^-22, one step gives ~2^-45 of s, the next its last bit or
// that +- 1, which the remainder decides: -s < N - s^2 <= s, and |2 (2^105 - q s)| <= s
// (neither has ties).  ~25 dependent integer instructions of 4 - 5 cycles each for both, where the
// FP64 forms are ~20 dependent FP64 instructions of 64 cycles and queue for
// the FP64 unit.
__device__ __forceinline__ void sw_sqrt_rcp(double d, double &root, double &rcp) {
    const uint64_t b = (uint64_t)__double_as_longlong(d);
    const int e = (int)((b >> 52) & 0x7FF);
    uint64_t man = b & 0xFFFFFFFFFFFFFull;
    int ex = e - 1023;
    if (e == 0) {   // subnormal
        const int sh = __clzll((long long)man) - 11;
        man <<= sh;
        ex = -1022 - sh;
    }
    man |= 1ull << 52;
    const int odd = ex & 1, k = (ex - odd) >> 1;                  // root in [2^k, 2^(k + 1)]
    const uint64_t lo = man << (52 + odd);                        // N mod 2^64; N >> 43 = man << (9 + odd)
    const float x = __uint_as_float(((uint32_t)(man >> 29) & 0x7FFFFFu) | ((uint32_t)(125 + odd) << 23));   // [1/4, 1)
    float y = rsqrtf(x);
    y = fmaf(0.5f * y, fmaf(-(x * y), y, 1.0f), y);
    y = fminf(fmaxf(y, 1.0f), 1.9999999f);
    float h = x * y;
    h = fmaf(0.5f * y, fmaf(-h, h, x), h);
    h = fminf(fmaxf(h, 0.5f), 0.99999994f);
    const uint32_t h24 = (__float_as_uint(h) & 0x7FFFFFu) | 0x800000u;   // h 2^24
    const uint32_t y24 = (__float_as_uint(y) & 0x7FFFFFu) | 0x800000u;   // y 2^23
    const int y31 = (int)(y24 << 7);                                     // y 2^30
    // the steps' corrections are rem / (2 s) = rem y 2^-54 and rem / s; the upper halves of
    // the remainders stay below 2^31 (a seventh of it at most)
    const int64_t r0 = (int64_t)((man << (9 + odd)) - (((uint64_t)h24 * h24) << 15));   // (N - s^2) >> 43
    int64_t s = (int64_t)((uint64_t)h24 << 29) + (((int64_t)(int)(r0 >> 10) * y31) >> 31);
    int64_t r = (int64_t)(lo - (uint64_t)s * (uint64_t)s);
    s += ((int64_t)(int)(r >> 31) * y31 + (1ll << 52)) >> 53;
    r = (int64_t)(lo - (uint64_t)s * (uint64_t)s);
    s += (r > s ? 1 : 0) - (r <= -s ? 1 : 0);
    int64_t t = (int64_t)(0ull - (uint64_t)y24 * (uint64_t)s);                          // (2^105 - q s) >> 29
    int64_t q = (int64_t)((uint64_t)y24 << 29) + (((int64_t)(int)(t >> 24) * y31) >> 30);
    t = (int64_t)(0ull - (uint64_t)q * (uint64_t)s);
    q += ((int64_t)(int)(t >> 31) * y31 + (1ll << 51)) >> 52;
    t = (int64_t)(0ull - (uint64_t)q * (uint64_t)s);
    q += (2 * t > s ? 1 : 0) - (2 * t < -s ? 1 : 0);
    // a significand of 2^53 carries into the exponent
    root = __longlong_as_double((long long)(((uint64_t)(k + 1022) << 52) + (uint64_t)s));
    rcp = __longlong_as_double((long long)(((uint64_t)(1021 - k) << 52) + (uint64_t)q));
    if (e == 0x7FF) {   // infinite
        root = d;
        rcp = 0.0;
    }
}

}  // namespace omm
