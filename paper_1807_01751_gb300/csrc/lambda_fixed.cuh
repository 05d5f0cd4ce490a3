// Box-Muller normals in 64-bit fixed point.
//
// FP64 instructions issue at 1/64 of the 32-bit integer and float rate on this
// chip, and a Box-Muller normal takes some eighty of them (log, sqrt, cos).  Here
// the normal is evaluated with 32-bit integer multiplies on 64-bit fixed-point
// words instead.  Against extended precision, over 3e6 draws with the ends of both
// ranges among them, its largest error is 7.9e-17 and the mean 2.6e-18; the same
// formula in FP64 is off by up to 5.7e-15 and by 2.0e-16 on average.  (-ln u has steps of
// 2^-58, so just below u = 1 - 2^-12, where it is smallest, FP64 is the more
// exact: mean errors of the normal 2.1e-17 and 3.2e-18.)
//
//   -ln u    u = n 2^-53, n = M 2^(e-52) with M in [2^52, 2^53).  An 11-bit
//            reciprocal c of M's top 9 bits makes M c = 2^63 (1 + r) an exact
//            64-bit product with |r| < 2^-8.6, and
//            -ln u = (53 - e) ln 2 - (-ln(c / 2^11)) - ln(1 + r), the middle term
//            from a table of 256 entries, the last from its Taylor series
//            (argument reduction by a table of reciprocals, as in Tang, "Table-driven
//            implementation of the logarithm function", 1990).
//            u within 2^-12 of 1 takes log1p in FP64 (the sum above cancels there).
//   sqrt     a float reciprocal square root and two Newton corrections of the
//            integer residual.
//   cos      cos(2 pi x) = sin(2 pi (1/4 - x)) after folding x to [0, 1/2]; the
//            Taylor series of sin(pi t / 2) on [0, 1] to t^23 (the remainder is
//            below 2^-66).
#pragma once

#include <math.h>
#include <stdint.h>

namespace bfm {
namespace fixedpt {

// Counts of steps and paths go up to 2^31 - 1; a loop over them ends one stride later,
// which 32 signed bits do not hold.
typedef uint32_t Count;

constexpr uint64_t kLn2Q64 = 0xB17217F7D1CF79ABull;  // ln 2 * 2^64

// floor(a b / 2^64) or one less (the product of the low halves is dropped), for a and b
// up to 2^63, where the sum of the middle products cannot overflow: three wide
// multiply-adds and no additions, which would go to the integer pipe.
__host__ __device__ __forceinline__ uint64_t mulhi(uint64_t a, uint64_t b) {
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32), b0 = (uint32_t)b, b1 = (uint32_t)(b >> 32);
    uint64_t mid = (uint64_t)a1 * b0;
    mid += (uint64_t)a0 * b1;
    return (uint64_t)a1 * b1 + (mid >> 32);
}

__host__ __device__ __forceinline__ uint32_t mulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
__host__ __device__ __forceinline__ int32_t mulhi32s(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }

__host__ __device__ __forceinline__ int clz64(uint64_t x) {  // x > 0
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}

// The reciprocal of table interval i: 2^11 over the midpoint of [1 + i/256, 1 + (i+1)/256).
__host__ __device__ __forceinline__ uint32_t log_recip(uint32_t i) {
    const uint32_t den = 512u + 2u * i + 1u;
    return ((1u << 20) + den / 2u) / den;
}

// -ln(c / 2^11) * 2^64 = 2 atanh((2048 - c) / (2048 + c)), summed in integers with 2^-80 steps.
inline uint64_t log_entry(uint32_t i) {
    const uint32_t c = log_recip(i);
    typedef unsigned __int128 u128;
    const u128 num = 2048u - c, den = 2048u + c;
    u128 pw = (num << 80) / den, sum = 0;
    for (uint32_t j = 1; pw != 0; j += 2) {
        sum += pw / j;
        pw = pw * num / den * num / den;
    }
    return (uint64_t)((2 * sum + (1u << 15)) >> 16);
}

struct LogTable {
    uint64_t ln[256];
};

// -ln(n 2^-53) = x 2^-64 2^(6 - z), x in [2^62, 2^64), z even; n < 2^53.
__host__ __device__ __forceinline__ void neg_log(uint64_t n, const uint64_t* ln, const uint32_t* rec, uint64_t& x, int& z) {
    const uint64_t w = (1ull << 53) - n;
    if (w < (1ull << 41)) {
        const double l = -log1p(-(double)w * (1.0 / 9007199254740992.0));
        uint64_t b;
#ifdef __CUDA_ARCH__
        b = (uint64_t)__double_as_longlong(l);
#else
        __builtin_memcpy(&b, &l, 8);
#endif
        x = (b << 11) | (1ull << 63);                  // l = x 2^-64 2^(6 - z)
        z = 1028 - (int)((b >> 52) & 0x7ff);
        if (z & 1) {
            x >>= 1;
            --z;
        }
        return;
    }
    const int e = 63 - clz64(n);  // <= 52
    const uint64_t M = n << (52 - e);
    const uint32_t i = (uint32_t)(M >> 44) & 255u;
    const int64_t s = (int64_t)((M * rec[i] - (1ull << 63)) << 8);  // r = s 2^-71
    const uint64_t a = (uint64_t)(s < 0 ? -s : s);
    const int32_t rr = (int32_t)(s >> 32);  // r = rr 2^-39
    // ln(1 + r) = r - r^2 p, p = 1/2 - r (1/3 - r (1/4 - r (1/5 - r (1/6 - r / 7))))
    int32_t h = (int32_t)(2147483648.0 / 6.0) - mulhi32s(rr, (int32_t)(16777216.0 / 7.0));
    h = (int32_t)(2147483648.0 / 5.0) - (mulhi32s(rr, h) >> 7);
    h = (int32_t)(2147483648.0 / 4.0) - (mulhi32s(rr, h) >> 7);
    const uint64_t g = (uint64_t)((int64_t)(0x5555555555555555ull >> 2) - (((int64_t)rr * h) >> 8)) << 2;  // 2^64 (1/3 - ...)
    const uint64_t rg = mulhi(a, g) >> 7;
    const uint64_t p = (1ull << 63) + (s < 0 ? rg : 0ull - rg);
    const int64_t l1p = (s >> 7) - (int64_t)(mulhi(mulhi(a, a), p) >> 14);
    // k ln2 - ln[i] - l1p in units of 2^-58 (k < 54, the sum below 37)
    const uint32_t k = (uint32_t)(53 - e);
    const uint64_t sub = (ln[i] >> 6) + (uint64_t)(l1p >> 6);
    const uint64_t lo = (uint64_t)k * (uint32_t)kLn2Q64, hi = (uint64_t)k * (uint32_t)(kLn2Q64 >> 32) + (lo >> 32);  // k ln2 2^32
    const uint64_t m = ((hi << 26) | ((uint32_t)lo >> 6)) - sub;
    z = clz64(m) & ~1;
    x = m << z;
}

// sqrt(x 2^-64) * 2^63 for x >= 2^62
__host__ __device__ __forceinline__ uint64_t sqrt_q63(uint64_t x) {
    const float xf = (float)(uint32_t)(x >> 32) * (1.f / 4294967296.f);
#ifdef __CUDA_ARCH__
    const float y = rsqrtf(xf);
#else
    const float y = 1.f / sqrtf(xf);
#endif
    const uint32_t Y = (uint32_t)(y * 1073741824.f);              // 2^30 / sqrt(x)
    const uint32_t s0 = (uint32_t)(xf * y * 16777216.f);          // 2^24 sqrt(x)
    const int64_t e0 = (int64_t)(x - (((uint64_t)s0 * s0) << 16));  // 2^64 (x - s0^2), below 2^43
    const int64_t s1 = ((int64_t)s0 << 24) + (((e0 >> 12) * (int64_t)Y) >> 35);  // 2^48
    const int64_t e1 = (int64_t)((x << 32) - (uint64_t)s1 * (uint64_t)s1);       // 2^96 (x - s1^2)
    return (uint64_t)((s1 << 15) + (((e1 >> 24) * (int64_t)Y) >> 40));
}

// |cos(2 pi f 2^-53)| * 2^61 and whether it is negative
__host__ __device__ __forceinline__ uint64_t cos_q61(uint64_t f, bool& neg) {
    uint64_t x = f << 11;                     // turns * 2^64
    if (x >> 63) x = 0ull - x;                // cos is even
    const int64_t d = (int64_t)((1ull << 62) - x);  // 1/4 - x
    neg = d < 0;
    const uint64_t t = (uint64_t)(d < 0 ? -d : d) << 1;  // 2^63 t, cos = sin(pi t / 2)
    const uint64_t u = mulhi(t, t) << 1;                 // 2^63 t^2
    const uint32_t uh = (uint32_t)(u >> 32);             // 2^31 t^2
    // a_k = (pi/2)^(2k+1) / (2k+1)!, k = 11 .. 0.  A product with u loses one bit of scale, so
    // each a_k is held with one bit more than the one before: 2^72 a_11 .. 2^69 a_8 in 32
    // bits, 2^69 a_7 .. 2^62 a_0 in 64.
    uint32_t g = 607160u - mulhi32(uh, 5921u);
    g = 51675268u - mulhi32(uh, g);
    g = 3581286744u - mulhi32(uh, g);
    uint64_t h = 394791910485ull - (((uint64_t)uh * g) >> 31);
    h = 16800329138375ull - mulhi(u, h);
    h = 531095520970866ull - mulhi(u, h);
    h = 11838469898620675ull - mulhi(u, h);
    h = 172726240700510392ull - mulhi(u, h);
    h = 1470069480924832210ull - mulhi(u, h);
    h = 5957967193751243515ull - mulhi(u, h);
    h = 7244019458077122842ull - mulhi(u, h);
    return mulhi(t, h);
}

// |z| 2^59 / sqrt(2) of the normal z = sqrt(-2 ln(n 2^-53)) cos(2 pi f 2^-53), n in [1, 2^53], f in [0, 2^53)
__host__ __device__ __forceinline__ uint64_t normal_q59(uint64_t n, uint64_t f, const uint64_t* ln, const uint32_t* rec,
                                                        bool& neg) {
    const uint64_t c = cos_q61(f, neg);
    if (n == (1ull << 53)) return 0;
    uint64_t x;
    int z;
    neg_log(n, ln, rec, x, z);
    return mulhi(sqrt_q63(x) >> (z / 2), c << 2);  // 2^60 sqrt(-ln u), 2^63 |cos|
}

}  // namespace fixedpt
}  // namespace bfm
