// Exponential, product and reciprocal of FP64 numbers on the integer units.
//
// GB300 issues one FP64 instruction of a warp per SM every 16 cycles, and in
// that time 64 others, so a 64-bit exponential is some 20 times cheaper in
// fixed point than in FP64 instructions.  Numbers are a 64-bit significand and
// an exponent; errors are a few units of 2^-63, so results rounded to FP64 are
// within 0.51 ulp (CUDA's exp: 1 ulp, and the FP64 product in front of it).
//
// exp2 is table-driven (P. T. P. Tang, Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic, ACM TOMS 15, 1989):
// 2^(i/128) from a table times the Taylor polynomial of 2^r, r < 1/128.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN inline
#endif

namespace fx {

// value m 2^(e - 63), m >= 2^63
struct Num {
    uint64_t m;
    int e;
};

FX_FN uint64_t mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return uint64_t((unsigned __int128)a * b >> 64);
#endif
}
FX_FN int64_t mulhis(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return int64_t((__int128)a * b >> 64);
#endif
}
FX_FN uint64_t bits(double x) {
#ifdef __CUDA_ARCH__
    return uint64_t(__double_as_longlong(x));
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
#endif
}
FX_FN double from_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}
// exponent field: 1 .. 2046 for normal numbers
FX_FN int field(double x) { return int(bits(x) >> 52) & 0x7ff; }

// |x| of a normal number (zero and subnormals come out as 2^-1023 .. 2^-1022)
FX_FN Num unpack(double x) {
    const uint64_t b = bits(x);
    return Num{b << 11 | 1ull << 63, (int(b >> 52) & 0x7ff) - 1023};
}
// nearest FP64 number; e must lie in the normal range
FX_FN double pack(Num a) { return from_bits((uint64_t(a.e + 1022) << 52) + (a.m >> 11) + (a.m >> 10 & 1)); }

FX_FN Num mul(Num a, Num b) {
    const uint64_t h = mulhi(a.m, b.m);
    const int low = h >> 63 ? 0 : 1;
    return Num{h << low, a.e + b.e + 1 - low};
}

// 1 / a: an FP32 estimate y0 and the first terms of y0 / (1 - (1 - a y0))
FX_FN Num reciprocal(Num a) {
    uint32_t fb = 0x3f800000u | (uint32_t(a.m >> 40) & 0x7fffffu);
    float f;
#ifdef __CUDA_ARCH__
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(__uint_as_float(fb)));
    fb = __float_as_uint(f);
#else
    memcpy(&f, &fb, 4);
    f = 1.0f / f;
    memcpy(&fb, &f, 4);
#endif
    fb = fb < 0x3f000000u ? 0x3f000000u : fb;  // the estimate may be off by an ulp
    // y0 in (1/2, 1] as 2^64 y0; 1 does not fit
    const uint64_t y = fb >= 0x3f800000u ? 0xffffffff00000000ull : uint64_t(fb << 8 | 0x80000000u) << 32;
    const int64_t s = int64_t((1ull << 63) - mulhi(a.m, y)) << 20;  // 2^83 (1 - a y0), below 2^62
    const int64_t t = s + (mulhis(s, s) >> 19);                     // ... + its square
    const uint64_t q = y + uint64_t(mulhis(int64_t(y >> 1), t) >> 18);
    return Num{q >> 63 ? q : 1ull << 63, -a.e - 1};
}

// floor(2^63 2^(i/128)), by the exponential series in 120-bit fixed point
struct Table {
    uint64_t t[128];
};
constexpr uint64_t kLn2 = 0xB17217F7D1CF79ABull;   // 2^64 ln 2
constexpr uint64_t kLog2e = 0xB8AA3B295C17F0BCull;  // 2^63 log2 e
constexpr Table make_table() {
    Table r{};
    for (int i = 0; i < 128; ++i) {
        const uint64_t y = uint64_t((unsigned __int128)kLn2 * unsigned(i) >> 7);
        unsigned __int128 term = (unsigned __int128)1 << 120, sum = term;
        for (int n = 1; n < 40; ++n) {
            term = ((term >> 64) * y + ((unsigned __int128)uint64_t(term) * y >> 64)) / unsigned(n);
            sum += term;
        }
        r.t[i] = uint64_t(sum >> 57);
    }
    return r;
}
constexpr uint64_t ln2_power(int n) {  // 2^64 ln(2)^n
    uint64_t p = kLn2;
    for (int i = 1; i < n; ++i) p = uint64_t((unsigned __int128)p * kLn2 >> 64);
    return p;
}
// Taylor coefficients of 2^(u / 128), times 2^64; the next one is 2^-65
constexpr uint64_t kA1 = ln2_power(1) >> 7, kA2 = ln2_power(2) / 2 >> 14, kA3 = ln2_power(3) / 6 >> 21;
constexpr uint32_t kA4 = uint32_t(ln2_power(4) / 24 >> 28), kA5 = uint32_t(ln2_power(5) / 120 >> 35),
                   kA6 = uint32_t(ln2_power(6) / 720 >> 42);

// 2^-t for t < 1024 (t.e <= 9)
FX_FN Num exp2_neg(Num t, const uint64_t *table) {
    uint64_t k = 0, f = 0;  // integer part and fraction x 2^64
    if (t.e >= 0) {
        k = t.m >> (63 - t.e);
        f = t.m << t.e << 1;
    } else if (t.e >= -64) {
        f = t.m >> (-t.e - 1);
    }
    const uint64_t g = 0 - f, u = g << 7;
    const uint32_t v = uint32_t(u >> 32);
    const uint32_t h5 = kA5 + uint32_t((uint64_t)v * kA6 >> 32);
    const uint32_t h4 = kA4 + uint32_t((uint64_t)v * h5 >> 32);
    const uint64_t h3 = kA3 + ((uint64_t)v * h4 >> 32);
    const uint64_t p = mulhi(u, kA1 + mulhi(u, kA2 + mulhi(u, h3)));
    const uint64_t b = table[g >> 57];
    return Num{b + mulhi(b, p), -int(k) - (f ? 1 : 0)};
}

}  // namespace fx
