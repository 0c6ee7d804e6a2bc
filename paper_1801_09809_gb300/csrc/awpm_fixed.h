// Double-precision division and logarithm in 64-bit integer arithmetic, for
// the weights (Section 6.1).
//
// A GB300 SM issues about two FP64 operations per clock, and an FP64 division
// or logarithm is a chain of ten to twenty-five of them; its integer units
// issue 64 32-bit multiply-adds per clock.  So the two functions that the
// weights call per entry are done in integers:
//
//   quotient(a, s): the correctly rounded a / s.v.  The divisors are shared
//     by whole columns and rows, so a fixed-point reciprocal is computed once
//     per divisor (make_scale) and an entry costs one 64-bit high product, one
//     low product for the exact remainder, and the rounding.
//   neg_log(x): -log(x) for x in (0, 1), by table and series: x = m 2^-k with
//     m in [1/2, 1); c = C/1024 is the largest such fraction with m c <= 1 over
//     m's interval of 2^-10, z = 1 - m c is exact in 64 bits, and
//     -log(x) = k ln 2 + log(c) - log(1 - z), every term >= 0, so nothing
//     cancels; for the interval next to 1, where k ln 2 = log(c) = 0, the
//     series' product is normalised first, which keeps full relative
//     precision up to x = 1 - 2^-53.  Within 0.53 units in the last place.
//
// (Table-driven logarithms: P. T. P. Tang, "Table-driven implementation of
// the logarithm function in IEEE floating-point arithmetic", ACM TOMS 16,
// 1990; the table here comes from the series of artanh, evaluated in 128-bit
// integers when the program is compiled.)
//
// Plain C++ with host and device forms, so that both are tested on the CPU.
#pragma once

#include <stdint.h>
#ifndef __CUDACC__
#include <cstring>
#endif

#ifdef __CUDACC__
#define AWPM_HD __host__ __device__ __forceinline__
#else
#define AWPM_HD inline
#endif

namespace awpm {

AWPM_HD uint64_t fx_mulhi(uint64_t a, uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

AWPM_HD int fx_clz(uint64_t a)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)a);
#else
    return a ? __builtin_clzll(a) : 64;
#endif
}

AWPM_HD uint64_t fx_bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    __builtin_memcpy(&b, &x, sizeof b);
    return b;
#endif
}

AWPM_HD double fx_double(uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    __builtin_memcpy(&x, &b, sizeof x);
    return x;
#endif
}

constexpr uint64_t kFxMant = (1ull << 52) - 1;
constexpr uint64_t kFxOne = 0x3ff0000000000000ull;

// A divisor (a positive finite double, as its bits) and 2^116 / mantissa,
// low by at most kFxInvSlack units (0 for a divisor without a normal
// mantissa, which quotient() hands to the FP64 division).
struct alignas(16) Scale {
    uint64_t v;
    uint64_t inv;
};

AWPM_HD Scale make_scale(uint64_t bits)
{
    Scale s;
    s.v = bits;
    s.inv = 0;
    const uint32_t e = (uint32_t)(bits >> 52);
    if (e == 0 || e >= 0x7ff)
        return s;
    // D / 2^63 in [1, 2); y / 2^63 tends to 2^63 / D: a 22-bit start from the
    // single-precision reciprocal, then two Newton steps (44, then 62 bits)
    const uint64_t D = ((bits & kFxMant) | (1ull << 52)) << 11;
    const float f = (float)(uint32_t)(D >> 40) * 1.1920928955078125e-07f;  // 2^-23
    uint64_t y = (uint64_t)(uint32_t)(2147483648.0f / f) << 32;
    if (y > (1ull << 63))
        y = 1ull << 63;
    for (int it = 0; it < 2; ++it) {
        const int64_t e62 = (int64_t)((1ull << 62) - fx_mulhi(D, y));
        // y * e62 / 2^62, with the sign taken out of the product
        const uint64_t m = (uint64_t)(e62 < 0 ? -e62 : e62) << 2;
        const uint64_t d = fx_mulhi(y, m);
        y = e62 < 0 ? y - d : y + d;
    }
    // an underestimate: the error of y is a few units, of 2 y twice that
    s.inv = 2 * (y - 12);
    return s;
}

// a / s.v, correctly rounded (a positive finite).  `ok` is false, and the
// result unspecified, when an operand or the quotient is not normal.
AWPM_HD uint64_t quotient(uint64_t a, const Scale &s, bool &ok)
{
    const uint64_t ma = (a & kFxMant) | (1ull << 52);
    const uint64_t mb = (s.v & kFxMant) | (1ull << 52);
    const int lt = ma < mb ? 1 : 0;
    // q = floor(ma 2^(53 + lt) / mb), 54 bits: at most one too low at first
    uint64_t q = fx_mulhi(ma << (1 + lt), s.inv);
    uint64_t rem = (ma << (53 + lt)) - q * mb;  // exact modulo 2^64
    if (rem >= mb) {
        rem -= mb;
        ++q;
    }
    const int e = (int)(a >> 52) - (int)(s.v >> 52) + 1023 - lt;
    uint64_t m = q >> 1;
    if ((q & 1) && (rem != 0 || (m & 1)))
        ++m;
    ok = s.inv != 0 && (a >> 52) != 0 && e >= 1 && e <= 2045;
    return ((uint64_t)(uint32_t)e << 52) + (m - (1ull << 52));
}

// ---- logarithm -----------------------------------------------------------

// log(c) for c = C / 1024, in units of 2^-71 (64 low bits and the rest), and C.
struct alignas(16) LogEntry {
    uint64_t lo;
    uint32_t hi;
    uint32_t C;
};

// log(C / 1024) 2^71, rounded: 2 artanh((C - 1024) / (C + 1024)), the terms
// in units of 2^-100.
constexpr unsigned __int128 fx_log_ratio(uint32_t C)
{
    const unsigned __int128 a = C - 1024, b = C + 1024;
    unsigned __int128 t = (a << 100) / b, s = 0;
    for (int i = 0; i < 40; ++i) {
        s += t / (2 * i + 1);
        t = t * (a * a) / (b * b);
    }
    return (2 * s + ((unsigned __int128)1 << 28)) >> 29;
}

struct LogTable {
    LogEntry e[512];
};

// Entry x serves m in [(512 + x) / 1024, (513 + x) / 1024).
constexpr LogTable fx_make_log_table()
{
    LogTable t{};
    for (int x = 0; x < 512; ++x) {
        const uint32_t C = (1u << 20) / (513u + (uint32_t)x);
        const unsigned __int128 v = fx_log_ratio(C);
        t.e[x].lo = (uint64_t)v;
        t.e[x].hi = (uint32_t)(v >> 64);
        t.e[x].C = C;
    }
    return t;
}

constexpr unsigned __int128 kFxLn2 = fx_log_ratio(2048);
constexpr uint64_t kFxLn2Lo = (uint64_t)kFxLn2;
constexpr uint32_t kFxLn2Hi = (uint32_t)(kFxLn2 >> 64);

// log(x) as bits for a normal x (as its bits) in (0, 1); table as above.
AWPM_HD uint64_t log_below_one(uint64_t x, const LogEntry *table)
{
    const uint32_t k = 1022u - (uint32_t)(x >> 52);
    const uint64_t M = (x & kFxMant) | (1ull << 52);
    const LogEntry te = table[(uint32_t)(M >> 43) & 511u];
    // z = 1 - m c, exact in units of 2^-71 (z < 2^-8)
    const uint64_t zz = ((1ull << 63) - M * te.C) << 8;
    const bool near1 = (k == 0u) & (te.C == 1024u);
    const int sh = near1 ? fx_clz(zz) - 1 : 0;
    // Q = 1 + z/2 + z^2/3 + ... + z^7/8; the inner terms in 32 bits
    const uint32_t z32 = (uint32_t)(zz >> 31);  // units of 2^-40
    auto step = [z32](uint32_t c, uint32_t r) {
        return c + (uint32_t)(((uint64_t)z32 * r) >> 40);
    };
    uint32_t r = 0x20000000u;    // 1/8
    r = step(0x24924925u, r);    // 1/7
    r = step(0x2aaaaaabu, r);    // 1/6
    r = step(0x33333333u, r);    // 1/5
    r = step(0x40000000u, r);    // 1/4
    const uint64_t q2 = 0x5555555555555555ull + (((uint64_t)z32 * r) >> 8);  // 1/3
    const uint64_t q1 = (1ull << 63) + (fx_mulhi(zz, q2) >> 7);
    const uint64_t q = (1ull << 63) + (fx_mulhi(zz, q1) >> 8);
    const uint64_t P = fx_mulhi(zz << sh, q) << 1;
    // the sum, in units of 2^(-71 - sh)
    uint64_t lo = P, hi = 0;
    if (!near1) {
        const uint64_t kl = (uint64_t)k * kFxLn2Lo;
        hi = fx_mulhi(k, kFxLn2Lo) + (uint64_t)k * kFxLn2Hi + te.hi;
        const uint64_t a = kl + te.lo;
        hi += a < kl ? 1 : 0;
        lo = a + P;
        hi += lo < a ? 1 : 0;
    }
    const int nz = fx_clz(hi ? hi : lo);
    uint64_t top = lo << nz;
    int e = -nz - 8 - sh;
    if (hi) {
        top = (hi << nz) | (lo >> (64 - nz));
        e += 64;
    }
    const uint64_t m = (top >> 11) + ((top >> 10) & 1);
    return 0x8000000000000000ull | (((uint64_t)(uint32_t)(e + 1023) << 52) + (m - (1ull << 52)));
}

}  // namespace awpm
