// mlkd_fixed.h -- FP64-accurate functions of the FP64 modes in 64-bit
// fixed-point integer arithmetic.
//
// GB300 executes two FP64 operations per clock and SM (measured: 1.81 FMA,
// conversion or comparison), against 64 32x32 -> 64-bit integer products.
// CUDA's FP64 functions cost about 34 (log), 29 (sincospi), 18 (exp), 9 (sqrt)
// and 5 (rsqrt) FP64 operations, and the Taylor polynomials of the KD
// coefficients 17 to 22 each; together they kept the FP64 pipe 85 % busy.
// The values these functions return lie in a known range, so a 64-bit
// fraction holds them with more than FP64's 53 bits: a product of two
// fractions takes three 32-bit products, and the error of a function before
// its one rounding to FP64 is a few 2^-62.
//
// Plain integer C++ (the one FP32 instruction is the seed of the square
// roots), so the same code runs and is tested on the host.
#pragma once

#include <cstdint>
#include <cstring>
#ifndef __CUDACC__
#include <cmath>
#endif

#include "mlkd_fixed_tables.h"

#ifdef __CUDACC__
#define MLKD_HD __host__ __device__ __forceinline__
#else
#define MLKD_HD inline
#endif

namespace mlkd {
namespace fx {

MLKD_HD int clz64(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}

MLKD_HD int max_int(int a, int b) { return a > b ? a : b; }

MLKD_HD uint64_t bits_of(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
#endif
}

MLKD_HD double from_bits(uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}

// 1/sqrt(x), relative error below 2^-22.9 (the hardware's seed)
MLKD_HD float rsqrt_seed(float x)
{
#ifdef __CUDA_ARCH__
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / sqrtf(x);
#endif
}

// a b 2^-64 and a b 2^-32, rounded down, at most one unit below
MLKD_HD uint64_t mul64(uint64_t a, uint64_t b)
{
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
    const uint32_t bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    const uint64_t p = (uint64_t)ah * bl;
    const uint64_t q = (uint64_t)al * bh + (uint32_t)p;
    return (uint64_t)ah * bh + (p >> 32) + (q >> 32);
}
MLKD_HD uint64_t mul64x32(uint64_t a, uint32_t b)
{
    return (a >> 32) * b + ((uint64_t)(uint32_t)a * b >> 32);
}
MLKD_HD uint32_t mul32(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }

// c0 - x (c1 - x (c2 - ...)) for a fraction x: the tail of the sum (terms
// below 2^-29) in 32 bits, the rest in 64
template <typename P, int I> MLKD_HD uint32_t poly_tail(uint32_t x)
{
    constexpr uint32_t c = P::tail[I];
    if constexpr (I + 1 < P::kTail) return c - mul32(x, poly_tail<P, I + 1>(x));
    else return c;
}
template <typename P, int I = 0> MLKD_HD uint64_t poly(uint64_t x)
{
    constexpr uint64_t c = P::lead[I];
    if constexpr (I + 1 < P::kLead) {
        return c - mul64(x, poly<P, I + 1>(x));
    } else {
        const uint32_t xh = (uint32_t)(x >> 32);
        return c - ((uint64_t)xh * poly_tail<P, 0>(xh) >> P::kShift);
    }
}

// v 2^-e rounded to nearest (0 for v = 0); the result must be a normal number
MLKD_HD double to_double(uint64_t v, int e)
{
    const int lz = clz64(v | 1u);
    const uint64_t m = v << lz;
    // the leading bit of m >> 11 adds one to the exponent field
    const uint64_t b = ((uint64_t)(1023 + 63 - 1 - lz - e) << 52) + (m >> 11) + ((m >> 10) & 1u);
    return from_bits(v ? b : 0u);
}

// The same for v in [2^62, 2^63]
MLKD_HD double to_double_62(uint64_t v, int e)
{
    return from_bits(((uint64_t)(1023 + 62 - 1 - e) << 52) + ((v + (1u << 9)) >> 10));
}

// The fraction x 2^64 of a double 0 <= x < 1 (rounded down)
MLKD_HD uint64_t fraction(double x)
{
    const uint64_t b = bits_of(x);
    const int sh = 1022 - (int)(b >> 52);                     // x = m 2^(-sh), m in [1/2, 1)
    const uint64_t m = (b << 11) | 0x8000000000000000ull;
    return sh < 64 ? m >> sh : 0u;
}

// n as a double, n >= 1
MLKD_HD double from_u32(uint32_t n)
{
#ifdef __CUDA_ARCH__
    const int lz = __clz((int)n);
#else
    const int lz = __builtin_clz(n);
#endif
    const uint32_t m = n << lz;
    return from_bits(((uint64_t)(uint32_t)((1023 + 31 - 1 - lz) << 20) << 32) + ((uint64_t)m << 21));
}

// A flight q >= 0 in steps: whole = floor(q) (at most 2^31 - 1) and
// left = (whole + 1 - q) 2^64, the part of the collision's step that is left
// (2^64 - 1 for a whole step)
struct Flight {
    int whole;
    uint64_t left;
};
MLKD_HD Flight split_flight(double q)
{
    const uint64_t b = bits_of(q);
    const int ex = (int)(b >> 52) - 1023;
    const uint64_t m = (b << 11) | 0x8000000000000000ull;     // q = m 2^(ex - 63)
    Flight f;
    uint64_t frac;
    if (ex < 0) {
        f.whole = 0;
        frac = ex > -64 ? m >> ((-1 - ex) & 63) : 0u;
    } else {
        f.whole = ex < 31 ? (int)(uint32_t)(m >> ((63 - ex) & 63)) : 0x7fffffff;
        frac = ex < 63 ? m << ((ex + 1) & 63) : 0u;
    }
    f.left = frac ? 0u - frac : ~(uint64_t)0;
    return f;
}

// steps + left 2^-64 as a double (steps >= 0)
MLKD_HD double steps_left(int steps, uint64_t left)
{
    if (steps == 0) return to_double(left, 64);
#ifdef __CUDA_ARCH__
    const int lz = __clz(steps);
#else
    const int lz = __builtin_clz((uint32_t)steps);
#endif
    // the leading bit of the 96-bit number comes to bit 63; lz >= 1
    const uint64_t v = ((uint64_t)(uint32_t)steps << (32 + lz)) | (left >> (32 - lz));
    return from_bits(((uint64_t)(1023 + 31 - 1 - lz) << 52) + (v >> 11) + ((v >> 10) & 1u));
}

// ---------------------------------------------------------------------------
// -ln u = v 2^-e for the uniform u = n 2^-B, 1 <= n <= 2^B.  n is normalised
// to x in [1/2, 1); with the reciprocal c of the upper end of x's interval
// (128 of them), 1 - x c = rho < 2^-7 and -ln x = ln c + rho + rho^2/2 + ...
// + rho^8/8.  Above 1 - 2^-12 (one draw in 4096), where the logarithm is about
// the small difference itself, the caller takes log_near_one: it keeps FP64's
// relative error there.
// ---------------------------------------------------------------------------
struct Fixed {
    uint64_t v;
    int e;
};

template <int B, typename Tab> MLKD_HD Fixed neg_log(uint64_t n, const Tab &tab)
{
    const int lz = clz64(n);
    const uint64_t x = n << lz;
    const int j = (int)(x >> 56) & 127;
    const uint32_t c = tab.recip(j);
    const uint64_t rho = 0u - (((uint64_t)(uint32_t)(x >> 32) * c << 17) + ((uint64_t)(uint32_t)x * c >> 15));
    const uint64_t y = rho << 7;                              // 2^7 rho as a fraction
    const uint32_t yh = (uint32_t)(y >> 32);
    // 1/4 + rho/5 + rho^2/6 + rho^3/7 + rho^4/8, then 1/3 + rho (.), 1/2 + rho (.)
    uint32_t t = (1u << 11) / 7u + (yh >> 28);
    t = (1u << 18) / 6u + mul32(yh, t);
    t = (1u << 25) / 5u + mul32(yh, t);
    t = (1u << 30) + mul32(yh, t);
    const uint64_t s = 0x5555555555555555ull + ((uint64_t)yh * t >> 7);
    const uint64_t w = 0x8000000000000000ull + (mul64(y, s) >> 7);
    const uint64_t l = tab.ln(j) + rho + (mul64(y, mul64(y, w)) >> 14);
    const int k = lz + B - 64;                                // whole powers of two in 1/u
    Fixed r;
    r.v = k > 0 ? (l >> 6) + (uint64_t)k * kLn2_58 : l;
    r.e = k > 0 ? 58 : 64;
    return r;
}

// -ln(1 - w) for 0 <= w < 2^-12, in FP64
MLKD_HD double log_near_one(double w)
{
    return w + w * w * (0.5 + w * (1.0 / 3.0 + w * (0.25 + w * 0.2)));
}

// ---------------------------------------------------------------------------
// Square roots.  For x = m 2^-64 in [1/4, 1): the seed y0 = (1 + d)/sqrt(x),
// d < 0, of 32 bits gives e = 1 - x y0^2 = 1 - (1 + d)^2 < 2^-20 exactly
// enough, and sqrt(x) = x y0 (1 - e)^(-1/2) = x y0 (1 + e/2 + 3 e^2/8 + ...).
// ---------------------------------------------------------------------------
struct Seed {
    uint32_t y0;      // 2^31 (1 + d)/sqrt(x)
    uint64_t c;       // 2^84 (e/2 + 3 e^2/8)
};
MLKD_HD Seed sqrt_seed(uint64_t m)
{
    Seed r;
    // the factor keeps d below 0 (seed 2^-22.9, conversion 2^-25)
    const float y = rsqrt_seed((float)(uint32_t)(m >> 32)) * (140737488355328.0f * (1.0f - 0x1p-22f));
    r.y0 = (uint32_t)y;
    const uint64_t e = (1ull << 62) - mul64(m, (uint64_t)r.y0 * r.y0);    // 2^62 e
    const uint64_t eh = e >> 22;
    r.c = (e << 21) + ((eh * eh * 3u) << 1);                  // 2^84: e 2^22/2 + 3/8 e^2 2^22
    return r;
}

// sqrt(m 2^-64) 2^63 for m in [2^62, 2^64): a value in [2^62, 2^63]
MLKD_HD uint64_t sqrt63(uint64_t m)
{
    const Seed r = sqrt_seed(m);
    const uint64_t s = mul64x32(m, r.y0);
    return s + (mul64(s, r.c) >> 20);
}

// 2^62/sqrt(m 2^-64) for m in [2^62, 2^64): a value in [2^62, 2^63]
MLKD_HD uint64_t rsqrt62(uint64_t m)
{
    const Seed r = sqrt_seed(m);
    const uint64_t s = (uint64_t)r.y0 << 31;
    return s + (mul64(s, r.c) >> 20);
}

// sqrt(v 2^-e), v != 0
MLKD_HD double sqrt_fixed(uint64_t v, int e)
{
    const int lz = clz64(v);
    uint64_t m = v << lz;
    const int p = e + lz;                                     // v 2^-e = m 2^-p
    m >>= p & 1;
    // sqrt(m) 2^(-p'/2) = (s 2^-63) 2^32 2^(-p'/2), p' = p - (p & 1)
    return to_double_62(sqrt63(m), 31 + (p >> 1));
}

// sqrt and 1/sqrt of a positive normal double
MLKD_HD double sqrt_normal(double x)
{
    const uint64_t b = bits_of(x);
    const int p = 1023 + 63 - (int)(b >> 52);                 // x = m 2^-p
    uint64_t m = (b << 11) | 0x8000000000000000ull;
    m >>= p & 1;
    return to_double_62(sqrt63(m), 31 + (p >> 1));
}
MLKD_HD double rsqrt_normal(double x)
{
    const uint64_t b = bits_of(x);
    const int p = 1023 + 63 - (int)(b >> 52);
    uint64_t m = (b << 11) | 0x8000000000000000ull;
    m >>= p & 1;
    // 1/sqrt(x) = 2^(p'/2) / sqrt(m) = (r 2^-62) 2^-32 2^(p'/2)
    return to_double_62(rsqrt62(m), 94 - (p >> 1));
}

// ---------------------------------------------------------------------------
// cos and sin of 2 pi phase 2^-64: the nearest quarter turn, z in [-pi/4, pi/4]
// ---------------------------------------------------------------------------
MLKD_HD void sincos_turn(uint64_t phase, double *sn, double *cs)
{
    const uint32_t k = (uint32_t)((phase + (1ull << 61)) >> 62);
    const uint64_t r = phase - ((uint64_t)k << 62);           // signed residual
    const bool neg = (int64_t)r < 0;
    const uint64_t a = (neg ? 0u - r : r) << 2;               // |residual| 2^66 <= 2^63
    const uint64_t z = mul64(a, kTwoPi_61) << 1;              // a 2^-66 2 pi, in 2^-64
    const uint64_t z2 = mul64(z, z);
    const uint64_t s = z - mul64(z, mul64(z2, poly<PolySin>(z2)));
    const uint64_t c = mul64(z2, poly<PolyCos>(z2));          // 1 - cos z <= 0.293
    const double ds = to_double(s, 64);
    const double dc = to_double(0x8000000000000000ull - (c >> 1), 63);
    // sin(z + k pi/2) and cos(z + k pi/2)
    const uint64_t sz = bits_of(ds) ^ (neg ? 0x8000000000000000ull : 0u);
    const uint64_t cz = bits_of(dc);
    const uint64_t sp = (k & 1u) ? cz : sz, cp = (k & 1u) ? sz : cz;
    *sn = from_bits(sp ^ ((uint64_t)(k & 2u) << 62));
    *cs = from_bits(cp ^ ((uint64_t)((k + 1u) & 2u) << 62));
}

// ---------------------------------------------------------------------------
// e^-x 2^64 for x >= 2^-4 (0 from x = 44 on): x log2 e = k + f,
// e^-x = 2^-k (1 - f P(f))
// ---------------------------------------------------------------------------
MLKD_HD uint64_t exp_neg(double x)
{
    const uint64_t b = bits_of(x);
    const int ex = max_int((int)(b >> 52) - 1023, -2);        // x = m 2^(ex - 63)
    const uint64_t m = ((b << 11) | 0x8000000000000000ull) >> ((ex + 1023 - (int)(b >> 52)) & 63);
    const uint64_t y = mul64(m, kLog2e_63);                   // x log2 e 2^(62 - ex)
    const uint64_t f = y << ((ex + 2) & 63);
    const uint64_t p = ~mul64(f, poly<PolyE>(f));
    return (uint32_t)(b >> 32) < 0x40460000u ? p >> (int)(((y >> 1) >> ((61 - ex) & 63)) & 63u) : 0u;    // 44.0
}

}  // namespace fx
}  // namespace mlkd
