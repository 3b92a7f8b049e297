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
// fractions takes three 32-bit products (a quarter of an FP64 one's time), and the error of a function before
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

#ifdef __CUDACC__
#define MLKD_HD __device__ __forceinline__
#define MLKD_CONSTANT static __constant__
#else
#define MLKD_HD inline
#define MLKD_CONSTANT static const
#endif

#include "mlkd_fixed_tables.h"

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

MLKD_HD uint32_t umulhi(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)((uint64_t)a * b >> 32);
#endif
}

// a b 2^-64 and a b 2^-32, rounded down, at most two units below.  The high
// halves of the cross products and one wide product: 8.2 per clock and SM
// measured, against 6.6 with the carry of the low halves and 6.4 for
// __umul64hi (2^20 pairs of level 8 of the periodic problem: 8.52, 9.51 and
// 9.41 ms).
MLKD_HD uint64_t mul64(uint64_t a, uint64_t b)
{
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
    const uint32_t bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    return (uint64_t)ah * bh + umulhi(ah, bl) + umulhi(al, bh);
}
MLKD_HD uint64_t mul64x32(uint64_t a, uint32_t b)
{
    return (a >> 32) * b + umulhi((uint32_t)a, b);
}

// c0 - x (c1 - x (c2 - ...)) for a fraction x: the tail of the sum (terms
// below 2^-29) in 32 bits, the rest in 64.
template <typename P, int K, int I = 0> MLKD_HD uint32_t poly_tail(uint32_t x)
{
    uint32_t c;
    if constexpr (K == 0) {
        constexpr uint32_t c0 = P::tail0[I];
        c = c0;
    } else {
        constexpr uint32_t c1 = P::tail1[I];
        c = c1;
    }
    if constexpr (I + 1 < P::kTail) return c - umulhi(x, poly_tail<P, K, I + 1>(x));
    else return c;
}
template <typename P> MLKD_HD uint64_t poly(const uint64_t (&c)[P::kLead][1], uint64_t x)
{
    const uint32_t xh = (uint32_t)(x >> 32);
    uint64_t a = c[P::kLead - 1][0] - ((uint64_t)xh * poly_tail<P, 0>(xh) >> P::kShift0);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int i = P::kLead - 2; i >= 0; --i) a = c[i][0] - mul64(x, a);
    return a;
}
// Two polynomials in the same argument.  The 64-bit steps are a rolled loop
// over coefficients in constant memory: the FP64 event loop is longer than the
// instruction caches like (unrolled here too, 2^20 pairs of level 8 of the
// periodic problem take 10.2 ms, so 8.52 ms; rolled in poly() as well 8.69 ms, and
// of level 6 at eps = 1e-3 7.95 ms, so 7.07 ms).
struct Two {
    uint64_t a, b;
};
template <typename P> MLKD_HD Two poly_two(const uint64_t (&c)[P::kLead][2], uint64_t x)
{
    const uint32_t xh = (uint32_t)(x >> 32);
    Two t;
    t.a = c[P::kLead - 1][0] - ((uint64_t)xh * poly_tail<P, 0>(xh) >> P::kShift0);
    t.b = c[P::kLead - 1][1] - ((uint64_t)xh * poly_tail<P, 1>(xh) >> P::kShift1);
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
    for (int i = P::kLead - 2; i >= 0; --i) {
        t.a = c[i][0] - mul64(x, t.a);
        t.b = c[i][1] - mul64(x, t.b);
    }
    return t;
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

// ---------------------------------------------------------------------------
// A positive number m 2^-e with m in [2^63, 2^64): products of quantities of
// any size, at 2^-62 relative error, without the FP64 pipe.
// ---------------------------------------------------------------------------
struct Pos {
    uint64_t m;
    int e;
};
MLKD_HD Pos pos_of(double x)          // x a positive normal number (0: a number below 2^-1000)
{
    const uint64_t b = bits_of(x);
    Pos r;
    r.m = (b << 11) | 0x8000000000000000ull;
    r.e = 1023 + 63 - (int)(b >> 52);
    return r;
}
MLKD_HD Pos pos_fixed(uint64_t v, int e)                      // v 2^-e, v != 0
{
    const int lz = clz64(v);
    Pos r;
    r.m = v << lz;
    r.e = e + lz;
    return r;
}
// the same of v + low 2^-32, for v >= 2^32
MLKD_HD Pos pos_fixed(uint64_t v, uint32_t low, int e)
{
    const int lz = clz64(v) & 31;
    Pos r;
#ifdef __CUDA_ARCH__
    const uint32_t h = __funnelshift_l((uint32_t)v, (uint32_t)(v >> 32), lz), m = __funnelshift_l(low, (uint32_t)v, lz);
    r.m = (uint64_t)h << 32 | m;
#else
    r.m = v << lz | (uint64_t)low << lz >> 32;
#endif
    r.e = e + lz;
    return r;
}
MLKD_HD Pos pos_norm(uint64_t p, int e)                       // p 2^-e, p in [2^62, 2^64)
{
    const int sh = (int)(p >> 63) ^ 1;
    Pos r;
    r.m = p << sh;
    r.e = e + sh;
    return r;
}
MLKD_HD Pos operator*(const Pos &a, const Pos &b) { return pos_norm(mul64(a.m, b.m), a.e + b.e - 64); }
// a times a fraction f 2^-64 of at least 1/2
MLKD_HD Pos times(const Pos &a, uint64_t f) { return pos_norm(mul64(a.m, f), a.e); }
// The bits of the nearest double, for a.e <= 1084 (a number of at least 2^-1021;
// e = 1086 with m = 2^63 gives 0).  The exponent field of a smaller one wraps:
// draws, their products and squares, which can be below that, go through
// to_double_or_0.
MLKD_HD uint64_t bits_of(const Pos &a)
{
    return ((uint64_t)(1023 + 63 - 1 - a.e) << 52) + (a.m >> 11) + ((a.m >> 10) & 1u);
}
MLKD_HD double to_double(const Pos &a) { return from_bits(bits_of(a)); }
// the same, 0 below 2^-1021
MLKD_HD uint64_t bits_or_0(const Pos &a) { return a.e <= 1084 ? bits_of(a) : 0u; }
MLKD_HD double to_double_or_0(const Pos &a) { return from_bits(bits_or_0(a)); }
// a 2^k rounded down, for a 2^k < 2^64
MLKD_HD uint64_t scaled(const Pos &a, int k)
{
    const int sh = a.e - k;
    return sh < 64 ? a.m >> sh : 0u;
}

// v 2^-sh rounded down, for either sign of sh (sh > -64)
MLKD_HD uint64_t shift_to(uint64_t v, int sh) { return sh < 0 ? v << -sh : sh < 64 ? v >> sh : 0u; }

// x, or 0 where x is negative
MLKD_HD double not_negative(double x)
{
    const uint64_t b = bits_of(x);
    return from_bits((int64_t)b < 0 ? 0u : b);
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

// A flight q in steps: whole = floor(q) (at most 2^31 - 1) and
// left = (whole + 1 - q) 2^64, the part of the collision's step that is left
// (2^64 - 1 for a whole step)
struct Flight {
    int whole;
    uint64_t left;
};
MLKD_HD Flight split_flight(const Pos &q)
{
    Flight f;
    uint64_t frac;
    if (q.e >= 64) {
        f.whole = 0;
        frac = scaled(q, 64);
    } else {
        f.whole = q.e > 32 ? (int)(uint32_t)(q.m >> q.e) : 0x7fffffff;
        frac = q.e > 0 ? q.m << (64 - q.e) : 0u;
    }
    f.left = frac ? 0u - frac : ~(uint64_t)0;
    return f;
}

// steps + left 2^-64 (steps >= 0, the sum not 0)
MLKD_HD Pos steps_left(int steps, uint64_t left)
{
    const Pos a = pos_fixed(left | 1u, 64);
#ifdef __CUDA_ARCH__
    const int lz = __clz(steps | 1);
#else
    const int lz = __builtin_clz((uint32_t)steps | 1u);
#endif
    // the leading bit of the 96-bit number comes to bit 63; lz >= 1
    const uint64_t v = ((uint64_t)(uint32_t)steps << (32 + lz)) | (left >> (32 - lz));
    Pos r;
    r.m = steps ? v : a.m;
    r.e = steps ? 32 + lz : a.e;
    return r;
}

// ---------------------------------------------------------------------------
// -ln u for the uniform u = n 2^-B, 1 <= n <= 2^B.  n is normalised
// to x in [1/2, 1); with the reciprocal c of the upper end of x's interval
// (128 of them), 1 - x c = rho < 2^-7 and -ln x = ln c + rho + rho^2/2 + ...
// + rho^8/8, in units of 2^-64 and 14 bits more of the series.  In the last
// interval below u = 1, where c = 1, ln c and rho are exact and those bits hold
// FP64's precision down to 2^-12 (elsewhere they change nothing).  Above
// 1 - 2^-12 (one draw in 4096) the caller takes log_near_one.
// ---------------------------------------------------------------------------
template <int B, typename Tab> MLKD_HD Pos neg_log(uint64_t n, const Tab &tab)
{
    const int lz = clz64(n);
    const uint64_t x = n << lz;
    const int j = (int)(x >> 56) & 127;
    const uint32_t c = tab.recip(j);
    const uint64_t rho = 0u - (((uint64_t)(uint32_t)(x >> 32) * c << 17) + ((uint64_t)(uint32_t)x * c >> 15));
    const uint64_t y = rho << 7;                              // 2^7 rho as a fraction
    const uint32_t yh = (uint32_t)(y >> 32);
    // 1/4 + rho/5 + rho^2/6 + rho^3/7 + rho^4/8 in 2^-33, then 1/3 + rho (.), 1/2 + rho (.)
    uint32_t t = ((1u << 12) + 3u) / 7u + (yh >> 27);
    t = ((1u << 19) + 3u) / 6u + umulhi(yh, t);
    t = ((1u << 26) + 2u) / 5u + umulhi(yh, t);
    t = (1u << 31) + umulhi(yh, t);
    const uint64_t s = 0x5555555555555555ull + ((uint64_t)yh * t >> 8);
    const uint64_t w = 0x8000000000000000ull + (mul64(y, s) >> 7);
    const uint64_t q = mul64(y, mul64(y, w));                 // 2^14 (rho^2/2 + ...)
    const uint64_t l = tab.ln(j) + rho + (q >> 14);
    const int k = lz + B - 64;                                // whole powers of two in 1/u
    return pos_fixed(k > 0 ? (l >> 6) + (uint64_t)k * kLn2_58 : l, (uint32_t)q << 18, k > 0 ? 58 : 64);
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

MLKD_HD Pos sqrt(const Pos &x)
{
    const int odd = x.e & 1;
    // sqrt(m 2^-e) = sqrt(m/2^odd) 2^((odd - e)/2) = (s 2^-63) 2^32 2^((odd - e)/2)
    const uint64_t s = sqrt63(x.m >> odd);                    // [2^62, 2^63]
    Pos r;
    r.m = s >> 63 ? ~(uint64_t)0 : s << 1;
    r.e = 32 + (x.e >> 1);
    return r;
}

// sqrt and 1/sqrt of a positive normal double
MLKD_HD double sqrt_normal(double x) { return to_double(sqrt(pos_of(x))); }
MLKD_HD double rsqrt_normal(double x)
{
    const Pos p = pos_of(x);
    // 1/sqrt(x) = 2^(e'/2) / sqrt(m) = (r 2^-62) 2^-32 2^(e'/2)
    return to_double_62(rsqrt62(p.m >> (p.e & 1)), 94 - (p.e >> 1));
}

// ---------------------------------------------------------------------------
// cos and sin of 2 pi phase 2^-64: the nearest quarter turn, z in [-pi/4, pi/4].
// |z| is formed from the normalised residual, so that sin z keeps its relative
// precision (2^-61) however small it is; on an axis it is 0 (0 2^-3063).
// ---------------------------------------------------------------------------
struct Residual {
    uint64_t a;                   // |phase - k 2^62| 2^2, at most 2^63
    uint32_t k;                   // quarter turns
    bool neg;
};
MLKD_HD Residual quarter_turns(uint64_t phase)
{
    Residual q;
    q.k = (uint32_t)((phase + (1ull << 61)) >> 62);
    const uint64_t r = phase - ((uint64_t)q.k << 62);
    q.neg = (int64_t)r < 0;
    q.a = (q.neg ? 0u - r : r) << 2;
    return q;
}
// the signs of sin(z + k pi/2) and cos(z + k pi/2)
MLKD_HD uint64_t sin_sign_of(const Residual &q)
{
    return (!(q.k & 1u) && q.neg ? 0x8000000000000000ull : 0u) ^ ((uint64_t)(q.k & 2u) << 62);
}
MLKD_HD uint64_t cos_sign_of(const Residual &q)
{
    return ((q.k & 1u) && q.neg ? 0x8000000000000000ull : 0u) ^ ((uint64_t)((q.k + 1u) & 2u) << 62);
}

struct TurnPos {
    Pos sin, cos;                 // magnitudes
    uint64_t sin_sign, cos_sign;  // the sign bits of doubles
};
MLKD_HD TurnPos sincos_pos(uint64_t phase)
{
    const Residual q = quarter_turns(phase);
    const int lz = clz64(q.a | 1u);
    const uint64_t zn = mul64(q.a << lz, kTwoPi_61);          // |z| 2^(63 + lz), at least 2^62 (or 0)
    const uint64_t z = (zn >> lz) << 1;                       // |z| 2^64
    const uint64_t z2 = mul64(z, z);
    const Two p = poly_two<PolySC>(kPolySC, z2);
    const Pos s = pos_norm(zn - mul64(zn, mul64(z2, p.a)), q.a ? 63 + lz : 3063);
    const uint64_t c = ~mul64(z2, p.b);                       // cos z >= 0.707
    const bool odd = q.k & 1u;
    TurnPos t;
    t.sin.m = odd ? c : s.m;
    t.sin.e = odd ? 64 : s.e;
    t.cos.m = odd ? s.m : c;
    t.cos.e = odd ? s.e : 64;
    t.sin_sign = sin_sign_of(q);
    t.cos_sign = cos_sign_of(q);
    return t;
}

// The same as fractions, right to 2^-62 absolute
struct Turn {
    uint64_t sin, cos;            // magnitudes, in 2^-64 (below 1)
    uint64_t sin_sign, cos_sign;
};
MLKD_HD Turn sincos_turn(uint64_t phase)
{
    const Residual q = quarter_turns(phase);
    const uint64_t z = mul64(q.a, kTwoPi_61) << 1;
    const uint64_t z2 = mul64(z, z);
    const Two p = poly_two<PolySC>(kPolySC, z2);
    const uint64_t s = z - mul64(z, mul64(z2, p.a));
    const uint64_t c = ~mul64(z2, p.b);
    const bool odd = q.k & 1u;
    Turn t;
    t.sin = odd ? c : s;
    t.cos = odd ? s : c;
    t.sin_sign = sin_sign_of(q);
    t.cos_sign = cos_sign_of(q);
    return t;
}

// ---------------------------------------------------------------------------
// e^-x 2^64 for x >= 2^-4 (0 from x = 44 on): x log2 e = k + f,
// e^-x = 2^-k (1 - f P(f))
// ---------------------------------------------------------------------------
MLKD_HD uint64_t exp_neg(const Pos &x)
{
    const int ex = max_int(63 - x.e, -2);                     // x = m 2^(ex - 63)
    const uint64_t m = x.m >> ((ex + x.e - 63) & 63);
    const uint64_t y = mul64(m, kLog2e_63);                   // x log2 e 2^(62 - ex)
    const uint64_t f = y << ((ex + 2) & 63);
    const uint64_t p = ~mul64(f, poly<PolyE>(kPolyE, f));
    const bool in_range = x.e > 58 || (x.e == 58 && x.m < 0xb000000000000000ull);    // x < 44
    return in_range ? p >> (int)(((y >> 1) >> ((61 - ex) & 63)) & 63u) : 0u;
}

}  // namespace fx
}  // namespace mlkd
