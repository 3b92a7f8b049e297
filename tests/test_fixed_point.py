"""The 64-bit fixed-point functions of the FP64 modes (csrc/mlkd_fixed.h),
compiled for the host and compared with extended-precision library functions.

Bounds, derived from the arithmetic: every function ends in one rounding to
FP64 (half an ulp) of a fixed-point value whose own error is below 2^-58 (the
logarithm with whole powers of two, held in units of 2^-58) or 2^-60 (the
others).  Near u = 1 the logarithm is FP64 arithmetic of five operations,
each at most half an ulp of a term no larger than the result (2 ulp).
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2004_04071_gb300", "csrc")

SHIM = r"""
#include "mlkd_fixed.h"
using namespace mlkd;
static const uint32_t rc[128] = {MLKD_LOG_RECIPROCALS};
static const uint64_t ln_[128] = {MLKD_LOG_TABLE};
struct Tab {
    uint32_t recip(int j) const { return rc[j]; }
    uint64_t ln(int j) const { return ln_[j]; }
};
template <int B> static fx::Pos nl(uint64_t n) { return fx::neg_log<B>(n, Tab()); }
extern "C" void neg_log(int B, const uint64_t *n, int64_t count, double *E, double *r)
{
    for (int64_t i = 0; i < count; ++i) {
        fx::Pos f = B == 53 ? nl<53>(n[i]) : nl<24>(n[i]);
        E[i] = fx::to_double(f);
        f.e -= 1;
        r[i] = fx::to_double(fx::sqrt(f));
    }
}
extern "C" void near_one(const double *w, int64_t count, double *E)
{
    for (int64_t i = 0; i < count; ++i) E[i] = fx::log_near_one(w[i]);
}
extern "C" void sincos_turn(const uint64_t *p, int64_t count, double *s, double *c)
{
    for (int64_t i = 0; i < count; ++i) {
        const fx::Turn t = fx::sincos_turn(p[i]);
        s[i] = fx::from_bits(fx::bits_of(fx::to_double(t.sin, 64)) ^ t.sin_sign);
        c[i] = fx::from_bits(fx::bits_of(fx::to_double(t.cos, 64)) ^ t.cos_sign);
    }
}
extern "C" void roots(const double *x, int64_t count, double *s, double *r)
{
    for (int64_t i = 0; i < count; ++i) {
        s[i] = fx::sqrt_normal(x[i]);
        r[i] = fx::rsqrt_normal(x[i]);
    }
}
extern "C" void flights(const double *q, int64_t count, int32_t *whole, uint64_t *left)
{
    for (int64_t i = 0; i < count; ++i) {
        const fx::Flight f = fx::split_flight(fx::pos_of(q[i]));
        whole[i] = f.whole;
        left[i] = f.left;
    }
}
extern "C" void steps(const int32_t *n, const uint64_t *left, int64_t count, double *t, double *u)
{
    for (int64_t i = 0; i < count; ++i) {
        t[i] = fx::to_double(fx::steps_left(n[i], left[i]));
        u[i] = n[i] > 0 ? fx::from_u32((uint32_t)n[i]) : 0.0;
    }
}
extern "C" void kd(const double *s, int64_t count, double *H, double *F, double *W, double *e)
{
    for (int64_t i = 0; i < count; ++i) {
        const uint64_t x = fx::fraction(s[i] < 1.0 ? s[i] : 0.0);
        const fx::Two p = fx::poly_two<fx::PolyHF>(fx::kPolyHF, x);
        H[i] = fx::to_double(p.a, 65);
        F[i] = fx::to_double(p.b, 64);
        W[i] = fx::to_double_62(fx::poly<fx::PolyW>(fx::kPolyW, fx::fraction(s[i] < 1.0 ? s[i] * 0.36787944117144233 : 0.0)) >> 1, 63);
        e[i] = s[i] >= 0.0625 ? fx::to_double(fx::exp_neg(fx::pos_of(s[i])), 64) : 0.0;
    }
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, so = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as fh:
        fh.write(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    return ctypes.CDLL(so)


def call(f, *args):
    f.restype = None
    f(*[ctypes.c_int64(a) if isinstance(a, int) else a.ctypes.data_as(ctypes.c_void_p) for a in args])


def ulp(x):
    return np.spacing(np.abs(x).astype(np.float64)).astype(np.longdouble)


@pytest.mark.parametrize("B", [53, 24])
def test_logarithm_and_radius(fx, B):
    """Every power of two and its neighbours, both ends of every table
    interval, the smallest uniform, the largest below the near-one branch, and
    random ones."""
    rng = np.random.default_rng(B)
    top = 1 << B
    n = [1, 2, 3, top - (1 << (B - 12)), top - (1 << (B - 12)) - 1]
    for k in range(B):
        n += [(1 << k) - 1, 1 << k, (1 << k) + 1]
    for j in range(129):
        edge = (128 + j) << (B - 8)
        n += [edge - 1, edge, edge + 1]
    n += [int(v) for v in rng.integers(1, top, 20000)] + [int(v) >> int(s) for v, s in
                                                         zip(rng.integers(top // 2, top, 5000), rng.integers(0, B - 1, 5000))]
    n = np.array([v for v in n if 1 <= v <= top - (1 << (B - 12))], np.uint64)
    E, r = np.zeros(len(n)), np.zeros(len(n))
    fx.neg_log.restype = None
    fx.neg_log(B, n.ctypes.data_as(ctypes.c_void_p), ctypes.c_int64(len(n)), E.ctypes.data_as(ctypes.c_void_p),
               r.ctypes.data_as(ctypes.c_void_p))
    exact = -np.log(n.astype(np.longdouble) / np.longdouble(top))
    assert np.all(np.abs(E - exact) <= ulp(E) + np.longdouble(2.0) ** -58)
    root = np.sqrt(2 * exact)
    assert np.all(np.abs(r - root) <= ulp(r) + np.longdouble(2.0) ** -58 / root)


def test_logarithm_near_one(fx):
    w = np.concatenate([[0.0, 2.0**-53, 2.0**-24, 2.0**-12 - 2.0**-53], 2.0 ** -np.random.default_rng(1).uniform(12.01, 52, 2000)])
    E = np.zeros(len(w))
    call(fx.near_one, w, len(w), E)
    exact = -np.log1p(-w.astype(np.longdouble))
    assert E[0] == 0.0
    assert np.all(np.abs(E - exact) <= 2 * ulp(exact))


def test_sine_and_cosine(fx):
    """All octant boundaries and their neighbours, the axes, random phases."""
    rng = np.random.default_rng(3)
    p = [(k << 60) + d for k in range(16) for d in (-2048, -1, 0, 1, 2048)]
    p = np.array([v % (1 << 64) for v in p] + [int(v) << 11 for v in rng.integers(0, 1 << 53, 20000)]
                 + [int(v) << 40 for v in rng.integers(0, 1 << 24, 20000)], np.uint64)
    s, c = np.zeros(len(p)), np.zeros(len(p))
    call(fx.sincos_turn, p, len(p), s, c)
    # the residual from the nearest quarter turn is exact
    k = ((p >> np.uint64(61)) + np.uint64(1)) >> np.uint64(1)
    z = (p - (k << np.uint64(62))).view(np.int64).astype(np.longdouble) * (8 * np.arctan(np.longdouble(1))) / np.longdouble(2) ** 64
    q = (k & np.uint64(3)).astype(int)
    es = np.choose(q, [np.sin(z), np.cos(z), -np.sin(z), -np.cos(z)])
    ec = np.choose(q, [np.cos(z), -np.sin(z), -np.cos(z), np.sin(z)])
    bound = np.longdouble(2.0) ** -54 + np.longdouble(2.0) ** -60
    assert np.all(np.abs(s - es) <= bound) and np.all(np.abs(c - ec) <= bound)
    assert s[2] == 0.0 and c[2] == 1.0


def test_square_roots(fx):
    rng = np.random.default_rng(4)
    x = np.concatenate([[1.0, 2.0, 4.0, 0.25, np.nextafter(1.0, 0), np.nextafter(4.0, 0), np.nextafter(1.0, 2), 2.0**-1022, 1.7e308],
                        2.0 ** rng.uniform(-1000, 1000, 20000)])
    s, r = np.zeros(len(x)), np.zeros(len(x))
    call(fx.roots, x, len(x), s, r)
    xl = x.astype(np.longdouble)
    assert np.all(np.abs(s - np.sqrt(xl)) <= 0.6 * ulp(s))
    assert np.all(np.abs(r - 1 / np.sqrt(xl)) <= 0.6 * ulp(r))


def taylor(coef, n0, s, terms=30):
    """sum_{n >= n0} coef(n) s^(n - n0), smallest terms first."""
    out = np.zeros_like(s)
    for n in range(n0 + terms, n0 - 1, -1):
        out = out * s + coef(n)
    return out


def test_coefficient_polynomials_and_exponential(fx):
    """H = h/s^2, F = f/s^3, W = sqrt(2 h)/h-argument and e^-s over their
    ranges, the ends and tiny arguments among them (e^-s to 2^-58
    absolute)."""
    rng = np.random.default_rng(5)
    s = np.concatenate([[0.0, 2.0**-1000, 2.0**-64, 2.0**-63, 1e-5, 0.5, np.nextafter(1.0, 0)], rng.uniform(0, 1, 20000),
                        2.0 ** -rng.uniform(1, 60, 3000), [1.0, 1.0000001, 43.999999, 44.0, 63.9, 64.0, 1e9],
                        rng.uniform(1, 46, 20000)])
    H, F, W, e = (np.zeros(len(s)) for _ in range(4))
    call(fx.kd, s, len(s), H, F, W, e)
    small = s < 1
    fact = np.cumprod(np.concatenate([[1], np.arange(1, 40)]).astype(np.longdouble))
    t = s[small].astype(np.longdouble)
    h = lambda n: (-1.0) ** n / fact[n]                                # noqa: E731
    f = lambda n: (-1.0) ** n * (2 - n) / fact[n]                      # noqa: E731
    eps = np.longdouble(2.0) ** -60
    for got, exact in ((H[small], taylor(h, 2, t)), (F[small], taylor(f, 3, t)),
                       (W[small], np.sqrt(2 * taylor(h, 2, (s[small] * 0.36787944117144233).astype(np.longdouble))))):
        assert np.all(np.abs(got - exact) <= 0.5 * ulp(exact) + eps)
    big = s >= 0.0625
    exact = np.exp(-s[big].astype(np.longdouble))
    assert np.all(np.abs(e[big] - exact) <= 0.5 * ulp(exact) + np.longdouble(2.0) ** -58)


def test_flights_and_step_counts(fx):
    """Whole steps and the rest of the collision's step of a flight (exact
    down to 2^-64), and their sum back in FP64."""
    from fractions import Fraction
    rng = np.random.default_rng(6)
    q = np.concatenate([[0.0, 5e-324, 2.0**-70, 2.0**-64, 2.0**-63, 0.5, np.nextafter(1.0, 0), 1.0, 1.5, 2.0, 1000.0,
                         2.0**30 - 0.5, 2.0**31 - 1.0, 2.0**31, 2.0**52 + 1, 2.0**63, 2.0**64, 1e300],
                        rng.uniform(0, 3, 2000), 2.0 ** rng.uniform(-60, 40, 2000)])
    w, left = np.zeros(len(q), np.int32), np.zeros(len(q), np.uint64)
    call(fx.flights, q, len(q), w, left)
    for x, a, b in zip(q, w, left):
        f = Fraction(float(x))
        whole = f.numerator // f.denominator
        assert a == min(whole, 2**31 - 1)
        rest = (1 - (f - whole)) * 2**64
        assert 0 <= rest - int(b) <= 1 or abs(rest - int(b)) < 1      # a whole step is 2^64 - 1
    n = np.concatenate([[0, 0, 1, 2, 3, 2**30, 2**31 - 1], rng.integers(0, 2**20, 3000)]).astype(np.int32)
    left = np.concatenate([np.array([1, 2**64 - 1, 2**64 - 1, 0, 1, 2**63, 2**64 - 1], np.uint64),
                           rng.integers(0, 2**63, 3000).astype(np.uint64) * np.uint64(2)])
    t, u = np.zeros(len(n)), np.zeros(len(n))
    call(fx.steps, n, left, len(n), t, u)
    assert np.array_equal(u, n.astype(np.float64))
    for a, b, x in zip(n, left, t):
        exact = Fraction(int(a)) + Fraction(int(b), 2**64)
        assert abs(Fraction(float(x)) - exact) <= Fraction(float(np.spacing(x))) * Fraction(51, 100)
