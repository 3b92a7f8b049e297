"""The FP64 draws, unit coefficients and pairs of the kernels, compiled for the
host (host_pairs.py), at values that ordinary streams hardly ever meet,
against extended precision and the oracle (no GPU).
"""
import numpy as np
import pytest

import host_pairs
from helpers import fp64_close, oracle_problem

LD = np.longdouble


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_pairs.build(str(tmp_path_factory.mktemp("host")))


def unit_exact(s, nu):
    """D, om and beta of a phase of length s with nu, in extended precision."""
    s, nu = s.astype(LD), nu.astype(LD)
    e, om = np.exp(-s), -np.expm1(-s)

    def h(x):                                                          # e^-x + x - 1
        small, t = np.minimum(x, 1), np.zeros_like(x)
        for n in range(30, 1, -1):
            t = (t + 1) * -small / (n + 1)
        return np.where(x < 1, small * small / 2 * (1 + t), np.exp(-x) + x - 1)

    # f = 2(e - 1) + s(e + 1) = sum_{n>=3} (-s)^n (2 - n)/n!
    small, f = np.minimum(s, 1), np.zeros_like(s)
    fact = np.cumprod(np.concatenate([[1], np.arange(1, 40)]).astype(LD))
    for n in range(35, 2, -1):
        f = f * -small + (2 - n) / fact[n]
    f = np.where(s < 1, -f * small ** 3, s * (1 + e) - 2 * om)
    g = np.where(s < 1, h(s) * om - f, 1 - 2 * s * e - e * e)          # g = h om - f
    return np.sqrt(2 * f + nu * nu * g), om, np.sqrt(2 * h(h(s)))


S = np.array([1e-300, 1e-9, 2.0**-64, 0.03, 0.5, np.nextafter(1.0, 0), 1.0, 1.5, 20.0, 43.99, 44.0, np.nextafter(64.0, 0), 64.0, 65.0,
              1e3, 1e9, 1e100])


@pytest.mark.parametrize("B", [53, 24])
def test_coefficients_at_the_largest_uniform(lib, B):
    """u1 = 1 gives nu = chi = 0 to FP64, at every phase and length: D is that
    of nu = 0.  D: the terms are fixed-point numbers or two FP64 operations,
    then a root (2 ulp); om: one rounding (1 ulp); beta for s >= 1: FP64
    roundings of h (half an ulp each of h and om), magnified up to 2.5 times
    in the root of 2 (e^-h + h - 1) (4 ulp)."""
    phases = np.concatenate([np.arange(1, 17) << (B - 4), (np.arange(1, 17) << (B - 4)) - 3, [1, (1 << (B - 3)) + 1]])
    n = np.array([[1 << B, p, 1 << B] for p in phases for _ in S], np.uint64)
    s = np.tile(S, len(phases))
    nu, chi, E, D, om, beta = host_pairs.draws(lib, B, n, s)
    assert np.all(np.abs(nu) < 1e-150) and np.all(np.abs(chi) < 1e-150) and np.all(E == 0.0)
    for got, exact, k in zip((D, om, beta), unit_exact(s, np.zeros(len(s))), (2, 1, 4)):
        seen = exact >= 2.0**-1021                                     # smaller coefficients are 0
        err = np.abs(got - exact)[seen] / np.spacing(got[seen])
        assert np.all(err <= k), (float(np.max(err)), k, s[seen][np.argmax(err)])
        assert np.all(got[~seen] == 0.0)


@pytest.mark.parametrize("B", [53, 24])
def test_coefficients_of_ordinary_draws(lib, B):
    rng = np.random.default_rng(B)
    n = rng.integers(1, 1 << B, (20000, 3)).astype(np.uint64)
    s = np.concatenate([2.0 ** rng.uniform(-50, 0, 8000), rng.uniform(1, 64, 8000), 2.0 ** rng.uniform(6, 40, 4000)])
    nu, _, _, D, om, beta = host_pairs.draws(lib, B, n, s)
    for got, exact, k in zip((D, om, beta), unit_exact(s, nu), (2, 1, 4)):
        assert np.max(np.abs(got - exact) / np.spacing(got)) <= k


# pairs whose first coarse step is closed by an event with u1 = 1
AT_ONE = [(41, 40879657), (41, 105628815), (1209, 2325), (1815, 9310), (80, 14745)]


@pytest.mark.parametrize("seed,pair", AT_ONE)
def test_pairs_that_draw_the_largest_uniform(lib, orc, seed, pair):
    d = dict(eps=0.01, T=1.0, dt0=0.5, M=2, L=1, qoi=0, init=0, seed=seed)
    xf_o, xc_o, kf_o, kc_o = orc.pairs(oracle_problem(orc, d, recipe=orc.RECIPE_24), 1, pair - 1, 3)
    xf, xc, kf, kc, _ = host_pairs.pairs(lib, d, 1, pair - 1, 3, u24=True)
    assert np.array_equal(kf, kf_o) and np.array_equal(kc, kc_o)
    assert np.all(fp64_close(xf, xf_o)) and np.all(fp64_close(xc, xc_o))


@pytest.mark.parametrize("eps,level", [(0.7, 15), (0.1, 15), (0.7, 13), (0.05, 3)])
def test_warp_form_with_the_most_steps(lib, eps, level):
    """One pair per warp at 2^30 fine steps, the most there are, and at fewer:
    the events of the one-lane form, and its positions to the order of their
    sums (some 100 numbers of order 1, rounded at 2^-53)."""
    d = dict(eps=eps, T=1.0, dt0=1.0, M=4, seed=41)
    lane = host_pairs.pairs(lib, d, level, 0, 24)
    warp = host_pairs.pairs(lib, d, level, 0, 24, warp=400)
    for a, b in zip(warp[2:4], lane[2:4]):
        assert np.array_equal(a, b)
    for a, b in zip(warp[:2], lane[:2]):
        assert np.all(fp64_close(a, b, 1e-13))


@pytest.mark.parametrize("eps,pair,u24", host_pairs.AT_BOUNDARY)
def test_both_forms_decide_alike_at_a_step_boundary(lib, eps, pair, u24):
    d = dict(host_pairs.BOUNDARY, eps=eps)
    lane = host_pairs.pairs(lib, d, 6, pair, 1, u24)
    warp = host_pairs.pairs(lib, d, 6, pair, 1, u24, warp=100)
    for a, b in zip(warp[2:4], lane[2:4]):
        assert np.array_equal(a, b)
    for a, b in zip(warp[:2], lane[:2]):
        assert np.all(fp64_close(a, b, 1e-13))


@pytest.mark.parametrize("B", [53, 24])
def test_normal_variates_keep_their_relative_precision(lib, B):
    """nu and chi near every axis, down to the smallest residual of the phase,
    and on it, where one of them is 0: radius, sine and cosine are right to
    2^-57 relative, and each product is rounded to FP64 once (0.6 ulp)."""
    quarter = 1 << (B - 2)
    off = sorted({0, 1, 2, 3} | {(1 << k) + d for k in range(2, B - 3) for d in (-1, 0, 1)})
    rng = np.random.default_rng(B)
    p = np.array([(q * quarter + s * o) % (1 << B) for q in range(4) for o in off for s in (-1, 1)]
                 + list(rng.integers(0, 1 << B, 4000)), np.uint64)
    p = np.where(p == 0, np.uint64(1 << B), p)                         # uniforms are 1 to 2^B
    n = np.stack([rng.integers(1, 1 << (B - 1), len(p)).astype(np.uint64), p, p], axis=1)
    nu, chi = host_pairs.draws(lib, B, n, 0.5)[:2]
    r = np.sqrt(-2 * np.log(n[:, 0].astype(LD) / LD(1 << B)))
    k = (p + np.uint64(quarter // 2)) // np.uint64(quarter)
    z = (p.astype(np.int64) - k.astype(np.int64) * quarter).astype(LD) * (8 * np.arctan(LD(1))) / LD(1 << B)
    q = (k & np.uint64(3)).astype(int)
    for got, exact in ((nu, r * np.choose(q, [np.cos(z), -np.sin(z), -np.cos(z), np.sin(z)])),
                       (chi, r * np.choose(q, [np.sin(z), np.cos(z), -np.sin(z), -np.cos(z)]))):
        assert np.all(got[exact == 0] == 0.0)
        at = exact != 0
        err = np.abs(got - exact)[at] / np.spacing(np.abs(got[at]))
        assert np.all(err <= 0.6), float(np.max(err))


@pytest.mark.parametrize("B", [53, 24])
def test_logarithm_keeps_its_precision_near_one(lib, B):
    """E = -ln u.  In the last interval, E = rho (1 + rho/2 + ...) < 2^-7.99, the
    inner sum in 32 bits is off by 2 units of 2^-33 and the step above it drops
    2^-41: 2^-55.5 of E, 0.18 ulp.  In the next ones sums of at most 3 units of
    2^-64 and the same of rho^4 at E >= 2^-8: 0.2 ulp.  With one rounding 0.75
    ulp, and below 2^-12 FP64 with a term of 2^-13 at most: a rounding to nearest.  Every power of two of
    1 - u and its neighbours, and the ends of the last intervals."""
    top = 1 << B
    rng = np.random.default_rng(B)
    v = {(1 << k) + d for k in range(B - 1) for d in (-1, 0, 1)} | {int(j * top / 256) + d for j in range(1, 5) for d in (-1, 0, 1)}
    v |= {int(top * 2.0 ** -e) for e in rng.uniform(6, min(40, B - 1), 20000)}
    n = np.array(sorted(top - u for u in v if 0 <= u < top), np.uint64)
    E = host_pairs.draws(lib, B, np.stack([n, n, n], axis=1), 0.5)[2]
    exact = -np.log1p(-((np.uint64(top) - n).astype(LD) / LD(top)))
    at = exact > 0
    assert np.all(E[~at] == 0.0)
    err = ((E - exact)[at] / np.spacing(E[at])).astype(float)
    assert np.max(np.abs(err)) <= 0.75, np.max(np.abs(err))
    small = exact[at] < 2.0**-12
    assert abs(np.mean(err[small])) <= 5 * 0.29 / np.sqrt(np.sum(small)) and np.max(np.abs(err[small])) <= 0.51


@pytest.mark.parametrize("eps,pair,u24", host_pairs.AT_COARSE_END)
def test_coarse_flights_are_not_negative(lib, eps, pair, u24):
    assert host_pairs.pairs(lib, dict(host_pairs.FLIGHTS, eps=eps), 2, pair, 1, u24)[4] >= 0.0


def test_coefficients_of_the_heterogeneous_pairs(lib):
    """kd_coeffs: s < 1 from polynomials (each one rounding, then at most four
    products and a root: 4 ulp of d, 2 of h and om); beyond, FP64 sums of a
    few terms, each rounded at its size, at most ten times the sum's."""
    rng = np.random.default_rng(9)
    s = np.concatenate([2.0 ** rng.uniform(-40, 0, 4000), rng.uniform(1, 70, 4000), [1.0, np.nextafter(1.0, 0), 44.0, 64.0, 1e6]])
    nu = np.abs(rng.standard_normal(len(s)))
    a, d, h, om = host_pairs.units(lib, s, nu, het=True)
    D, om_x, _ = unit_exact(s, nu)
    for got, exact, k in ((d, D, 10), (om, om_x, 2), (a, nu * om_x, 3)):
        assert np.max(np.abs(got - exact) / np.spacing(got)) <= k
