"""Per-level launches of few long FP64 pairs run one pair per warp (GPU only):
the same pairs in a launch of many run one per lane.  Event counts agree
exactly, positions to the order of their sums.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBLEMS = {
    # one event in every step; of differing lengths; long flights; coarse windows of 3, 8 and 64 steps
    "deep": (dict(eps=1e-2, T=1.0, dt0=0.5, M=2, L=7, qoi=1, init=1), 7),
    "mixed": (dict(eps=0.1, T=1.0, dt0=0.5, M=2, L=8, qoi=1, init=1, nbins=32, lo=0.0, hi=1.0), 8),
    "long": (dict(eps=0.1, T=1.0, dt0=0.5, M=2, L=13, qoi=1, init=1), 13),
    "m3": (dict(eps=0.05, T=0.5, dt0=0.1, M=3, L=4, qoi=0, init=0, mu=0.3), 4),
    "m8": (dict(eps=0.05, T=0.5, dt0=0.1, M=8, L=3, qoi=0, init=2, x0=-0.7), 3),
    "m64": (dict(eps=0.03, T=0.5, dt0=0.5, M=64, L=1, qoi=1, init=1), 1),
}


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_warp_form_equals_lane_form(name, prec):
    import paper_2004_04071_gb300 as mk
    kw, level = PROBLEMS[name]
    p = mk.make_problem(precision=prec, seed=31, **kw)
    first = (1 << 32) - 500                        # the pair number crosses 32 bits
    ctx = mk.Context(0)
    try:
        lane = ctx.debug_pairs(p, level, first, 40000)
        for n in (1, 3, 4, 5, 33, 1000, 3041, 5000):
            part = ctx.debug_pairs(p, level, first, n)
            for a, b in zip(part[2:], lane[2:]):
                assert np.array_equal(a, b[:n]), n
            # up to 1024 additions of numbers below about 4, each rounded at 2^-53, in either form
            for a, b in zip(part[:2], lane[:2]):
                assert np.max(np.abs(a - b[:n]) / np.maximum(1.0, np.abs(b[:n]))) <= 1e-12, n
            xf, xc, kf, kc = (np.asarray(v, np.float64) for v in part)
            for s in (ctx.run_level(p, level, first, n), mk.run_level_noalloc(p, level, first, n)):
                assert (s["n"], s["events_f"], s["events_c"]) == (n, int(kf.sum()), int(kc.sum()))
                ff, fc = (x - np.floor(x) if kw["qoi"] == 1 else x for x in (xf, xc))
                for k, v in dict(sqf=ff**2, sqf2=ff**4, sqc=fc**2, sqc2=fc**4).items():
                    assert abs(s[k] - v.sum()) <= 1e-12 * v.sum(), (n, k)
                if kw.get("nbins"):
                    assert int(np.sum(s["hist_f"])) == n and int(np.sum(s["hist_c"])) == n
    finally:
        ctx.close()
