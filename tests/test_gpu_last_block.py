"""The last block of a per-level launch closes it (GPU only): calls of one to
thousands of blocks in any order, with and without histograms, leave nothing
behind for the next call, and the allocation-free form gives the same results.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = (1, 127, 129, 700000, 2, 40000, 128)


@pytest.mark.parametrize("prec", [0, 2])
def test_calls_leave_nothing_behind(prec):
    import paper_2004_04071_gb300 as mk
    kw = dict(eps=0.5, T=0.5, dt0=0.1, M=2, L=2, qoi=0, init=0, precision=prec, seed=41, lo=-3.0, hi=3.0)
    first = {}
    ctx = mk.Context(0)
    try:
        for turn, nbins in enumerate((0, 8, 128, 8)):
            p = mk.make_problem(nbins=nbins, **kw)
            for n in SIZES:
                runs = [ctx.run_level(p, 1, 5, n), mk.run_level_noalloc(p, 1, 5, n)]
                for r in runs:
                    assert r["n"] == n
                    # the two forms may split the pairs over different grids
                    want = first.setdefault(n, r)
                    for k in ("events_f", "events_c"):
                        assert r[k] == want[k], (turn, n, k)
                    for k in ("sy", "sy2", "sqf", "sqf2", "sqc", "sqc2"):
                        assert abs(r[k] - want[k]) <= 1e-9 * (want["sqf"] + want["sqc"] + want["sqf2"]), (turn, n, k)
                    if nbins:
                        assert int(np.sum(r["hist_f"])) <= n
                if nbins:
                    hist = first.setdefault((n, nbins), runs[0])
                    for r in runs:
                        for k in ("hist_f", "hist_c", "hist_both"):
                            assert np.array_equal(r[k], hist[k]), (turn, n, nbins, k)
    finally:
        ctx.close()


@pytest.mark.parametrize("prec", [0, 2])
def test_row_groups(prec):
    """Grids around the sizes where block rows fall into groups: the sums are
    those of the pairs."""
    import paper_2004_04071_gb300 as mk
    p = mk.make_problem(eps=0.5, T=0.5, dt0=0.1, M=2, L=1, qoi=0, init=0, precision=prec, seed=43)
    ctx = mk.Context(0)
    try:
        whole = ctx.debug_pairs(p, 1, 0, 128 * 300)
        for blocks in (1, 2, 15, 16, 63, 64, 65, 66, 75, 76, 90, 91, 225, 226, 300):
            for n in (128 * blocks - 127, 128 * blocks):
                xf, xc, kf, kc = (np.asarray(v[:n], np.float64) for v in whole)
                for s in (ctx.run_level(p, 1, 0, n), mk.run_level_noalloc(p, 1, 0, n)):
                    assert (s["n"], s["events_f"], s["events_c"]) == (n, int(kf.sum()), int(kc.sum()))
                    # the square of a position in FP32 is rounded once (2^-24) over positive terms
                    rel = 1e-12 if prec == 0 else 1e-6
                    for k, x in (("sqf", xf), ("sqc", xc)):
                        assert abs(s[k] - (x * x).sum()) <= rel * (x * x).sum(), (n, k)
    finally:
        ctx.close()
