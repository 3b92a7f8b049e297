"""FP64 pairs at the edges of the fixed-point branches (GPU only): s = R theta
below and above 1 and 64, tiny and huge R dt, on both FP64 streams, against
the oracle at the FP64 parity bar, 1e-12 max(1, |x|), with equal event counts.
"""
import math

import numpy as np
import pytest

from helpers import fp64_close, gpu_problem, oracle_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("u24", [False, True])
@pytest.mark.parametrize("rdt", [1e-12, 1e-6, 0.03, 0.5, 0.9999999, 1.0, 1.0000001, 2.0, 43.9, 63.9999, 64.0, 64.0001, 1e3, 1e7])
def test_pairs_at_branch_edges(orc, rdt, u24):
    import paper_2004_04071_gb300 as mk
    d = dict(eps=math.sqrt(0.125 / rdt), T=1.0, dt0=0.5, M=2, L=2, qoi=0, init=0, nbins=0, seed=41)
    ctx = mk.Context(0)
    try:
        for level in (0, 2):
            po = oracle_problem(orc, d, recipe=orc.RECIPE_24 if u24 else None)
            pg = gpu_problem(mk, d, precision=mk.PREC_FP64_U24 if u24 else mk.PREC_FP64)
            xf_o, xc_o, kf_o, kc_o = orc.pairs(po, level, 0, 4001, threads=4)
            xf, xc, kf, kc = ctx.debug_pairs(pg, level, 0, 4001)
            assert np.array_equal(kf, kf_o) and np.array_equal(kc, kc_o)
            assert np.all(fp64_close(xf, xf_o)) and np.all(fp64_close(xc, xc_o))
    finally:
        ctx.close()


@pytest.mark.parametrize("u24", [False, True])
@pytest.mark.parametrize("nbins", [1, 7, 100, 1024])
def test_cosine_start_and_bins(orc, nbins, u24):
    """Initial positions (paths that hardly move, so that x(T) is x_0 and some
    hundred of them lie where the FP64 iteration takes over) and their bins,
    for bin widths that are not powers of two as well: equal counts."""
    import paper_2004_04071_gb300 as mk
    d = dict(eps=50.0, T=0.5, dt0=0.5, M=2, L=0, qoi=1, init=1, nbins=nbins, lo=0.0, hi=1.0, seed=43)
    n = 300007
    ctx = mk.Context(0)
    try:
        po = oracle_problem(orc, d, recipe=orc.RECIPE_24 if u24 else None)
        pg = gpu_problem(mk, d, precision=mk.PREC_FP64_U24 if u24 else mk.PREC_FP64)
        xf_o, xc_o, kf_o, kc_o = orc.pairs(po, 0, 5, n, threads=4)
        xf, _, kf, _ = ctx.debug_pairs(pg, 0, 5, n)
        assert np.array_equal(kf, kf_o) and np.all(fp64_close(xf, xf_o))
        h = ctx.run_level(pg, 0, 5, n)["hist_f"]
        assert np.array_equal(h, orc.level_sums(po, 0, xf_o, xc_o, kf_o, kc_o).hist_f)
    finally:
        ctx.close()
