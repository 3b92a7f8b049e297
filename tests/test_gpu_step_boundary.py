"""FP64 pairs with a flight that ends closer to a step boundary than FP64
resolves (GPU only): one pair per lane and one pair per warp, in the per-level
and the batched form, take the same events and end in the same positions, to
the order of their sums (some 100 numbers of order 1).
"""
import numpy as np
import pytest

import host_pairs
from helpers import fp64_close, gpu_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps,pair,u24", host_pairs.AT_BOUNDARY)
def test_both_forms_decide_alike(eps, pair, u24):
    import paper_2004_04071_gb300 as mk
    d = dict(host_pairs.BOUNDARY, eps=eps, n_fixed=[2] * 6 + [32])
    p = gpu_problem(mk, d, precision=mk.PREC_FP64_U24 if u24 else mk.PREC_FP64)
    cfgs = [mk.batch_config(max_requests=2, max_nbins=8, warp_pair_min_events=w) for w in (-1, 1)]
    ctx = mk.Context(0, arena_bytes=max(mk.batch_workspace_bytes(c) for c in cfgs))
    try:
        # 40 000 pairs run one per lane, 32 one per warp
        got = [ctx.debug_pairs(p, 6, 0, n) for n in (40000, 32)] + [ctx.debug_batch_pairs(p, c, 6)[1:] for c in cfgs]
    finally:
        ctx.close()
    want = [v[:32] for v in got[0]]
    for g in got[1:]:
        for a, b in zip(g[2:], want[2:]):
            assert np.array_equal(a[:32], b)
        for a, b in zip(g[:2], want[:2]):
            assert np.all(fp64_close(a[:32], b, 1e-13))


@pytest.mark.parametrize("eps,pair,u24", host_pairs.AT_COARSE_END)
def test_coarse_flights_are_not_negative(eps, pair, u24):
    import paper_2004_04071_gb300 as mk
    p = gpu_problem(mk, dict(host_pairs.FLIGHTS, eps=eps), precision=mk.PREC_FP64_U24 if u24 else mk.PREC_FP64)
    ctx = mk.Context(0)
    try:
        _, E, _, _, taken = ctx.debug_coarse_draws(p, 2, pair, 1, 64)
    finally:
        ctx.close()
    assert len(E) == taken[0] >= 5 and np.all(E >= 0.0)
