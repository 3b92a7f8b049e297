"""FP64 pairs that draw the largest uniform of the 24-bit stream, nu = chi = 0
(GPU only), through the per-level and the batched form, one pair per lane,
against the oracle at the FP64 parity bar.
"""
import numpy as np
import pytest

from helpers import fp64_close, gpu_problem, oracle_problem

pytestmark = pytest.mark.gpu


# pairs whose first coarse step is closed by such an event
@pytest.mark.parametrize("seed,pair", [(41, 40879657), (41, 105628815), (1209, 2325), (1815, 9310)])
def test_pairs_that_draw_the_largest_uniform(orc, seed, pair):
    import paper_2004_04071_gb300 as mk
    d = dict(eps=0.01, T=1.0, dt0=0.5, M=2, L=1, qoi=0, init=0, seed=seed)
    want = orc.pairs(oracle_problem(orc, d, recipe=orc.RECIPE_24), 1, pair - 1, 3)
    ctx = mk.Context(0)
    try:
        got = [ctx.debug_pairs(gpu_problem(mk, d, precision=mk.PREC_FP64_U24), 1, pair - 1, 3)]
    finally:
        ctx.close()
    if pair < 20000:
        cfg = mk.batch_config(max_requests=2, max_nbins=8, warp_pair_min_events=-1)
        ctx = mk.Context(0, arena_bytes=mk.batch_workspace_bytes(cfg))
        try:
            fixed = gpu_problem(mk, dict(d, n_fixed=[100, pair + 2]), precision=mk.PREC_FP64_U24)
            got.append([v[pair - 1:] for v in ctx.debug_batch_pairs(fixed, cfg, 1)[1:]])
        finally:
            ctx.close()
    for xf, xc, kf, kc in got:
        assert np.array_equal(kf, want[2]) and np.array_equal(kc, want[3])
        assert np.all(fp64_close(xf, want[0])) and np.all(fp64_close(xc, want[1]))
