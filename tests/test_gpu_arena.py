"""The arena belongs to the caller (GPU only): whatever its bytes are when a
call starts, the call's results are the same.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("nbins", [0, 7, 1024])
def test_calls_do_not_read_what_is_left_in_the_arena(prec, nbins):
    """Grids of one block, of one group of blocks and of several groups."""
    import torch
    import paper_2004_04071_gb300 as mk
    kw = dict(eps=0.5, T=0.5, dt0=0.1, M=2, L=2, qoi=0, init=0, precision=prec, seed=47, nbins=nbins, lo=-3.0, hi=3.0)
    p, q = mk.make_problem(**kw), mk.make_problem(n_fixed=[3000, 20000, 100], **kw)
    ctx = mk.Context(0)
    try:
        def estimate():
            e = ctx.estimate(q)
            return dict(enumerate(e.levels), estimate=e.estimate, variance=e.variance)

        gen = torch.Generator(device="cuda:0").manual_seed(1)
        fills = (lambda: ctx.arena.fill_(0xFF), lambda: ctx.arena.fill_(0x01),
                 lambda: ctx.arena.random_(0, 256, generator=gen))
        for n in (100, 5000, 100000):
            for call in (lambda: ctx.run_level(p, 1, 5, n), lambda: dict(enumerate(ctx.debug_pairs(p, 1, 5, n))), estimate):
                want = call()
                for fill in fills:
                    fill()
                    torch.cuda.synchronize()
                    got = call()
                    assert all(np.array_equal(np.asarray(got[k]), np.asarray(want[k])) for k in want), (n, call)
    finally:
        ctx.close()
