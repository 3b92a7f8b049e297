"""Launches with a second, partial wave of blocks (GPU only): pairs of at least
8 events, and more of them than 32 per warp of one wave but fewer than twice
that (FP32 pairs of one event a step: up to seven times).  Sizes on both sides
of a wave for every number of blocks an SM may hold, so that the split is met
whatever the build's occupancy.  Every pair runs exactly once: a launch equals
the same range run in parts that fit one wave, counts, events and histograms
exactly, sums to the summation order; and the same range in the form without a
context, whose rows limit the split.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBLEMS = {
    # events expected per pair: 17 of 32 steps, 16 of 16, 30 of 32
    "mixed": (dict(eps=0.2, T=1.0, dt0=0.5, M=2, L=4, qoi=1, init=1, lo=0.0, hi=1.0), 4),
    "deep": (dict(eps=1e-3, T=1.0, dt0=0.5, M=2, L=3, qoi=0, init=0, lo=-3.0, hi=3.0), 3),
    "b1": (dict(eps=1.0, T=1.0, dt0=1.0, M=2, L=5, qoi=3, init=2, x0=1.0, lo=0.0, hi=2.0, background=1, bg_a=10.0, bg_b=100.0), 5),
}


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_every_pair_once(name, prec):
    import torch
    import paper_2004_04071_gb300 as mk
    kw, level = PROBLEMS[name]
    assert kw["qoi"] != 3 or mk.QOI_X == 3
    p = mk.make_problem(precision=prec, seed=29, nbins=24, **kw)
    wave = torch.cuda.get_device_properties(0).multi_processor_count * 128
    sizes = sorted({wave * b + d for b in range(2, 14) for d in (0, 1, wave // 3)})
    if name == "deep":
        sizes += [wave * b * k - 5 for b in (6, 7, 8) for k in (3, 5, 7)]
    ctx = mk.Context(0)
    try:
        # parts of one warp-load for every warp of the smallest wave
        step, part = wave, []
        for i in range(max(sizes) // step + 1):
            part.append(ctx.run_level(p, level, 3 + i * step, step))
        for n in sizes:
            m = n // step
            tail = [ctx.run_level(p, level, 3 + m * step, n - m * step)] if n % step else []
            for whole in (ctx.run_level(p, level, 3, n), mk.run_level_noalloc(p, level, 3, n)):
                for k in ("n", "events_f", "events_c"):
                    assert whole[k] == sum(v[k] for v in part[:m] + tail), (n, k)
                for k in ("hist_f", "hist_c", "hist_both"):
                    assert np.array_equal(whole[k], sum(v[k] for v in part[:m] + tail)), (n, k)
                for k in ("sy", "sy2", "sqf", "sqf2", "sqc", "sqc2"):
                    want = sum(v[k] for v in part[:m] + tail)
                    assert abs(whole[k] - want) <= 1e-9 * (whole["sqf"] + whole["sqc"] + whole["sqf2"]), (n, k)
    finally:
        ctx.close()
