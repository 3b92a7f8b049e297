"""Launches around full waves of the per-level kernel (GPU only): every pair of
a range runs exactly once whatever the split over blocks, so a launch equals
the same range run as two launches: counts, events and histograms exactly,
sums to the summation order.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBLEMS = {
    # one or two events a path; pairs of differing lengths; one event in every step
    "start": (dict(eps=0.5, T=0.5, dt0=0.1, M=2, L=1, qoi=0, init=0), 0),
    "mixed": (dict(eps=0.2, T=1.0, dt0=0.5, M=2, L=3, qoi=1, init=1), 2),
    "deep": (dict(eps=1e-3, T=1.0, dt0=0.5, M=2, L=3, qoi=1, init=1), 1),
}


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_ranges_around_full_waves(name, prec):
    import torch
    import paper_2004_04071_gb300 as mk
    kw, level = PROBLEMS[name]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    p = mk.make_problem(precision=prec, seed=23, nbins=24, lo=-3.0, hi=3.0, **kw)
    ctx = mk.Context(0)
    try:
        for blocks in (4, 5, 6, 8, 9):
            full = sms * blocks * 128
            for n in (full - 1, full, full + 1, full + full // 3, 2 * full - 1, 2 * full + 5, 6 * full + 77):
                whole, cut = ctx.run_level(p, level, 3, n), n // 3 + 1
                a, b = ctx.run_level(p, level, 3, cut), ctx.run_level(p, level, 3 + cut, n - cut)
                for k in ("n", "events_f", "events_c"):
                    assert whole[k] == a[k] + b[k], (n, k)
                for k in ("hist_f", "hist_c", "hist_both"):
                    assert np.array_equal(whole[k], a[k] + b[k]), (n, k)
                for k in ("sy", "sy2", "sqf", "sqf2", "sqc", "sqc2"):
                    assert abs(whole[k] - a[k] - b[k]) <= 1e-9 * (whole["sqf"] + whole["sqc"] + whole["sqf2"]), (n, k)
    finally:
        ctx.close()
