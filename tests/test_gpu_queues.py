"""Started and finished pairs of the per-level kernel are queued 32 at a time
(GPU only): whatever the length of a warp's range, every pair has the same
final state, and the sums are those of the pairs.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBLEMS = {
    # hardly a pair collides; pairs of one to a few events; of differing lengths; of about equal lengths
    "straight": (dict(eps=1.0, T=0.05, dt0=0.05, M=2, L=2, qoi=0, init=2, x0=0.3), 1),
    "few": (dict(eps=0.5, T=0.5, dt0=0.1, M=3, L=1, qoi=0, init=0), 1),
    "mixed": (dict(eps=0.2, T=1.0, dt0=0.5, M=2, L=5, qoi=1, init=1), 5),
    "deep": (dict(eps=1e-2, T=1.0, dt0=0.5, M=2, L=2, qoi=1, init=1), 2),
}


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_pairs_do_not_depend_on_the_range(name, prec):
    import torch
    import paper_2004_04071_gb300 as mk
    kw, level = PROBLEMS[name]
    p = mk.make_problem(precision=prec, seed=19, **kw)
    full = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 128
    first = (1 << 32) - 1000                       # the pair number crosses 32 bits
    ctx = mk.Context(0)
    try:
        whole = ctx.debug_pairs(p, level, first, 3 * full)
        for n in (1, 31, 32, 33, 65, 2049, full + 1, 2 * full + 31, 3 * full):
            part = ctx.debug_pairs(p, level, first, n)
            for a, b in zip(part, whole):
                assert np.array_equal(a, b[:n]), n
            xf, xc, kf, kc = (np.asarray(v[:n], np.float64) for v in whole)
            s = ctx.run_level(p, level, first, n)
            assert (s["n"], s["events_f"], s["events_c"]) == (n, int(kf.sum()), int(kc.sum()))
            ff, fc = (x - np.floor(x) if kw["qoi"] == 1 else x for x in (xf, xc))
            want = dict(sqf=ff**2, sqf2=ff**4, sqc=fc**2, sqc2=fc**4)
            # F of one pair and its square are rounded to float in the FP32 forms (2^-24 each, a few
            # of them, over positive terms), and summed with a compensated or FP64 sum
            rel = 1e-12 if prec in (0, 3) else 1e-6
            for k, v in want.items():
                assert abs(s[k] - v.sum()) <= rel * v.sum(), (n, k)
    finally:
        ctx.close()
