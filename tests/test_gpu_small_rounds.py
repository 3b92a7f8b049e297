"""Rounds of little work in the batched form (GPU only): split over many
chunks, with ragged counts, they give the per-level form's pairs exactly once
each: equal counts, events and histograms, sums to 1e-12 of the magnitudes.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("substeps", [0, 16])
@pytest.mark.parametrize("counts", [[1, 1, 1, 1], [2, 31, 32, 33], [1000, 257, 100, 65], [300001, 4099, 1021, 97]])
def test_small_rounds_cover_every_pair_once(counts, substeps):
    import paper_2004_04071_gb300 as mk
    kw = dict(eps=0.2, T=1.0, dt0=0.5, M=2, L=3, qoi=mk.QOI_X2_PERIODIC, init=mk.INIT_COSINE, nbins=32, lo=0.0, hi=1.0, seed=19)
    cfg = mk.batch_config(substeps_per_launch=substeps, max_requests=4, max_nbins=32)
    ctx = mk.Context(0, arena_bytes=mk.batch_workspace_bytes(cfg))
    try:
        p = mk.make_problem(n_fixed=counts, **kw)
        (r,) = ctx.estimate_batch([p], cfg)
        density = np.zeros(32)
        for level, n in enumerate(counts):
            s = ctx.run_level(p, level, 0, n)
            lv = r.levels[level]
            assert lv["n"] == n and lv["events_f"] == s["events_f"] and lv["events_c"] == s["events_c"]
            for k in ("sy", "sy2", "sqf", "sqf2", "sqc", "sqc2"):
                assert abs(lv[k] - s[k]) <= 1e-12 * max(1.0, s["sqf"] + s["sqc"])
            density += (s["hist_f"].astype(float) - s["hist_c"].astype(float)) / n * 32
        assert np.allclose(r.density, density, rtol=0, atol=1e-9)
    finally:
        ctx.close()
