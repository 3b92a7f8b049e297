"""mlkd_debug_kd_coeffs returns what the FP64 pairs use (GPU only): the unit
coefficients D, om, beta and h(s) of the same source compiled for the host.
The two differ in the seed of their square roots only, by a few units of 2^-62
before the rounding to FP64, which then falls to the other side in less than
one value of 50, by one ulp.
"""
import numpy as np
import pytest

import host_pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 3])
def test_readout_is_what_the_pairs_use(precision, tmp_path):
    import torch
    import paper_2004_04071_gb300 as mk
    rng = np.random.default_rng(7)
    s = np.concatenate([2.0 ** rng.uniform(-40, 0, 6000), rng.uniform(1, 64, 6000), 2.0 ** rng.uniform(6, 30, 2000),
                        [np.nextafter(1.0, 0), 1.0, np.nextafter(64.0, 0), 64.0, 65.0, 1e3]])
    nu = np.abs(rng.standard_normal(len(s)))
    nu[::7] = 2.0 ** -rng.uniform(20, 900, len(nu[::7]))
    nu[::31] = 0.0
    D, om, beta, h = host_pairs.units(host_pairs.build(str(tmp_path)), s, nu)
    # R = sigma = 1: s = theta, nu = dv, and no scaling
    t, w = (torch.tensor(v, dtype=torch.float64, device="cuda:0") for v in (s, nu))
    a, d, hs, o, b2 = (v.cpu().numpy() for v in mk.debug_kd_coeffs(precision, 1.0, 0.0, 1.0, t, w))
    for name, got, want in (("d", d, D), ("om", o, om), ("h", hs, h), ("beta^2", b2, beta * beta), ("a", a, nu * om)):
        assert np.all(np.abs(got - want) <= (2 if name == "beta^2" else 1) * np.spacing(want)), name
        assert np.mean(got != want) < 0.02, (name, np.mean(got != want))
