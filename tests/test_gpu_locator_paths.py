"""The ways through the locator: systems of up to eight unknowns solved directly when they certainly have full rank (s
adversaries at work), the singular-value iteration otherwise (fewer adversaries, larger s), nothing solved without adversaries;
the decode vector's elimination for up to eight, up to sixteen and more flags."""
import numpy as np
import pytest
import torch

import draco_inputs as di
from gpu_util import dev, host
from oracle import draco_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s", [1, 2, 3, 4, 5, 6, 7, 8, 9])
@pytest.mark.parametrize("missing", ["none", "one", "all"])
def test_flags_decode_vector_and_sweeps(s, missing):
    import paper_1803_09877_b200 as dr
    n, d = 4 * s + 3, 700
    n_adv = {"none": s, "one": s - 1, "all": 0}[missing]
    plan = dr.Plan(n, s, d, dr.CYC)
    G = di.gradient_rows(900 + s, n, d)
    R = orc.cyc_encode(G, n, s)
    # every other node: far enough apart for complex64 vectors at every s here
    adv = np.arange(0, 2 * n_adv, 2)
    di.apply_adversaries(R, adv, [di.ADV_REVGRAD] * n_adv, [100.0] * n_adv, seed=3)
    f = di.projection_vector(901 + s, d)
    want = orc.cyc_locate(R, f, n, s)
    flags = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
    u = torch.empty(d, dtype=torch.float32, device="cuda")
    plan.locate_decode(dev(R), dev(f), flags, u)
    info = plan.info()
    fl = host(flags).astype(bool)
    np.testing.assert_array_equal(fl, want["flags"])
    assert info["n_flagged"] == int(fl.sum()) and info["n_active"] == n - int(fl.sum())
    assert fl.sum() == n_adv                               # and so the passes end with one that finds nothing and solves nothing
    if n_adv == 0 or n_adv == s <= 8:
        assert info["svd_sweeps"] == 0
    else:
        assert 0 < info["svd_sweeps"] < 60
    b, bo = plan.cyc_decode_vector(), orc.cyc_decode_vector(n, s, fl)
    assert np.abs(b - bo).max() <= 1e-9 * np.abs(bo).max()
    uo = orc.cyc_decode(R, n, s, fl)
    assert np.abs(host(u) - uo).max() <= 1e-6 * np.abs(uo).max()
