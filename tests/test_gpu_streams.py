"""Calls on streams that do not wait for the default one."""
import numpy as np
import pytest
import torch

import draco_inputs as di
from gpu_util import dev, host, normwise
from oracle import draco_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("code,n,s,d", [("CYC", 45, 5, 4100), ("CYC", 15, 2, 300_000), ("CYC_PACKED", 70, 2, 9001), ("CYC", 20, 8, 3001),
                                        ("REP", 15, 2, 20_003)])
def test_first_call_on_a_new_plan_on_a_side_stream(code, n, s, d):
    """Whatever plan creation enqueued (clears, table uploads) is complete when it returns, also while the default stream is busy:
    the plan's first call runs at once on a stream that waits for nothing."""
    import paper_1803_09877_b200 as dr
    cyc, packed = code != "REP", code == "CYC_PACKED"
    v = (d + 1) // 2 if packed else d
    G = di.gradient_rows(5100 + n, n, d)
    R = (orc.cyc_encode_packed if packed else orc.cyc_encode if cyc else orc.rep_encode)(G, n, s)
    adv = di.choose_adversaries(5200 + n, n, s)
    di.apply_adversaries(R, adv, [di.ADV_REVGRAD] * s, [100.0] * s, seed=3)
    f = di.projection_vector(5300 + n, v)
    want = (orc.cyc_locate(R, f, n, s)["flags"] if cyc else orc.rep_decode(R, n, s)["flags"]).astype(bool)
    assert sorted(np.flatnonzero(want)) == adv.tolist()
    Gd, Rd, fd = dev(G), dev(R), dev(f) if cyc else None
    side = torch.cuda.Stream()
    busy = torch.randn(4096, 4096, device="cuda")
    for _ in range(4):
        flags = torch.full((n,), 7, dtype=torch.uint8, device="cuda")
        u = torch.full((d,), 7.0, dtype=torch.float32, device="cuda")
        Z = torch.empty_like(Rd)
        torch.cuda.synchronize()
        for _ in range(8):
            busy = (busy @ busy).clamp_(-1, 1)
        plan = dr.Plan(n, s, d, getattr(dr, code))
        plan.locate_decode(Rd, fd, flags, u, stream=side)
        plan.encode(Gd, Z, stream=side)
        side.synchronize()
        assert np.array_equal(host(flags).astype(bool), want)
        assert plan.info(stream=side)["n_flagged"] == s
        ref = (orc.cyc_decode_packed(R, n, s, want, d) if packed else orc.cyc_decode(R, n, s, want) if cyc
               else orc.rep_decode(R, n, s)["u"])
        assert normwise(host(u), ref) <= 1e-6
        honest = [j for j in range(n) if j not in adv]
        assert normwise(host(Z).reshape(n, -1)[honest], np.ascontiguousarray(R[honest]).view(np.float32)) <= 1e-6
