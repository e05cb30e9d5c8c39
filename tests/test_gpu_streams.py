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


@pytest.mark.parametrize("code,n,s,d", [("REP", 15, 2, 20_003), ("REP", 42, 10, 4096), ("CYC", 20, 8, 3001), ("CYC", 15, 7, 4100),
                                        ("CYC_PACKED", 15, 2, 8002)])
def test_two_chains_captured_on_forked_streams(code, n, s, d):
    """Copies, encodes, adversaries and decodes of two plans in one graph, on two streams that fork and join: replays give the bits of
    the eager calls (kernels set up early, kernels launched in the ordinary way and copies follow one another in it)."""
    import paper_1803_09877_b200 as dr
    cyc, packed = code != "REP", code == "CYC_PACKED"
    v = (d + 1) // 2 if packed else d
    adv = di.choose_adversaries(5400 + n, n, s)
    fd = dev(di.projection_vector(5500 + n, v)) if cyc else None

    class Chain:
        def __init__(self, seed):
            self.plan = dr.Plan(n, s, d, getattr(dr, code))
            self.src = dev(di.gradient_rows(seed, n, d))
            self.G = torch.empty_like(self.src)
            self.Z = torch.empty((n, 2 * v if cyc else v), dtype=torch.float32, device="cuda")
            self.flags = torch.empty(n, dtype=torch.uint8, device="cuda")
            self.u = torch.empty(d, dtype=torch.float32, device="cuda")
            self.outputs = (self.Z, self.flags, self.u)

        def run(self):
            self.G.copy_(self.src)
            self.plan.encode(self.G, self.Z)
            self.plan.corrupt(self.Z, adv, [di.ADV_REVGRAD] * s, [100.0] * s, seed=3)
            self.plan.locate_decode(self.Z, fd, self.flags, self.u)

    a, b = Chain(5600 + n), Chain(5700 + n)
    a.run()
    b.run()
    torch.cuda.synchronize()
    want = [t.clone() for t in a.outputs + b.outputs]
    main, side, graph = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        side.wait_stream(main)
        a.run()
        with torch.cuda.stream(side):
            b.run()
        main.wait_stream(side)
    for _ in range(2):
        for t in (a.G, b.G) + a.outputs + b.outputs:
            t.fill_(3)
        graph.replay()
        torch.cuda.synchronize()
        for got, ref in zip(a.outputs + b.outputs, want):
            assert torch.equal(got, ref)
