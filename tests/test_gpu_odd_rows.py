"""Vectors whose rows start on no 16-byte boundary, at the edges of the kernels' tiles, against the oracle."""
import numpy as np
import pytest
import torch

import draco_inputs as di
from gpu_util import dev, host
from oracle import draco_oracle as orc

pytestmark = pytest.mark.gpu

# a block of the fp64 encoder computes 256 coordinates (packed: 128) and writes 252 (124) of each row
ENCODE = ([("CYC", n, s, d) for n, s in [(3, 1), (15, 2), (9, 3), (45, 5), (16, 7)] for d in (1, 3, 251, 253, 255, 257, 505, 1511)]
          + [("CYC_PACKED", n, s, d) for n, s in [(3, 1), (15, 2), (45, 5), (16, 7)] for d in (1, 2, 6, 247, 249, 255, 257, 996, 1511)]
          + [("CYC", 15, 2, 254), ("CYC", 15, 2, 506)])


@pytest.mark.parametrize("code,n,s,d", ENCODE)
def test_cyclic_encode_writes_every_entry_rounded_once(code, n, s, d):
    """The sums are fp64 (relative error of the terms' sum about (2 s + 4) 2^-53), so an entry is off by its rounding to fp32,
    2^-24 of it, and nothing else; Z is surrounded by guard values that stay."""
    import paper_1803_09877_b200 as dr
    plan = dr.Plan(n, s, d, getattr(dr, code))
    G = di.gradient_rows(77 + n + s + d, n, d)
    v = (d + 1) // 2 if code == "CYC_PACKED" else d
    buf = torch.full((2 * n * v + 64,), 7.0, dtype=torch.float32, device="cuda")
    plan.encode(dev(G), buf[32:])
    out = host(buf)
    assert (out[:32] == 7.0).all() and (out[32 + 2 * n * v:] == 7.0).all()
    got = np.ascontiguousarray(out[32:32 + 2 * n * v]).view(np.complex64).reshape(n, v)
    want = (orc.cyc_encode_packed if code == "CYC_PACKED" else orc.cyc_encode)(G, n, s, dtype=np.complex128)
    terms = np.abs(orc.cyc_W(n, s)).sum(axis=0)[:, None] * np.abs(G).max()
    for a, b in ((got.real, want.real), (got.imag, want.imag)):
        assert (np.abs(a - b) <= 2.0 ** -24 * np.abs(b) + 1e-14 * terms * n + 1e-37).all()
