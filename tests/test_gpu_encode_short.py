"""Encoders of short vectors (one or four outputs per thread) against those of long ones, which walk all rows: the same operations on
every entry, hence the same bits.  A long vector's first columns are encoded by themselves."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# (n, s): fewest rows, a last group of 1, 2, 3 and 4 outputs, every number of taps; d: one output, four and the walk (by the warps per SM)
NS = [(1, 0), (3, 1), (5, 2), (15, 2), (17, 2), (9, 3), (18, 4), (45, 5), (13, 6), (15, 7), (31, 7), (105, 3)]


@pytest.mark.parametrize("packed", [False, True])
@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("n,s", NS)
def test_short_vectors_have_the_bits_of_long_ones(n, s, aligned, packed):
    import paper_1803_09877_b200 as dr
    if s == 0 and not aligned:
        pytest.skip("one kernel for all lengths")
    code = dr.CYC_PACKED if packed else dr.CYC
    long = 20_000_000 // n // 16 * 16 + 16 + (0 if aligned else 3)              # more than 600 warps of outputs per SM
    gen = torch.Generator(device="cuda").manual_seed(n + s)
    G = torch.empty((n, long), dtype=torch.float32, device="cuda").normal_(generator=gen)
    vl = (long + 1) // 2 if packed else long
    Zl = torch.empty((n, vl, 2), dtype=torch.float32, device="cuda")
    dr.Plan(n, s, long, code).encode(G, Zl)
    for d in (8, 136, 264, 1000, 60_000 // n * 8, 1_200_000 // n * 8):
        if not aligned:
            d += 3
        v = (d + 1) // 2 if packed else d
        g = torch.zeros((n, d), dtype=torch.float32, device="cuda")
        g[:, :v] = G[:, :v]
        if packed:
            g[:, v:] = G[:, vl:vl + d - v]
        buf = torch.full((n * v * 2 + 64,), 7.0, dtype=torch.float32, device="cuda")
        dr.Plan(n, s, d, code).encode(g, buf[32:])
        assert (buf[:32] == 7.0).all() and (buf[32 + 2 * n * v:] == 7.0).all()
        Z = buf[32:32 + 2 * n * v].view(n, v, 2)
        whole = d - v                                                           # packed: the last entry may lack its second half
        assert torch.equal(Z[:, :whole if packed else v], Zl[:, :whole if packed else v])
