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


@pytest.mark.parametrize("packed", [False, True])
@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("n,s", [(1, 0), (4, 0), (5, 1), (9, 2), (9, 3), (15, 3), (17, 4), (45, 5), (13, 6), (45, 7)])
def test_both_sides_of_every_line(n, s, aligned, packed):
    """Lengths on either side of the lines between one output a thread, four, and the walk (warps of outputs per SM): the same bits."""
    import paper_1803_09877_b200 as dr
    if s == 0 and not aligned:
        pytest.skip("one kernel for all lengths")
    code = dr.CYC_PACKED if packed else dr.CYC
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per_warp = (64 if packed else 128) if aligned else (32 if packed else 64)      # coordinates of a warp
    lines = (16, 110 - 10 * s, 140, 180, 300, 9 * (n + 2 * s), 600) if aligned else (16, 60, 100, 140, 200, 300)
    lengths = sorted({int(f * line * sms / n) * per_warp for line in lines for f in (0.97, 1.05)} - {0})
    odd = 0 if aligned else 3
    long = max(lengths) + odd
    G = torch.empty((n, 2 * long if packed else long), dtype=torch.float32, device="cuda").normal_(generator=torch.Generator(device="cuda").manual_seed(n))
    Zl = torch.empty((n, long, 2), dtype=torch.float32, device="cuda")
    dr.Plan(n, s, G.shape[1], code).encode(G, Zl)
    for v in lengths:
        v += odd
        g = torch.cat([G[:, :v], G[:, long:long + v]], 1) if packed else G[:, :v].contiguous()
        if not aligned and packed:
            g = g[:, :-1].contiguous()                                             # an odd length: the last entry lacks its second half
        Z = torch.empty((n, v, 2), dtype=torch.float32, device="cuda")
        dr.Plan(n, s, g.shape[1], code).encode(g, Z)
        whole = v - 1 if packed else v
        assert torch.equal(Z[:, :whole], Zl[:, :whole])
