"""Vectors whose rows start on no 16-byte boundary, at the edges of the kernels' tiles, against the oracle."""
import numpy as np
import pytest
import torch

import draco_inputs as di
from gpu_util import dev, fp32_sequential_sum, host
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


# group sizes of every register variant and of the streamed one (21); a block takes 1024, 512 or 256 columns, fewer on short
# vectors, and the encoder writes 8 less
REPETITION = [(n, s, d) for n, s in [(7, 1), (4, 1), (15, 2), (45, 3), (45, 5), (42, 10)]
              for d in (1, 3, 63, 247, 249, 255, 257, 1021, 30_003)]


@pytest.mark.parametrize("n,s,d", REPETITION)
def test_repetition_rows_off_the_grid(n, s, d):
    import paper_1803_09877_b200 as dr
    plan = dr.Plan(n, s, d, dr.REP)
    G = di.gradient_rows(5 + n + d, n, d)
    buf = torch.full((n * d + 64,), 7.0, dtype=torch.float32, device="cuda")
    plan.encode(dev(G), buf[32:])
    out = host(buf)
    assert (out[:32] == 7.0).all() and (out[32 + n * d:] == 7.0).all()
    Z = out[32:32 + n * d].reshape(n, d)
    groups = orc.rep_groups(n, s)
    for first, size in groups:
        sums = fp32_sequential_sum(G[first:first + size])
        for j in range(first, first + size):
            np.testing.assert_array_equal(Z[j].view(np.uint32), sums.view(np.uint32))
    R = Z.copy()
    adv = di.choose_adversaries(n + d, n, s)
    di.apply_adversaries(R, adv, [di.ADV_REVGRAD] * s, [100.0] * s, seed=3)
    R[groups[0][0]:groups[0][0] + groups[0][1], d - 1] = np.arange(groups[0][1], dtype=np.float32) + 1     # no majority there
    want = orc.rep_decode(R, n, s)
    Rd = dev(R)
    u = torch.full((d + 8,), 7.0, dtype=torch.float32, device="cuda")
    maj = torch.empty((len(groups), d), dtype=torch.float32, device="cuda")
    flags = torch.empty(n, dtype=torch.uint8, device="cuda")
    for _ in range(2):                                    # the second call finds what the first left behind
        plan.rep_vote(Rd, u, maj, flags)
        info = plan.info()
        np.testing.assert_array_equal(host(flags).astype(bool), want["flags"])
        np.testing.assert_array_equal(host(u)[:d].view(np.uint32), fp32_sequential_sum(want["maj"]).view(np.uint32))
        assert (host(u)[d:] == 7.0).all()
        np.testing.assert_array_equal(host(maj).view(np.uint32), want["maj"].view(np.uint32))
        assert info["no_majority"] == want["no_majority"] and info["n_flagged"] == int(np.sum(want["flags"]))
    w = torch.ones(d, dtype=torch.float32, device="cuda")
    plan.decode_update(Rd, flags, w, 0.5)
    np.testing.assert_array_equal(host(w), np.float32(1.0) - np.float32(0.5) * host(u)[:d])


# The few-rows projection takes 512 coordinates per warp and splits the rows of short vectors over blocks.  The tile kernel takes 512
# coordinates per block up to 32,768, and also where full tiles would leave more partials than the locator adds up itself (3 n per
# tile, 8192) and small ones are at most two rounds of blocks (four per SM): n = 45 from 122,881 to 606,208 on 148 SMs, n = 105 from
# 53,249, n = 17 from 327,681; 2048 otherwise.  The recovery takes 64 per block
# up to 300 per SM (44,400), with at most 16 rows 140 (20,720), then 512.
DECODE = [(code, n, s, d) for code in ("CYC", "CYC_PACKED")
          for n, s, d in [(5, 1, 1), (15, 2, 511), (15, 2, 513), (16, 3, 4097), (15, 2, 8200), (17, 2, 513), (45, 5, 2047),
                          (45, 5, 4100), (45, 5, 32_767), (45, 5, 32_770), (45, 5, 65_539), (70, 2, 1025), (105, 2, 33_001), (15, 2, 94_720), (15, 2, 94_722), (15, 2, 95_003), (15, 2, 189_447)]]
DECODE += [(code, n, s, k * d + r) for code, k in (("CYC", 1), ("CYC_PACKED", 2)) for n, s, d in [(15, 2, 20_720), (17, 2, 44_400)] for r in (-1, 0, 1, 2)]
DECODE += [("CYC", n, s, d) for n, s, d in [(45, 5, 122_879), (45, 5, 122_883), (45, 5, 200_003), (45, 5, 303_203), (45, 2, 606_207), (45, 2, 606_211),
                                            (105, 2, 53_249), (105, 2, 100_001), (17, 2, 40_003), (32, 5, 50_001), (24, 4, 100_000), (17, 2, 400_003)]]
DECODE += [("CYC_PACKED", n, s, d) for n, s, d in [(45, 5, 245_767), (45, 5, 400_006), (105, 2, 200_003), (24, 4, 100_003), (45, 2, 1_212_421)]]


@pytest.mark.parametrize("code,n,s,d", DECODE)
def test_projection_and_recovery_at_the_edges_of_their_tiles(code, n, s, d):
    """Projection: exact products, so only the order of fp64 additions differs from the oracle (bars as in test_gpu_cyc.py);
    recovery: fp64 sums of the given vectors, rounded once to fp32 (2^-24 of the largest entry, 1e-7)."""
    import paper_1803_09877_b200 as dr
    packed = code == "CYC_PACKED"
    plan = dr.Plan(n, s, d, getattr(dr, code))
    v = (d + 1) // 2 if packed else d
    G = di.gradient_rows(11 + n + d, n, d)
    R = (orc.cyc_encode_packed if packed else orc.cyc_encode)(G, n, s)
    adv = di.choose_adversaries(n + d, n, s) if v > 64 else []
    di.apply_adversaries(R, adv, [di.ADV_REVGRAD] * len(adv), [100.0] * len(adv), seed=3)
    f = di.projection_vector(7 + d, v)
    Rd, fd = dev(R), dev(f)
    e = torch.empty(3 * n, dtype=torch.float64, device="cuda")
    plan.cyc_project(Rd, fd, e)
    got = host(e)
    eo, qo = orc.cyc_project(R, f), orc.cyc_project_energy(R)
    assert np.abs(got[:2 * n].view(np.complex128) - eo).max() <= 1e-11 * np.sqrt(2 * v * qo.max())
    assert (np.abs(got[2 * n:] - qo) <= 1e-12 * qo).all()
    flags = torch.empty(n, dtype=torch.uint8, device="cuda")
    u = torch.full((d + 8,), 7.0, dtype=torch.float32, device="cuda")
    plan.locate_decode(Rd, fd, flags, u)
    fl = host(flags).astype(bool)
    assert set(adv) <= set(np.flatnonzero(fl))
    want = orc.cyc_decode_packed(R, n, s, fl, d) if packed else orc.cyc_decode(R, n, s, fl)
    assert (host(u)[d:] == 7.0).all()
    assert np.abs(host(u)[:d] - want).max() <= 1e-7 * np.abs(want).max() + 1e-9
    w = torch.ones(d + 8, dtype=torch.float32, device="cuda")
    plan.decode_update(Rd, flags, w, 0.5)
    np.testing.assert_array_equal(host(w)[:d], np.float32(1.0) - np.float32(0.5) * host(u)[:d])
    assert (host(w)[d:] == 1.0).all()


@pytest.mark.parametrize("code", ["REP", "CYC"])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 7, 1021, 4099])
def test_adversary_rows_of_any_alignment(code, d):
    """The values before a row's first 16-byte boundary and after its last whole 16 bytes: same bits as the generator's."""
    import paper_1803_09877_b200 as dr
    n = 9
    plan = dr.Plan(n, 1, d, getattr(dr, code))
    R = di.gradient_rows(31 + d, n, d if code == "REP" else 2 * d)
    if code == "CYC":
        R = np.ascontiguousarray(R).view(np.complex64)
    models, params = [di.ADV_REVGRAD, di.ADV_CONST, di.ADV_GAUSS] * 3, [100.0, 1e4, 1e3] * 3
    Rd = dev(R)
    plan.corrupt(Rd, list(range(n)), models, params, seed=17)
    want = di.apply_adversaries(R.copy(), list(range(n)), models, params, seed=17)
    got = host(Rd, complex64=code == "CYC")
    np.testing.assert_array_equal(np.ascontiguousarray(got).view(np.uint32), np.ascontiguousarray(want).view(np.uint32))


# the second piece has what is left after a multiple of 4096 entries, an eighth of the vector or a little more: odd, a multiple of
# 2, 4 or more, for packed plans also a shorter second half (d odd); packed plans below 70,000 make one copy
@pytest.mark.parametrize("code,d", [(code, d) for code in ("REP", "CYC", "CYC_PACKED") for d in (39_999, 40_000, 40_002, 65_536)]
                         + [("CYC_PACKED", d) for d in (79_999, 80_000, 80_002, 80_004, 131_073)])
def test_host_pipeline_with_a_split_last_chunk(code, d):
    """More than 2 MB of G (packed plans: of its first half): the call copies it in two pieces, and gives the bits of the
    device-resident path."""
    import paper_1803_09877_b200 as dr
    n, s = 15, 2
    cyc, v = code != "REP", (d + 1) // 2 if code == "CYC_PACKED" else d
    plan = dr.Plan(n, s, d, getattr(dr, code))
    G = di.gradient_rows(63 + d, n, d)
    f = di.projection_vector(64 + d, v)
    adv = di.choose_adversaries(65 + d, n, s)
    model, param = [di.ADV_REVGRAD] * s, [100.0] * s
    Z = torch.empty((n, 2 * v if cyc else v), dtype=torch.float32, device="cuda")
    Zh = torch.empty_like(Z)
    plan.encode(dev(G), Z)
    plan.corrupt(Z, adv, model, param, seed=5)
    flags = torch.empty(n, dtype=torch.uint8, device="cuda")
    u = torch.empty(d, dtype=torch.float32, device="cuda")
    plan.locate_decode(Z, dev(f) if cyc else None, flags, u)
    torch.cuda.synchronize()
    Gh, fh = torch.from_numpy(G).pin_memory(), torch.from_numpy(f).pin_memory()
    uh, flh = torch.empty(d).pin_memory(), torch.empty(n, dtype=torch.uint8).pin_memory()
    info = plan.pipeline_host(Gh, fh if cyc else None, adv, model, param, 5, Zh, uh, flh)
    assert torch.equal(Zh, Z) and torch.equal(flh, flags.cpu())
    assert sorted(np.flatnonzero(flh.numpy())) == adv.tolist() and info["n_flagged"] == s
    assert np.abs(uh.numpy() - host(u)).max() <= 2.0 ** -22 * np.abs(host(u)).max()      # e sums in another order: b to 1e-12
