"""Performance cases: what a training loop asks of the library, through its public entry points.

An iteration encodes the n workers' vectors from the per-partition gradients (``Plan.encode``), the server receives them with
up to s of them adversarial, finds the adversaries and recovers the gradient sum (``Plan.locate_decode``, or ``Plan.locate`` +
``Plan.decode`` / ``Plan.decode_update``).  A case names one of these calls, or a whole iteration, for one code and size:

    encode   G -> Z
    decode   R -> flags, u                       (locate_decode)
    update   R -> flags, w <- w - scale D(R)     (locate, then the decoder fused with the SGD step)
    step     G -> Z -> adversaries -> flags, u   (encode, corrupt, locate, decode: the benchmark's iteration)
    host     the same from and to host buffers   (pipeline_host)

Code "rep" is the repetition code (fp32 vectors), "cyc" the cyclic code (complex64 vectors), "cycp" the cyclic code on the packed
gradient (half as many complex64 entries).  Inputs are drawn with torch on the GPU from the seed.  The received matrix of the
decode cases is formed here in fp64 from the code's coefficient matrix, so that it does not depend on the library's encoder.
"""
import math

import numpy as np
import torch

import paper_1803_09877_b200 as dr

CODES = {"rep": dr.REP, "cyc": dr.CYC, "cycp": dr.CYC_PACKED}
MODELS = {"revgrad": (dr.ADV_REVGRAD, 100.0), "const": (dr.ADV_CONST, 1e4), "gauss": (dr.ADV_GAUSS, 1e3)}
UPDATE_SCALE = 1e-3
MAX_BYTES = 32.5e9          # of a drawn case: the largest listed one


def listed():
    return [
        # the smallest configuration of the repetition code: 15 workers, groups of 5, 100 k coordinates; every iteration of a
        # small model pays these two calls, and launches count as much as bytes
        dict(name="rep_encode_n15_100k", op="encode", code="rep", n=15, s=2, d=100_000, adv=0, model="revgrad"),
        dict(name="rep_decode_n15_100k", op="decode", code="rep", n=15, s=2, d=100_000, adv=2, model="revgrad"),
        # a ResNet-18-sized gradient on 45 workers, adversaries of two kinds
        dict(name="rep_decode_n45_11.7M", op="decode", code="rep", n=45, s=3, d=11_700_000, adv=3, model="mixed"),
        # the paper's 45 workers and 5 adversaries with a parameter count that is no multiple of anything: groups of 11 and 12,
        # the sum goes straight into the weights
        dict(name="rep_update_n45_odd", op="update", code="rep", n=45, s=5, d=5_000_011, adv=5, model="revgrad"),
        # a very short vector: the decoder's latency (projection, locator, recovery) is all there is
        dict(name="cyc_decode_n45_4k", op="decode", code="cyc", n=45, s=5, d=4096, adv=5, model="revgrad"),
        # the small configuration of the cyclic code, whole iteration on the GPU, and the same from host buffers
        dict(name="cyc_step_n15_1M", op="step", code="cyc", n=15, s=2, d=1_000_000, adv=2, model="gauss"),
        dict(name="cyc_host_n15_1M", op="host", code="cyc", n=15, s=2, d=1_000_000, adv=2, model="gauss"),
        # a ResNet-152-sized gradient on 45 workers with s = 5, either direction
        dict(name="cyc_encode_n45_60.2M", op="encode", code="cyc", n=45, s=5, d=60_200_000, adv=0, model="revgrad"),
        dict(name="cyc_decode_n45_60.2M", op="decode", code="cyc", n=45, s=5, d=60_200_000, adv=5, model="revgrad"),
        # odd parameter counts: no row but the first starts on a 16-byte boundary
        dict(name="cyc_encode_n45_odd", op="encode", code="cyc", n=45, s=3, d=3_000_017, adv=0, model="revgrad"),
        dict(name="cyc_update_n45_odd", op="update", code="cyc", n=45, s=5, d=1_000_003, adv=4, model="const"),
        # the packed transport at full size, whole iteration
        dict(name="cycp_step_n45_60.2M", op="step", code="cycp", n=45, s=5, d=60_200_000, adv=5, model="revgrad"),
    ]


def draw(rng):
    """One more case of the same ranges: n, s and the vector lengths of the configurations and of what lies between them, half
    of the lengths multiples of four (as sharding leaves them), the others as they come."""
    while True:
        op = rng.choice(["encode", "encode", "decode", "decode", "update", "step", "host"])
        code = rng.choice(["rep", "cyc", "cyc", "cycp"])
        n = rng.choice([15, 15, 45, 45, 105, rng.randint(7, 64)])
        s = rng.choice([1, 2, 3, 5, 7])
        if 2 * s + 1 > n:
            continue
        if code != "rep" and op in ("step", "host") and _kappa(n, s) > 3e5:
            continue                    # the sum has too few digits to compare once the vectors are rounded to complex64
        if code != "rep" and _kappa(n, s) > 1e10:
            continue
        lo, hi = (4096, 2_000_000) if op == "host" else (4096, 60_200_000)
        d = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
        if rng.random() < 0.5:
            d -= d % 4
        adv = 0 if op == "encode" else rng.choice([0, s, s, rng.randint(1, s)])
        case = dict(op=op, code=code, n=n, s=s, d=d, adv=adv, model=rng.choice(["revgrad", "const", "gauss", "mixed"]))
        if work(case)["bytes"] <= MAX_BYTES:
            return case


def _vlen(case):
    return (case["d"] + 1) // 2 if case["code"] == "cycp" else case["d"]


def _kappa(n, s):
    """How far the cyclic decoder cancels: about the largest coefficient of the code, n^(-1/2) prod |w^s - w^m| over the
    n - 2 s - 1 roots m = 2 s + 1 .. n - 1."""
    p = n ** -0.5
    for m in range(2 * s + 1, n):
        p *= 2.0 * abs(math.sin(math.pi * (m - s) / n))
    return max(p, 1.0)


def _adversaries(case, seed):
    g = torch.Generator().manual_seed(seed + 1)
    nodes = torch.randperm(case["n"], generator=g)[: case["adv"]].sort().values.tolist()
    names = ["revgrad", "const"] if case["model"] == "mixed" else [case["model"]]
    kinds = [MODELS[names[k % len(names)]] for k in range(len(nodes))]
    return nodes, [k[0] for k in kinds], [k[1] for k in kinds]


def _received(case, plan, gen, seed):
    """R: the workers' vectors, formed in fp64 and rounded once, with the adversaries' rows in place."""
    n, d, v = case["n"], case["d"], _vlen(case)
    cyc = case["code"] != "rep"
    R = torch.empty((n, 2 * v if cyc else v), dtype=torch.float32, device="cuda")
    if cyc:
        W = torch.from_numpy(plan.cyc_W()).cuda()
        Wr, Wi = W.real.t().contiguous(), W.imag.t().contiguous()           # z_j = sum_k W[k][j] g_k
    for c0 in range(0, v, 1 << 20):
        c1 = min(v, c0 + (1 << 20))
        if not cyc:
            G = torch.randn((n, c1 - c0), generator=gen, device="cuda")
            for first, size in plan.groups():
                acc = G[first].clone()
                for k in range(1, size):
                    acc += G[first + k]
                R[first:first + size, c0:c1] = acc
        else:
            G = torch.randn((n, c1 - c0), generator=gen, device="cuda").double()
            zr, zi = Wr @ G, Wi @ G
            if case["code"] == "cycp":
                G = torch.randn((n, c1 - c0), generator=gen, device="cuda").double()
                if d % 2 and c1 == v:
                    G[:, -1] = 0.0                                         # the packed vector's last imaginary part
                zr, zi = zr - Wi @ G, zi + Wr @ G
            out = R.view(n, v, 2)[:, c0:c1]
            out[..., 0] = zr
            out[..., 1] = zi
    nodes, models, params = _adversaries(case, seed)
    if nodes:
        plan.corrupt(R, nodes, models, params, seed=seed + 2)
    return R


def prepare(case, seed):
    n, d, v, op = case["n"], case["d"], _vlen(case), case["op"]
    cyc = case["code"] != "rep"
    gen = torch.Generator(device="cuda").manual_seed(seed)
    plan = dr.Plan(n, case["s"], d, CODES[case["code"]])
    st = dict(op=op, code=case["code"], plan=plan, f=None)
    if cyc:
        st["f"] = torch.randn(v, generator=gen, device="cuda") + 1.0       # the locator's draw of N(1, 1)
    if op in ("encode", "step", "host"):
        st["G"] = torch.empty((n, d), dtype=torch.float32, device="cuda").normal_(generator=gen)
        st["Z"] = torch.empty((n, 2 * v if cyc else v), dtype=torch.float32, device="cuda")
        st["adv"], st["models"], st["params"] = _adversaries(case, seed)
        st["noise_seed"] = seed + 2
    else:
        st["R"] = _received(case, plan, gen, seed)
    st["flags"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    if op == "update":
        st["w"] = torch.empty(d, dtype=torch.float32, device="cuda").normal_(generator=gen)
    else:
        st["u"] = torch.empty(d, dtype=torch.float32, device="cuda")
    if op == "host":
        for k in ("G", "f", "u", "flags"):
            if st[k] is not None:
                st[k] = torch.empty(st[k].shape, dtype=st[k].dtype, pin_memory=True).copy_(st[k])
    return st


def run(st):
    plan, op = st["plan"], st["op"]
    if op == "encode":
        plan.encode(st["G"], st["Z"])
        return st["Z"]
    if op == "decode":
        plan.locate_decode(st["R"], st["f"], st["flags"], st["u"])
        return st["flags"], st["u"]
    if op == "update":
        plan.locate(st["R"], st["f"], st["flags"])
        plan.decode_update(st["R"], st["flags"], st["w"], UPDATE_SCALE)
        return st["flags"], st["w"]
    if op == "step":
        plan.encode(st["G"], st["Z"])
        plan.corrupt(st["Z"], st["adv"], st["models"], st["params"], seed=st["noise_seed"])
        if st["code"] == "rep":
            plan.locate_decode(st["Z"], None, st["flags"], st["u"])
        else:
            plan.locate(st["Z"], st["f"], st["flags"])
            plan.decode(st["Z"], st["flags"], st["u"])
        return st["Z"], st["flags"], st["u"]
    plan.pipeline_host(st["G"], st["f"], st["adv"], st["models"], st["params"], st["noise_seed"], st["Z"], st["u"], st["flags"])
    return st["Z"], st["flags"], st["u"]


def work(case):
    """Bytes: gradients, worker vectors, f, flags, sum or weights, each once.  Flops: the filter's, the projection's and the
    recovery's multiply-adds; additions and comparisons of the repetition code."""
    n, s, d, v, op = case["n"], case["s"], case["d"], _vlen(case), case["op"]
    cyc = case["code"] != "rep"
    vec = (8 if cyc else 4) * n * v
    taps = 4.0 * (2 * s + 1) * n * d if cyc else 1.0 * n * d
    back = (12.0 if cyc else 2.0) * n * v
    if op == "encode":
        return {"bytes": 4 * n * d + vec, "flops": taps}
    read = vec + (4 * v if cyc else 0) + n
    if op == "decode":
        return {"bytes": read + 4 * d, "flops": back}
    if op == "update":
        return {"bytes": read + 8 * d, "flops": back + 2.0 * d}
    return {"bytes": 4 * n * d + vec + (4 * v if cyc else 0) + n + 4 * d, "flops": taps + back}


def tolerance(case):
    """The repetition code is exact (copies, comparisons, one fixed order of fp32 additions).  Cyclic vectors are complex64
    roundings of sums taken in more than fp32: 2.5e-8 is the rounding alone, 3e-8 to 6e-8 was seen against fp64.  A decoded sum
    carries fp64 rounding times the code's cancellation k where the vectors are given (2.5e-8 seen, 5e-8 at k = 1e9), and the
    vectors' complex64 rounding times k where they were encoded in the same pass (0.8e-8 k to 1.4e-8 k seen)."""
    if case["code"] == "rep":
        return "exact"
    k = _kappa(case["n"], case["s"])
    if case["op"] == "encode":
        return {"rel": 2e-7, "max": 1e-6}
    if case["op"] in ("step", "host"):
        return {"rel": min(0.03, 2e-7 + 4e-8 * k), "max": min(1.0, 1e-6 + 2.5e-7 * k)}
    return {"rel": 1e-7 + 1e-16 * k, "max": 4e-7 + 1e-15 * k}


def _code_matrix(n, s):
    """W[j][k] = n^(-1/2) prod (w^k - w^m) over the n - 2 s - 1 columns m outside j .. j + 2 s, zero on those columns."""
    w = np.exp(np.clongdouble(2j) * np.arccos(np.longdouble(-1)) * np.arange(n) / n)
    W = np.zeros((n, n), dtype=np.clongdouble)
    for j in range(n):
        outside = [(j + t) % n for t in range(2 * s + 1, n)]
        for k in [(j + t) % n for t in range(2 * s + 1)]:
            W[j, k] = np.prod(w[k] - w[outside]) / np.sqrt(np.longdouble(n))
    return W.astype(np.complex128)


def _decode_vector(n, s, nodes):
    """The minimum-norm b, zero on the adversaries, with [C_L] b = (0, .., 0, 1)."""
    U = [j for j in range(n) if j not in nodes]
    C = np.exp(2j * np.pi * (np.outer(np.arange(n - 2 * s), U) % n) / n) / math.sqrt(n)
    last = np.zeros(n - 2 * s, dtype=np.complex128)
    last[-1] = 1.0
    b = np.zeros(n, dtype=np.complex128)
    b[U] = np.linalg.lstsq(C, last, rcond=None)[0]
    return b


def exact(case, seed):
    """The same in fp64: sums of the inputs by the code's definition, vectors combined with the decode vector of the true
    adversary set.  Adversaries' Gaussian noise has no counterpart outside the library: no worker vectors then."""
    n, s, d, v, op = case["n"], case["s"], case["d"], _vlen(case), case["op"]
    cyc, packed = case["code"] != "rep", case["code"] == "cycp"
    st = prepare(case, seed)
    nodes, models, params = _adversaries(case, seed)
    flags = torch.zeros(n, dtype=torch.uint8)
    flags[nodes] = 1
    r = 2 * s + 1
    sizes = [n // (n // r) + (g < n % (n // r)) for g in range(n // r)]
    first = [sum(sizes[:g]) for g in range(n // r)]
    if op in ("decode", "update"):
        R, u = st["R"], torch.empty(d, dtype=torch.float64, device="cuda")
        if cyc:
            honest = [j for j in range(n) if j not in nodes]
            b = _decode_vector(n, s, nodes)[honest]
            b = torch.from_numpy(np.stack([b.real, b.imag])).cuda()
        else:
            honest = [next(j for j in range(f, f + m) if j not in nodes) for f, m in zip(first, sizes)]
        for c0 in range(0, v, 1 << 20):
            c1 = min(v, c0 + (1 << 20))
            if not cyc:
                u[c0:c1] = R[honest, c0:c1].double().sum(0)
                continue
            x = R.view(n, v, 2)[honest, c0:c1].double()
            u[c0:c1] = b[0] @ x[..., 0] - b[1] @ x[..., 1]
            if packed:
                c2 = min(c1, d - v)
                u[v + c0:v + c2] = (b[0] @ x[..., 1] + b[1] @ x[..., 0])[: max(c2 - c0, 0)]
        return flags, u if op == "decode" else st["w"].double() - UPDATE_SCALE * u
    G = st["G"].cuda()
    Z = None
    if op == "encode" or not any(m == MODELS["gauss"][0] for m in models):
        Z = torch.empty((n, 2 * v if cyc else v), dtype=torch.float64, device="cuda")
        W = torch.from_numpy(_code_matrix(n, s)).cuda() if cyc else None
        for c0 in range(0, v, 1 << 20):
            c1 = min(v, c0 + (1 << 20))
            g = G[:, c0:c1].double()
            if not cyc:
                for f, m in zip(first, sizes):
                    Z[f:f + m, c0:c1] = g[f:f + m].sum(0)
            else:
                Wr, Wi, out = W.real.t().contiguous(), W.imag.t().contiguous(), Z.view(n, v, 2)[:, c0:c1]
                zr, zi = Wr @ g, Wi @ g
                if packed:
                    h = torch.zeros_like(g)
                    c2 = min(c1, d - v)
                    h[:, : c2 - c0] = G[:, v + c0:v + c2]
                    zr, zi = zr - Wi @ h, zi + Wr @ h
                out[..., 0], out[..., 1] = zr, zi
        if op != "encode":
            for j, model, param in zip(nodes, models, params):
                if model == MODELS["revgrad"][0]:
                    Z[j] *= -param
                else:
                    Z[j] = param
                    if cyc:
                        Z[j, 1::2] = 0.0
    if op == "encode":
        return Z
    u = torch.empty(d, dtype=torch.float64, device="cuda")
    for c0 in range(0, d, 1 << 20):
        u[c0:c0 + (1 << 20)] = G[:, c0:c0 + (1 << 20)].double().sum(0)
    return Z, flags, u
