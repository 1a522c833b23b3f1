"""Performance cases of the D2-MHE library: what its users have it compute, through the public calls.

The library's work is one private gradient update: encode, encrypt under the collective key, neighbour
sums, decryption shares, combination, decode.  Training loops call the whole round (d2mhe_round_device,
d2mhe_round_host); a user who sends the messages over a network makes the single calls and needs every
message; a user with primes below 2^30 makes the 32-bit-word calls; conversion to a recipient's own key,
the collective noise refresh and plain ring products are the other entry points.

`listed` holds the workloads that the repository's configurations and benchmark name, and odd sizes
between them; `draw` gives further cases of the same ranges.
"""
import numpy as np
import torch

from paper_2207_04604_b200 import d2mhe
from paper_2207_04604_b200 import workloads as wl

T = wl.PLAIN_MODULUS


def listed():
    return [
        # smallest call: four users on a ring of neighbours, two ciphertexts each; latency and launches count
        dict(name="round_tiny", kind="round", host=False, users=4, degree=2, log2_n=12, bits=36, limbs=3,
             cts=2, chunk=2, ct_first=0, sigma=0.0),
        # one D-PSGD iteration of ten users with a 101,770-parameter perceptron, gradients on the GPU
        dict(name="round_mnist", kind="round", host=False, users=10, degree=4, log2_n=13, bits=54, limbs=4,
             cts=13, chunk=13, ct_first=0, sigma=1e-2),
        # the same iteration when the gradients come from and the sums go to (pinned) host memory
        dict(name="round_mnist_host", kind="round", host=True, users=10, degree=4, log2_n=13, bits=54, limbs=4,
             cts=13, chunk=13, ct_first=0, sigma=1e-2),
        # twenty users with a 1.07 M-parameter convolutional network; the messages of 22 of the 66 indices
        # are in flight at a time
        dict(name="round_cifar", kind="round", host=False, users=20, degree=6, log2_n=14, bits=54, limbs=8,
             cts=66, chunk=22, ct_first=0, sigma=1e-2),
        # fifty users with an 11.2 M-parameter residual network: eight of its 683 ciphertext indices
        dict(name="round_resnet_slice", kind="round", host=False, users=50, degree=8, log2_n=14, bits=54, limbs=8,
             cts=8, chunk=8, ct_first=344, sigma=1e-3),
        # sending side, call by call: odd user and limb counts on the largest ring, all messages kept
        dict(name="send_odd", kind="send", users=7, degree=2, log2_n=14, bits=50, limbs=5, cts=3, ct_first=1000,
             sigma=1e-2),
        # receiving side, call by call: shares of nine holders for every user, combination, decode
        dict(name="receive_odd", kind="receive", users=9, degree=4, log2_n=13, bits=54, limbs=6, cts=11, ct_first=5,
             sigma=1e-2),
        # conversion of the sums to every recipient's own key and decryption under it (Algorithm 2)
        dict(name="convert", kind="convert", users=20, degree=6, log2_n=14, bits=54, limbs=8, cts=2, ct_first=0,
             sigma=1e-2),
        # collective noise refresh of the sums
        dict(name="bootstrap", kind="bootstrap", users=10, degree=4, log2_n=13, bits=54, limbs=4, cts=13, ct_first=0,
             sigma=1e-2),
        # ring multiply-add a b + c with b and c kept in the transform domain: forward, pointwise, inverse
        dict(name="product_8192", kind="product", log2_n=13, bits=54, limbs=8, batch=125),
        # the same on the largest ring, where one polynomial does not fit a thread block, 60-bit primes
        dict(name="product_65536", kind="product", log2_n=16, bits=60, limbs=5, batch=24),
        # the perceptron round on seven 30-bit limbs through the 32-bit-word calls
        dict(name="narrow_mnist", kind="narrow", users=10, degree=4, log2_n=13, bits=30, limbs=7, cts=13, ct_first=0,
             sigma=1e-2),
    ]


def _log_int(rng, lo, hi):
    """An integer of [lo, hi], spread over the logarithm of the range."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    most = max(_ops(c) for c in listed())
    while True:
        kind = rng.choice(["round", "round", "round", "send", "receive", "convert", "bootstrap", "product", "narrow"])
        if kind == "product":
            case = dict(kind=kind, log2_n=rng.randint(11, 16), bits=rng.choice([50, 52, 54, 55, 60]),
                        limbs=rng.randint(1, 12), batch=_log_int(rng, 1, 1024))
            if _ops(case) > most or _state_bytes(case) > 4 << 30:
                continue
            return case
        users = _log_int(rng, 3, 50)
        case = dict(kind=kind, users=users, degree=rng.choice([d for d in (2, 4, 6, 8) if d < users]),
                    log2_n=rng.choice([11, 12, 13, 13, 14, 14]),
                    bits=rng.choice([26, 28, 30]) if kind == "narrow" else rng.choice([36, 48, 50, 54, 54, 55, 60]),
                    limbs=rng.randint(2, 9), cts=_log_int(rng, 1, 60), ct_first=rng.randint(0, 100000),
                    sigma=rng.choice([0.0, 1e-3, 1e-2]))
        if case["bits"] * case["limbs"] < 80:  # the noise of a sum needs room below q / 2t
            continue
        if kind == "round":
            case["host"] = rng.random() < 0.3
            case["chunk"] = rng.randint(max(1, case["cts"] // 4), case["cts"])
        if _ops(case) > most or _state_bytes(case) > 8 << 30:
            continue
        return case


def _moduli(case):
    return wl.ntt_primes(case["bits"], 2 << case["log2_n"], case["limbs"])


def _state_bytes(case):
    n, limbs = 1 << case["log2_n"], case["limbs"]
    word = 4 if case["kind"] == "narrow" else 8
    poly = word * n * limbs
    if case["kind"] == "product":
        return 4 * case["batch"] * poly
    k, c = case["users"], case.get("chunk", case["cts"])
    per_share = 2 * poly if case["kind"] in ("convert", "bootstrap") else poly
    shares = 0 if case["kind"] == "send" else k * k * c * per_share
    return shares + 4 * k * c * poly + 8 * k * case["cts"] * n


def _gradients(case, seed):
    """int32 [users, cts, N] fixed-point gradients on the GPU, clipped so that sums over all users cannot wrap."""
    k, c, n = case["users"], case["cts"], 1 << case["log2_n"]
    clip = ((T - 1) // 2) // k
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["sigma"] > 0:
        g = torch.randn((k, c, n), generator=gen, device="cuda") * case["sigma"]
        return torch.round(g * wl.FIXED_POINT_SCALE).clamp_(-clip, clip).to(torch.int32)
    m = min(4096, clip)
    return torch.randint(-m, m + 1, (k, c, n), generator=gen, device="cuda", dtype=torch.int32)


def _residues(moduli, n, batch, gen):
    out = torch.empty((batch, len(moduli), n), dtype=torch.int64, device="cuda")
    for l, q in enumerate(moduli):
        out[:, l] = torch.randint(0, q, (batch, n), generator=gen, device="cuda", dtype=torch.int64)
    return out


def prepare(case, seed):
    kind, n, limbs = case["kind"], 1 << case["log2_n"], case["limbs"]
    moduli = _moduli(case)
    s = dict(case=case)
    if kind == "product":
        s["ctx"] = d2mhe.Context(case["log2_n"], moduli, 1, seed=seed)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        s["a"], s["b"], s["c"] = (_residues(moduli, n, case["batch"], gen) for _ in range(3))
        s["d"] = torch.empty_like(s["a"])
        return s
    k, c = case["users"], case["cts"]
    s["parties"] = np.arange(k, dtype=np.uint32)
    s["offsets"], s["rows"] = wl.regular_graph(k, case["degree"], seed)
    ctx = s["ctx"] = d2mhe.Context(case["log2_n"], moduli, k, seed=seed)
    ctx.keygen_share(s["parties"])
    ctx.collective_pk(s["parties"])
    values = _gradients(case, seed)
    if kind == "round":
        if case["host"]:
            s["values"] = values.cpu().pin_memory()
            s["sums"] = torch.empty((k, c, n), dtype=torch.int32, pin_memory=True)
        else:
            s["values"], s["sums"] = values, torch.empty_like(values)
        s["workspace"] = torch.empty(ctx.round_workspace_bytes(case["chunk"]), dtype=torch.uint8, device="cuda")
        return s
    s["values"], s["sums"] = values, torch.empty_like(values)
    s["plain"] = ctx.empty_u32(k, c, n)
    empty = ctx.empty_u32 if kind == "narrow" else ctx.empty_u64
    s["ct"], s["agg"] = empty(k, c, 2, limbs, n), empty(k, c, 2, limbs, n)
    if kind == "send":
        return s
    if kind in ("receive", "narrow"):
        s["shares"] = empty(k, k, c, limbs, n)
    else:
        s["shares"] = empty(k, k, c, 2, limbs, n)
        s["ct_out"] = empty(k, c, 2, limbs, n)
    if kind == "convert":
        ctx.user_keygen(s["parties"])
        s["scratch"] = empty(k, c, limbs, n)
    if kind != "narrow":  # the messages that arrived: the sums of every user's neighbourhood
        _send(s)
        s["sent"] = s.pop("ct")
    return s


def _send(s):
    ctx, case = s["ctx"], s["case"]
    k, c = case["users"], case["cts"]
    ctx.encode(s["values"], k * c, s["plain"])
    ctx.encrypt(s["parties"], case["ct_first"], c, s["plain"], s["ct"])
    ctx.aggregate(s["ct"], k, c, s["offsets"], s["rows"], s["agg"])


def run(s):
    ctx, case = s["ctx"], s["case"]
    kind = case["kind"]
    if kind == "product":
        ctx.ntt_forward(s["a"], case["batch"])
        ctx.poly_muladd(s["a"], s["b"], s["c"], s["d"], case["batch"])
        ctx.ntt_inverse(s["d"], case["batch"])
        return [s["a"], s["d"]]
    k, c, first, parties = case["users"], case["cts"], case["ct_first"], s["parties"]
    if kind == "round":
        call = ctx.round_host if case["host"] else ctx.round_device
        call(s["values"], first, c, s["offsets"], s["rows"], s["sums"], s["workspace"])
        return s["sums"]
    if kind == "send":
        _send(s)
        return [s["plain"], s["ct"], s["agg"]]
    if kind == "receive":
        ctx.partial_decrypt(s["agg"], parties, parties, first, c, s["shares"])
        ctx.combine_decrypt(s["agg"], s["shares"], k, k, c, s["plain"])
        ctx.decode(s["plain"], k * c, s["sums"])
        return [s["shares"], s["sums"]]
    if kind == "convert":
        ctx.convert_share(s["agg"], parties, parties, first, c, s["shares"])
        ctx.convert_combine(s["agg"], s["shares"], k, k, c, s["ct_out"])
        ctx.decrypt(parties, s["ct_out"], c, s["scratch"], s["plain"])
        ctx.decode(s["plain"], k * c, s["sums"])
        return [s["shares"], s["ct_out"], s["sums"]]
    if kind == "bootstrap":
        ctx.bootstrap_share(s["agg"], parties, parties, first, c, s["shares"])
        ctx.bootstrap_combine(s["agg"], s["shares"], parties, k, first, c, s["plain"], s["ct_out"])
        return [s["shares"], s["ct_out"]]
    if kind == "narrow":
        ctx.encode(s["values"], k * c, s["plain"])
        ctx.encrypt32(parties, first, c, s["plain"], s["ct"])
        ctx.aggregate32(s["ct"], k, c, s["offsets"], s["rows"], s["agg"])
        ctx.partial_decrypt32(s["agg"], parties, parties, first, c, s["shares"])
        ctx.combine_decrypt32(s["agg"], s["shares"], k, k, c, s["plain"])
        ctx.decode(s["plain"], k * c, s["sums"])
        return [s["ct"], s["agg"], s["shares"], s["sums"]]
    raise ValueError(kind)


def _ops(case):
    """Modular operations of one pass: a transform is (N/2) log2 N butterflies of three, a pointwise
    multiply-add is two, an addition one; a sample counts as ten."""
    n, limbs = 1 << case["log2_n"], case["limbs"]
    transform = 1.5 * n * case["log2_n"]
    if case["kind"] == "product":
        return case["batch"] * limbs * (2 * transform + 2 * n)
    k, units = case["users"], case["users"] * case["cts"]
    encrypt = units * (limbs * (3 * transform + 4 * n) + 30 * n)
    sums = units * limbs * 2 * n * (case["degree"] + 1)
    shares = units * (limbs * ((1 + k) * transform + 2 * k * n) + 10 * k * n)
    combine = units * limbs * n * (k + limbs)
    packing = 2 * units * transform
    if case["kind"] == "send":
        return encrypt + sums + packing / 2
    if case["kind"] == "receive":
        return shares + combine + packing / 2
    if case["kind"] == "convert":
        return units * (limbs * ((3 + 3 * k) * transform + 8 * k * n) + 30 * k * n) + combine + packing / 2
    if case["kind"] == "bootstrap":
        return units * (limbs * ((2 + 2 * k) * transform + 8 * k * n) + 30 * k * n) + combine
    return encrypt + sums + shares + combine + packing


def work(case):
    """Inputs read once, outputs written once.  The whole round leaves only the sums behind; the single
    calls leave every message."""
    n, limbs = 1 << case["log2_n"], case["limbs"]
    poly = (4 if case["kind"] == "narrow" else 8) * n * limbs
    if case["kind"] == "product":
        return {"bytes": 5.0 * case["batch"] * poly, "flops": float(_ops(case))}
    k, c = case["users"], case["cts"]
    packed, ct, share = 4 * n * k * c, 2 * poly * k * c, poly * k * k * c
    nbytes = {
        "round": 2 * packed,
        "send": 2 * packed + 2 * ct,
        "receive": ct + share + packed,
        "convert": ct + 2 * share + ct + packed,
        "bootstrap": ct + 2 * share + ct,
        "narrow": 2 * packed + 2 * ct + share,
    }[case["kind"]]
    return {"bytes": float(nbytes), "flops": float(_ops(case))}


def tolerance(case):
    return "exact"  # residues, plaintexts and sums are whole numbers
