"""The work that is timed: products of packed bit matrices over GF(2) and the
Boolean algebra, through the package's public entry points.

A case is a dict with "kind":
  product  one product of resident matrices (gf2 / boolean), sizes m, k, n;
           "depth", "variant", "workspace" where the caller chooses them
  noalloc  the product that allocates nothing (product_noalloc)
  batch    a kept BatchedPlan over many products of uneven sizes, run once
  host     a product of matrices in pinned host memory (product_host)
  transpose  the bit transpose alone

Operands: GF(2) bits are fair coins; Boolean bits are one with probability
1/sqrt(k), which makes about 63 % of the product's bits one (denser operands
give an all-ones product).
"""
import math
import random

import torch

import paper_1909_01554_gb300 as bmm

SIDE = 32768  # longest side of a single product
# bits of k * n that product_noalloc's fixed scratch holds
NOALLOC_BITS = 1 << 26


def listed():
    return [
        # The smallest calls: one product inside a latency-bound loop.
        {"name": "gf2_256x512x384", "kind": "product", "op": "gf2", "m": 256, "k": 512, "n": 384},
        # Ragged middle size, k / 64 odd: a reachability step of a graph of ~2000 nodes.
        {"name": "bool_2112x1984x2240", "kind": "product", "op": "bool", "m": 2112, "k": 1984, "n": 2240},
        # The ordinary size (the repository's first configuration).
        {"name": "gf2_4096", "kind": "product", "op": "gf2", "m": 4096, "k": 4096, "n": 4096},
        # A large matrix times a thin one: a code's generator matrix applied to a block of vectors.
        {"name": "gf2_thin_16384x12288x192", "kind": "product", "op": "gf2", "m": 16384, "k": 12288, "n": 192},
        # Strassen levels chosen by the caller, in a workspace that the caller keeps.
        {"name": "gf2_8192x4096x8192_depth1", "kind": "product", "op": "gf2", "m": 8192, "k": 4096, "n": 8192,
         "depth": 1, "variant": "chaining", "workspace": True},
        # The benchmark's two products: GF(2) with the library's own choice of depth, Boolean cubic.
        {"name": "gf2_32768", "kind": "product", "op": "gf2", "m": 32768, "k": 32768, "n": 32768},
        {"name": "bool_32768", "kind": "product", "op": "bool", "m": 32768, "k": 32768, "n": 32768},
        # The benchmark's batch (sides log-uniform in 256..8192, both products alternating), an eighth of it.
        {"name": "batch256_256_8192", "kind": "batch", "count": 256, "lo": 256, "hi": 8192, "shapes": 5},
        # Many small products in one plan: blocks of a sparse block matrix.
        {"name": "batch512_64_768", "kind": "batch", "count": 512, "lo": 64, "hi": 768, "shapes": 6},
        # A caller that may not allocate device memory while it runs.
        {"name": "noalloc_bool_4096x2048x3072", "kind": "noalloc", "op": "bool", "m": 4096, "k": 2048, "n": 3072},
        # Operands and result in host memory.
        {"name": "host_gf2_8192x16384x8192", "kind": "host", "op": "gf2", "m": 8192, "k": 16384, "n": 8192},
        # The transpose alone, both word counts odd.
        {"name": "transpose_16448x12224", "kind": "transpose", "m": 16448, "n": 12224},
    ]


def _side(rng, lo, hi):
    """A multiple of 64, log-uniform in [lo, hi]."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi, max(lo, int(x / 64 + 0.5) * 64))


def draw(rng):
    r = rng.random()
    op = "gf2" if rng.random() < 0.5 else "bool"
    if r < 0.55:
        c = {"kind": "product", "op": op, "m": _side(rng, 64, SIDE), "k": _side(rng, 64, SIDE), "n": _side(rng, 64, SIDE)}
        if op == "gf2" and rng.random() < 0.3:
            c["depth"] = d = rng.choice([1, 2])
            c["variant"] = rng.choice(["winograd", "self_inverse", "chaining"])
            c["workspace"] = rng.random() < 0.5
            unit = 64 << d
            for s in ("m", "k", "n"):
                c[s] = max(unit, c[s] // unit * unit)
        return c
    if r < 0.72:
        lo = _side(rng, 64, 256)
        hi = _side(rng, 512, 8192)
        # a batch no larger than the listed ones: fewer products where they are big
        most = max(8, min(1024, int(256 * (8192 / hi) ** 1.5)))
        return {"kind": "batch", "count": int(math.exp(rng.uniform(math.log(8), math.log(most)))),
                "lo": lo, "hi": hi, "shapes": rng.randrange(1 << 20)}
    if r < 0.82:
        while True:
            k, n = _side(rng, 64, 16384), _side(rng, 64, 16384)
            if k * n <= NOALLOC_BITS:
                return {"kind": "noalloc", "op": op, "m": _side(rng, 64, 16384), "k": k, "n": n}
    if r < 0.91:
        return {"kind": "host", "op": op, "m": _side(rng, 512, 16384), "k": _side(rng, 512, 16384), "n": _side(rng, 512, 16384)}
    return {"kind": "transpose", "m": _side(rng, 64, SIDE), "n": _side(rng, 64, SIDE)}


def _op(name):
    return bmm.GF2 if name == "gf2" else bmm.BOOL


def _shapes(case):
    """(op, m, k, n) of every product of a batch."""
    rng = random.Random(case["shapes"])
    return [("gf2" if i % 2 == 0 else "bool", *(_side(rng, case["lo"], case["hi"]) for _ in range(3)))
            for i in range(case["count"])]


def _bits(rows, cols, p, gen):
    """A packed rows x cols matrix, int64 words on the GPU; p None: fair coins."""
    words = rows * cols // 64
    if p is None:
        # torch's bounds are exclusive above, so the 64 bits come in two halves
        lo = torch.randint(0, 1 << 32, (words,), dtype=torch.int64, device="cuda", generator=gen)
        hi = torch.randint(0, 1 << 32, (words,), dtype=torch.int64, device="cuda", generator=gen)
        return lo | (hi << 32)
    out = torch.empty(words, dtype=torch.int64, device="cuda")
    shift = torch.arange(64, device="cuda")
    step = 1 << 20  # words at a time
    for at in range(0, words, step):
        w = min(step, words - at)
        ones = torch.rand((w, 64), device="cuda", generator=gen) < p
        out[at:at + w] = (ones.to(torch.int64) << shift).sum(1)
    return out


def _operands(op, m, k, n, gen):
    p = None if op == "gf2" else 1.0 / math.sqrt(k)
    return _bits(m, k, p, gen), _bits(k, n, p, gen)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "transpose":
        m, n = case["m"], case["n"]
        return {"case": case, "X": _bits(m, n, None, gen), "Xt": bmm.empty(n, m)}
    if kind == "batch":
        shapes = _shapes(case)
        ops = [_op(s[0]) for s in shapes]
        AB = [_operands(*s, gen) for s in shapes]
        As, Bs = [a for a, _ in AB], [b for _, b in AB]
        # the results side by side in one buffer, as the blocks of one matrix would be
        words = [m * n // 64 for _, m, _, n in shapes]
        C = torch.empty(sum(words), dtype=torch.int64, device="cuda")
        Cs = list(C.split(words))
        plan = bmm.BatchedPlan(ops, As, Bs, Cs, [s[1] for s in shapes], [s[2] for s in shapes], [s[3] for s in shapes])
        return {"case": case, "As": As, "Bs": Bs, "C": C, "plan": plan}
    m, k, n = case["m"], case["k"], case["n"]
    A, B = _operands(case["op"], m, k, n, gen)
    if kind == "host":
        A, B = A.cpu().pin_memory(), B.cpu().pin_memory()
        return {"case": case, "A": A, "B": B, "C": torch.empty(m * n // 64, dtype=torch.int64).pin_memory()}
    opts = {}
    if "depth" in case:
        opts = {"depth": case["depth"], "variant": {"winograd": bmm.WINOGRAD, "self_inverse": bmm.SELF_INVERSE,
                                                    "chaining": bmm.CHAINING}[case["variant"]]}
        if case.get("workspace"):
            size = bmm.workspace_size(bmm.GF2, m, k, n, **opts)
            opts["workspace"] = torch.empty(size, dtype=torch.uint8, device="cuda")
            opts["workspace_bytes"] = size
    return {"case": case, "A": A, "B": B, "C": bmm.empty(m, n), "opts": opts}


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "transpose":
        bmm.transpose(state["X"], state["Xt"], c["m"], c["n"])
        return state["Xt"]
    if kind == "batch":
        state["plan"].run()
    elif kind == "noalloc":
        bmm.product_noalloc(_op(c["op"]), state["A"], state["B"], state["C"], c["m"], c["k"], c["n"])
    elif kind == "host":
        bmm.product_host(_op(c["op"]), state["A"], state["B"], state["C"], c["m"], c["k"], c["n"])
    elif c["op"] == "gf2":
        bmm.gf2(state["A"], state["B"], state["C"], c["m"], c["k"], c["n"], **state["opts"])
    else:
        bmm.boolean(state["A"], state["B"], state["C"], c["m"], c["k"], c["n"], **state["opts"])
    return state["C"]


def work(case):
    """Operands read once, result written once; one AND and one XOR / OR per bit
    triple (Strassen levels do fewer, but which depth pays is the library's choice)."""
    if case["kind"] == "transpose":
        return {"bytes": 2 * case["m"] * case["n"] // 8, "flops": 0}
    shapes = _shapes(case) if case["kind"] == "batch" else [(case["op"], case["m"], case["k"], case["n"])]
    return {"bytes": sum(m * k + k * n + m * n for _, m, k, n in shapes) // 8,
            "flops": sum(2 * m * k * n for _, m, k, n in shapes)}


def tolerance(case):
    return "exact"  # every output is bits


def _unpack(words, rows, cols):
    """The bits of a packed matrix as float64."""
    shift = torch.arange(64, device="cuda")
    return ((words.reshape(rows, cols // 64, 1) >> shift) & 1).reshape(rows, cols).to(torch.float64)


def _pack(bits, rows, cols):
    shift = torch.arange(64, device="cuda")
    return (bits.reshape(rows, cols // 64, 64).to(torch.int64) << shift).sum(2).reshape(-1)


def _exact_product(op, A, B, m, k, n):
    """Counts in float64 (exact), 4096 rows at a time."""
    b = _unpack(B.cuda(), k, n)
    A = A.cuda().reshape(m, k // 64)
    out = []
    for at in range(0, m, 4096):
        rows = min(4096, m - at)
        count = _unpack(A[at:at + rows].reshape(-1), rows, k) @ b
        out.append(_pack(torch.remainder(count, 2) > 0.5 if op == "gf2" else count > 0.5, rows, n))
    return torch.cat(out)


def exact(case, seed):
    if work(case)["flops"] > 3e12 or case["kind"] == "transpose" and case["m"] * case["n"] > 1 << 28:
        return None
    state = prepare(case, seed)
    if case["kind"] == "transpose":
        m, n = case["m"], case["n"]
        return _pack(_unpack(state["X"], m, n).t().contiguous() > 0.5, n, m)
    if case["kind"] == "batch":
        return torch.cat([_exact_product(s[0], A, B, *s[1:]) for s, A, B in zip(_shapes(case), state["As"], state["Bs"])])
    C = _exact_product(case["op"], state["A"], state["B"], case["m"], case["k"], case["n"])
    return C.cpu() if case["kind"] == "host" else C
