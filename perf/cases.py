"""What the performance of this package is measured on: its products as a
user's program calls them, from the smallest call to the largest single
product, at ragged sizes, in every mode (multiple-precision, operand reuse,
batched in a CUDA graph, complex, binary64 forward and backward).

Matrices hold p random significand bits with the top bit set, random signs and
exponents uniform in a range per entry, some of them with exact zeros (the
recipe of ``synth``, drawn on the GPU); binary64 matrices are normal(0, 1)
times 2^u with u uniform in [-20, 20].

Every result is determined to the last bit: the rounding, once and to nearest
even, of an exact integer.  So outputs are compared exactly.
"""
import math
import random

import torch

import paper_2609_27831_gb300 as ozk
from paper_2609_27831_gb300.autograd import ozaki_matmul


def listed():
    return [
        # the smallest planned product: launches and latency count
        {"name": "gemm_256_p53", "kind": "gemm", "M": 256, "N": 256, "K": 256, "p": 53, "spread": 8, "zeros": 0.0},
        # one call with a cached plan at ragged sizes, about quad precision, a sparse-ish operand
        {"name": "call_ragged_p113", "kind": "call", "M": 611, "N": 347, "K": 923, "p": 113, "spread": 8, "zeros": 0.1},
        # the ordinary product at 256 bits, exponents spread enough to stress the shared scaling
        {"name": "gemm_1024_p256", "kind": "gemm", "M": 1024, "N": 1024, "K": 1024, "p": 256, "spread": 32, "zeros": 0.0},
        # ragged in every dimension, odd leading dimensions, K over one accumulation chunk
        {"name": "gemm_ragged_p512", "kind": "gemm", "M": 1531, "N": 1093, "K": 1777, "p": 512, "spread": 8, "zeros": 0.0},
        # a medium product at the largest precision
        {"name": "gemm_1024_p2048", "kind": "gemm", "M": 1024, "N": 1024, "K": 1024, "p": 2048, "spread": 64, "zeros": 0.0},
        # the largest product: planes streamed through the workspace in groups of moduli
        {"name": "gemm_4096_p2048", "kind": "gemm", "M": 4096, "N": 4096, "K": 4096, "p": 2048, "spread": 64, "zeros": 0.0},
        # large matrices at 53 bits
        {"name": "gemm_8192_p53", "kind": "gemm", "M": 8192, "N": 8192, "K": 8192, "p": 53, "spread": 8, "zeros": 0.0},
        # a matrix kept across products with new blocks of vectors (iterative refinement, block Krylov)
        {"name": "reuse_2048_p256", "kind": "reuse", "M": 2048, "N": 256, "K": 2048, "p": 256, "spread": 8, "zeros": 0.0},
        # many uneven problems in one captured launch
        {"name": "batch_64_graph", "kind": "batch", "count": 64, "lo": 128, "hi": 2048, "shapes": 1002, "spread": 8, "zeros": 0.0},
        # a complex product (three real ones in the residue domain), one call
        {"name": "complex_1024_p256", "kind": "complex", "M": 1024, "N": 1024, "K": 1024, "p": 256, "spread": 8, "zeros": 0.0},
        # binary64 inference at an ordinary ragged size: forward only
        {"name": "f64_forward_ragged", "kind": "f64", "M": 1000, "N": 1304, "K": 2017, "grad": False},
        # binary64 training step at the size of the largest layer: forward and both gradients
        {"name": "f64_train_4096", "kind": "f64", "M": 4096, "N": 4096, "K": 4096, "grad": True},
    ]


_LARGEST = 2.0 * 4096 ** 3 * 879        # plane products of the largest listed case


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "gemm", "call", "reuse", "batch", "complex", "f64", "f64"])
    spread, zeros = rng.choice([0, 8, 32, 64]), rng.choice([0.0, 0.0, 0.1])
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 24), "lo": rng.choice([32, 128]), "hi": rng.choice([512, 1024, 2048]),
                "shapes": rng.randrange(1 << 30), "spread": 8, "zeros": zeros}
    while True:
        if kind == "f64":
            case = {"kind": kind, "M": _log(rng, 64, 6000), "N": _log(rng, 64, 6000), "K": _log(rng, 64, 6000),
                    "grad": rng.random() < 0.5}
        else:
            case = {"kind": kind, "M": _log(rng, 64, 6000), "N": _log(rng, 64, 6000), "K": _log(rng, 64, 6000),
                    "p": _log(rng, 53, 2048), "spread": spread, "zeros": zeros}
        w = work(case)
        if w["flops"] <= 0.3 * _LARGEST and w["bytes"] <= 6e9:
            return case


# ---------------------------------------------------------------------------
# The work of a product: a p-bit entry is ceil(p / 64) limbs, an exponent and
# a sign; one exact integer product of int8-range planes per one-limb modulus
# and three per two-limb modulus (the paper's modulus set for t = p + 16 +
# ceil(log2 K) internal bits).
# ---------------------------------------------------------------------------
def _moduli():
    sieve = [True] * 16192
    primes = []
    for q in range(2, 16192):
        if sieve[q]:
            primes.append(q)
            sieve[q * q::q] = [False] * len(range(q * q, 16192, q))
    one = []
    for q in primes:
        if q > 255:
            break
        m = q
        while m * q <= 255:
            m *= q
        one.append(m)
    return sorted(one, reverse=True) + [q for q in reversed(primes) if q > 255]


_MODULI = _moduli()


def _planes(K, p, inner=None):
    inner = inner or K
    t = p + 16 + math.ceil(math.log2(inner))
    bits, need, g = 0.0, 2 * t + 2 + math.log2(inner), 0
    for m in _MODULI:
        if bits > need:
            break
        bits += math.log2(m)
        g += 1 if m <= 255 else 3
    return g


def _entry(p):
    return 8 * ((p + 63) // 64) + 5


def _shapes(case):
    r = random.Random(case["shapes"])
    return [(_log(r, case["lo"], case["hi"]), _log(r, case["lo"], case["hi"]), _log(r, case["lo"], case["hi"]),
             r.choice([113, 256, 512])) for _ in range(case["count"])]


def _product(M, N, K, p):
    return {"bytes": (M * K + K * N + M * N) * _entry(p), "flops": 2.0 * M * N * K * _planes(K, p)}


def work(case):
    if case["kind"] == "batch":
        each = [_product(*s) for s in _shapes(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    M, N, K = case["M"], case["N"], case["K"]
    if case["kind"] == "f64":
        one = 2.0 * M * N * K * _planes(K, 53, max(M, N, K) if case["grad"] else None)
        inout = M * K + K * N + M * N
        return {"bytes": 8 * inout * (2 if case["grad"] else 1) + (8 * (M * K + K * N) if case["grad"] else 0),
                "flops": one * (3 if case["grad"] else 1)}
    w = _product(M, N, K, case["p"])
    if case["kind"] == "complex":            # 3M: three plane products, two parts of every matrix
        return {"bytes": 2 * w["bytes"], "flops": 3 * w["flops"]}
    return w


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _matrix(gen, rows, cols, p, spread, zeros):
    nl = (p + 63) // 64
    limbs = torch.randint(-2 ** 63, 2 ** 63 - 1, (nl, rows, cols), dtype=torch.int64, device="cuda", generator=gen)
    if 64 * nl - p:
        limbs[0] &= -(1 << (64 * nl - p))
    limbs[nl - 1] |= -2 ** 63
    exp = torch.randint(-spread, spread + 1, (rows, cols), dtype=torch.int32, device="cuda", generator=gen)
    sign = torch.randint(0, 2, (rows, cols), dtype=torch.int8, device="cuda", generator=gen)
    if zeros:
        keep = torch.rand((rows, cols), device="cuda", generator=gen) >= zeros
        limbs *= keep
        exp *= keep
        sign *= keep
    return ozk.MPMatrix(limbs, exp, sign, p)


def _double(gen, rows, cols, scaled=True):
    x = torch.randn((rows, cols), dtype=torch.float64, device="cuda", generator=gen)
    if scaled:
        x = torch.ldexp(x, torch.randint(-20, 21, (rows, cols), device="cuda", generator=gen))
    return x


def _f64_inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    M, N, K = case["M"], case["N"], case["K"]
    return _double(gen, M, K), _double(gen, K, N), _double(gen, M, N, scaled=False) if case["grad"] else None


def prepare(case, seed):
    kind = case["kind"]
    if kind == "f64":
        A, B, dC = _f64_inputs(case, seed)
        return {"case": case, "A": A.requires_grad_(case["grad"]), "B": B.requires_grad_(case["grad"]), "dC": dC}
    gen = torch.Generator(device="cuda").manual_seed(seed)
    spread, zeros = case["spread"], case["zeros"]
    if kind == "batch":
        # outputs of all problems side by side in three buffers
        shapes = _shapes(case)
        size = sum(M * N for M, N, K, p in shapes)
        words = sum(M * N * ((p + 63) // 64) for M, N, K, p in shapes)
        out = (torch.empty(words, dtype=torch.int64, device="cuda"), torch.empty(size, dtype=torch.int32, device="cuda"),
               torch.empty(size, dtype=torch.int8, device="cuda"))
        triples, at, word = [], 0, 0
        for M, N, K, p in shapes:
            n, nl = M * N, (p + 63) // 64
            C = ozk.MPMatrix(out[0][word:word + nl * n].view(nl, M, N), out[1][at:at + n].view(M, N),
                             out[2][at:at + n].view(M, N), p)
            at, word = at + n, word + nl * n
            triples.append((_matrix(gen, M, K, p, spread, zeros), _matrix(gen, K, N, p, spread, zeros), C))
        plan = ozk.Plan(shapes)
        ws = plan.workspace()
        graph = plan.graph(triples, ws, torch.cuda.Stream())
        return {"case": case, "plan": plan, "triples": triples, "ws": ws, "graph": graph, "out": out}
    M, N, K, p = case["M"], case["N"], case["K"], case["p"]
    A, B = _matrix(gen, M, K, p, spread, zeros), _matrix(gen, K, N, p, spread, zeros)
    if kind == "call":
        return {"case": case, "A": A, "B": B}
    if kind == "complex":
        return {"case": case, "A": A, "Ai": _matrix(gen, M, K, p, spread, zeros), "B": B,
                "Bi": _matrix(gen, K, N, p, spread, zeros)}
    C = ozk.MPMatrix.empty(M, N, p)
    plan = ozk.Plan((M, N, K, p))
    ws = plan.workspace()
    state = {"case": case, "A": A, "B": B, "C": C, "plan": plan, "ws": ws}
    if kind == "reuse":
        if plan.info["plane_groups"] > 1:    # streamed planes cannot be kept
            plan = state["plan"] = ozk.Plan((M, N, K, p), plane_group=-1)
            ws = state["ws"] = plan.workspace()
        plan.execute(A, _matrix(gen, K, N, p, spread, zeros), C, ws)   # an earlier product with this A
    return state


def run(state):
    kind = state["case"]["kind"]
    if kind == "gemm":
        C = state["C"]
        state["plan"].execute(state["A"], state["B"], C, state["ws"])
    elif kind == "reuse":
        C = state["C"]
        state["plan"].execute_reuse(0, state["B"], C, state["ws"])
    elif kind == "call":
        C = ozk.gemm(state["A"], state["B"])
    elif kind == "complex":
        Cr, Ci = ozk.zgemm(state["A"], state["Ai"], state["B"], state["Bi"])
        return [Cr.limbs, Cr.exp, Cr.sign, Ci.limbs, Ci.exp, Ci.sign]
    elif kind == "batch":
        state["graph"].launch()
        return list(state["out"])
    else:
        A, B = state["A"], state["B"]
        if not state["case"]["grad"]:
            return [ozaki_matmul(A, B)]
        C = ozaki_matmul(A, B)
        dA, dB = torch.autograd.grad(C, (A, B), state["dC"])
        return [C.detach(), dA, dB]
    return [C.limbs, C.exp, C.sign]


def tolerance(case):
    return "exact"


def exact(case, seed):
    # multiple-precision outputs are whole numbers (significand words, exponents, signs)
    if case["kind"] != "f64":
        return None
    A, B, dC = _f64_inputs(case, seed)
    if not case["grad"]:
        return [A @ B]
    return [A @ B, dC @ B.T, A.T @ dC]
