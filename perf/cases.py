"""The work that users of this library have it do, as timed cases.

Every case is one call of a public entry point of
``paper_2601_11621_gb300.capi`` with the default options, on one context that
the process keeps, as a user's program does.  The operations and their ranges:

* ``mul``      bigint_mul of two random operands (the multiplication sweep of
               the benchmark: 2^11 .. 2^26 limbs, ratios 1:1 to 1:4, and below
               it the short operands of everyday calls);
* ``exact``    cat_exact: C(n), C(2n, n) and n!, from the plain sizes to the
               paper's n = 2,050,572,903;
* ``ratio``    cat_ratio_exact of a binomial n! / (k! (n-k)!);
* ``batch``    cat_exact_batch over requests of mixed kind, n log-uniform in
               [10^3, 10^6];
* ``decimal``  to_decimal of a long number;
* ``factor``   catalan_factor: Phase 1 alone, with its primes.

The seed picks the operands' limbs, the requests of a batch, and, where the
input is n itself, an n just below the case's.  Results whose length depends
on the input go into a buffer that the caller keeps, zero above the result,
and their length beside them.
"""
import math

import numpy as np
import torch

from paper_2601_11621_gb300 import capi, workloads

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = capi.Context(0)
    return _ctx


def listed():
    return [
        # one short product: the cost of a call (launch, read-back, binding)
        {"name": "mul_1k", "op": "mul", "na": 1_000, "nb": 700},
        # an everyday product of ragged lengths
        {"name": "mul_200k", "op": "mul", "na": 200_003, "nb": 150_001},
        # the benchmark's 1:4 sweep at 2^22 : 2^20 64-bit words
        {"name": "mul_8m_2m", "op": "mul", "na": 1 << 23, "nb": 1 << 21},
        # the benchmark's 1:1 sweep at 2^24 64-bit words
        {"name": "mul_32m", "op": "mul", "na": 1 << 25, "nb": 1 << 25},
        # the plain method's small size
        {"name": "catalan_1e5", "op": "exact", "kind": 0, "n": 100_000},
        # the plain method's large size
        {"name": "catalan_5e7", "op": "exact", "kind": 0, "n": 50_000_000},
        # the paper's own run
        {"name": "catalan_paper", "op": "exact", "kind": 0, "n": 2_050_572_903},
        # a factorial of the served stream
        {"name": "factorial_3e6", "op": "exact", "kind": 2, "n": 3_000_000},
        # a binomial through the factorial-ratio entry point
        {"name": "binomial_1e7", "op": "ratio", "n": 10_000_000, "k": 3_000_000},
        # the benchmark's batch
        {"name": "batch_4096", "op": "batch", "count": 4096},
        # the decimal text of a number as long as C(5 10^7)
        {"name": "decimal_3m", "op": "decimal", "limbs": 3_124_999},
        # Phase 1 alone
        {"name": "factor_1e8", "op": "factor", "n": 100_000_000},
    ]


def _log(rng, lo, hi):
    """An integer in [lo, hi], uniform in its logarithm."""
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    op = rng.choice(["mul", "mul", "mul", "exact", "exact", "ratio", "batch", "decimal", "factor"])
    if op == "mul":
        na = _log(rng, 500, 1 << 25)
        return {"op": op, "na": na, "nb": max(1, int(na / rng.uniform(1.0, 4.0)))}
    if op == "exact":
        kind = rng.choice([0, 0, 1, 2])
        return {"op": op, "kind": kind,
                "n": _log(rng, 10_000, 10_000_000 if kind == 2 else 1_000_000_000)}
    if op == "ratio":
        n = _log(rng, 10_000, 100_000_000)
        return {"op": op, "n": n, "k": int(n * rng.uniform(0.1, 0.5))}
    if op == "batch":
        return {"op": op, "count": _log(rng, 32, 4096)}
    if op == "decimal":
        return {"op": op, "limbs": _log(rng, 2_000, 1 << 24)}
    return {"op": op, "n": _log(rng, 100_000, 1_000_000_000)}


def _limbs(n, gen):
    """n random limbs on the device, the top bit set."""
    x = torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int32, device="cuda", generator=gen)
    x[-1] |= -(1 << 31)
    return x


def _below(n, seed):
    """An n for this seed: the case's, less at most a thousandth."""
    return n - int(workloads.rng(seed).integers(0, n // 1000 + 1))


def _prime_bound(n):
    """More than the primes of e >= 1 in C(n) (about 2 n ln 2 / ln n)."""
    return int(3 * n * math.log(2) / math.log(n)) + 100


def _buffer(n, dtype=torch.int32):
    return torch.zeros(n, dtype=dtype, device="cuda")


def prepare(case, seed):
    op = case["op"]
    state = {"op": op, "ctx": _context()}
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if op == "mul":
        state["a"], state["b"] = _limbs(case["na"], gen), _limbs(case["nb"], gen)
    elif op == "exact":
        state["kind"], state["n"] = case["kind"], _below(case["n"], seed)
        state["out"] = _buffer(capi.cat_bound_limbs(case["n"], case["kind"]))
    elif op == "ratio":
        n, k = _below(case["n"], seed), case["k"]
        state["num"], state["den"] = [n], [k, n - k]
        state["out"] = _buffer(capi.cat_ratio_bound_limbs([case["n"]], [k, case["n"] - k]))
    elif op == "batch":
        count = case["count"]
        state["reqs"] = workloads.batched_requests(count, seed=seed)
        # the mean request is 9,040 limbs long, with a deviation of 13,000
        state["out"] = _buffer(9_040 * count + int(110_000 * math.sqrt(count)))
    elif op == "decimal":
        state["x"] = _limbs(case["limbs"], gen)
        state["out"] = _buffer(capi.cat_decimal_bound(case["limbs"]), torch.uint8)
    else:
        state["n"] = _below(case["n"], seed)
        state["out"] = _buffer(_prime_bound(case["n"]))
    return state


def run(state):
    ctx, op = state["ctx"], state["op"]
    if op == "mul":
        return capi.bigint_mul(ctx, state["a"], state["b"])
    out = state["out"]
    if op == "exact":
        return [out, capi.cat_exact(ctx, state["kind"], state["n"], out=out).numel()]
    if op == "ratio":
        return [out, capi.cat_ratio_exact(ctx, state["num"], state["den"], out=out).numel()]
    if op == "batch":
        _, offsets, lengths = capi.cat_exact_batch(ctx, state["reqs"], out=out)
        return [out, offsets.astype(np.int64), lengths.astype(np.int64)]
    if op == "decimal":
        return [out, capi.to_decimal(ctx, state["x"], out=out).numel()]
    f = capi.catalan_factor(ctx, state["n"])
    out[:f.num_primes] = f.primes()
    groups = np.zeros((2, 64), dtype=np.int64)  # a Catalan number has at most 33
    groups[0, :len(f.exps)] = f.exps.astype(np.int64)
    groups[1, :len(f.offsets)] = f.offsets.astype(np.int64)
    f.free()
    return [out, groups]


def work(case):
    """Inputs read once, outputs written once.  The arithmetic is on whole
    numbers: there is no floating-point operation to count."""
    op = case["op"]
    if op == "mul":
        b = 8 * (case["na"] + case["nb"])
    elif op == "exact":
        b = 4 * capi.cat_bound_limbs(case["n"], case["kind"])
    elif op == "ratio":
        b = 4 * capi.cat_ratio_bound_limbs([case["n"]], [case["k"], case["n"] - case["k"]])
    elif op == "batch":
        b = 4 * capi.cat_batch_bound(workloads.batched_requests(case["count"], seed=0))
    elif op == "decimal":
        b = 4 * case["limbs"] + capi.cat_decimal_bound(case["limbs"])
    else:
        b = 4 * int(2 * case["n"] * math.log(2) / math.log(case["n"]))
    return {"bytes": b, "flops": 0}


def _int(t):
    return int.from_bytes(t.cpu().numpy().astype("<i4").tobytes(), "little")


def _to_limbs(v, size):
    """v in `size` limbs, and its length (as run returns it)."""
    n = (v.bit_length() + 31) // 32
    return [np.frombuffer(v.to_bytes(4 * size, "little"), dtype="<i4").copy(), n]


def exact(case, seed):
    """CPython's own integers, at the sizes they take a moment for."""
    op = case["op"]
    if op == "mul" and case["na"] + case["nb"] <= 100_000:
        gen = torch.Generator(device="cuda").manual_seed(seed)
        a = _int(_limbs(case["na"], gen))
        return _to_limbs(a * _int(_limbs(case["nb"], gen)), case["na"] + case["nb"])[0]
    if op == "exact" and case["n"] <= 200_000:
        n = _below(case["n"], seed)
        c = math.factorial(n) if case["kind"] == 2 else math.comb(2 * n, n)
        return _to_limbs(c // (n + 1) if case["kind"] == 0 else c,
                         capi.cat_bound_limbs(case["n"], case["kind"]))
    if op == "ratio" and case["n"] <= 200_000:
        n, k = _below(case["n"], seed), case["k"]
        return _to_limbs(math.comb(n, k), capi.cat_ratio_bound_limbs([case["n"]], [k, case["n"] - k]))
    return None
