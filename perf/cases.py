"""Workloads of the RNS-CKKS library, through the Python binding a program uses (paper_2606_10477_gb300.hedap).

A case is one call (or the two calls of Mul_P by a constant and its use) on resident ciphertexts of one of the
parameter presets; its outputs are the whole residue arrays of the resulting ciphertexts, copied on the device.
Every operation is exact modular arithmetic on 64-bit words, so equal inputs give equal words.

The server of the paper owns one key set and receives many inputs (Sec. 4.2): the contexts (prime tables and keys
from a fixed key seed) and their rotation keys are kept per preset, the inputs are new for every seed.
"""
import math

import numpy as np
import torch

from paper_2606_10477_gb300 import hedap, inputs

KEY_SEED = 1
_contexts = {}
_bootstrapped = set()  # (preset, log2 of the slots) whose keys and diagonals exist


def _context(preset):
    """The key owner's context of a preset (bootstrapping configured where its chain is made for it)."""
    if preset not in _contexts:
        p = inputs.PRESETS[preset]
        ctx = hedap.Context(p["log_n"], p["q_bits"], p["p_bits"], p["alpha"], p["log_scale"], p["hw"], KEY_SEED,
                            stream=torch.cuda.current_stream().cuda_stream)
        if preset.startswith("bts"):
            ctx.bts_setup(**inputs.BTS)
        _contexts[preset] = ctx
    return _contexts[preset]


def listed():
    return [
        # the smallest call: one addition in the toy ring (a record added to a running sum)
        {"name": "add_toy", "op": "add", "preset": "toy", "level": 11, "batch": 1},
        # one product with rescale in the smallest ring, the unit step of a Newton iteration there: launches count
        {"name": "mul_n10", "op": "mul", "preset": "n10", "level": 5, "batch": 1},
        # one rotation of a ragged batch below the top of a mid-size chain (rotate-and-add of statistics)
        {"name": "rotate_n13_b3", "op": "rotate", "preset": "n13", "level": 6, "batch": 3, "steps": -4},
        # the transform alone, forward: the batch the benchmark reports its rate on (16 polynomials of 24 limbs)
        {"name": "ntt_fwd_n16", "op": "ntt", "preset": "n16", "limbs": 24, "polys": 16, "first": 0, "inverse": False},
        # the inverse transform of one ciphertext of 23 limbs that begins inside the chain and ends in P
        {"name": "ntt_inv_n16", "op": "ntt", "preset": "n16", "limbs": 23, "polys": 2, "first": 3, "inverse": True},
        # Mul_P by a constant with its rescale: the pre-normalisation a / B of a full batch
        {"name": "mul_const_n16_b8", "op": "mul_const", "preset": "n16", "level": 23, "batch": 8, "value": 0.37},
        # one ciphertext product with rescale at the top of the benchmark's chain: the latency of a single query
        {"name": "mul_n16", "op": "mul", "preset": "n16", "level": 23, "batch": 1},
        # the same for the benchmark's batch of eight
        {"name": "mul_n16_b8", "op": "mul", "preset": "n16", "level": 23, "batch": 8},
        # the three-digit key switch (eight primes a digit) half-way down its chain, a ragged last digit
        {"name": "mul_n16d3_b3", "op": "mul", "preset": "n16d3", "level": 18, "batch": 3},
        # several rotations of one ciphertext that share one ModUp (baby steps of a linear transform)
        {"name": "hoisted_n16_b2", "op": "rotate_hoisted", "preset": "n16", "level": 14, "batch": 2, "count": 5},
        # a whole CryptoInvSqrt: the benchmark's batch, degree and Newton steps
        {"name": "invsqrt_n16_b8", "op": "invsqrt", "preset": "n16", "level": 23, "batch": 8, "degree": 15, "iters": 4},
        # a whole bootstrap of one ciphertext on the full-size chain (ModRaise, CoeffToSlot, EvalMod, SlotToCoeff)
        {"name": "bootstrap_bts16", "op": "bootstrap", "preset": "bts16", "level": 3, "batch": 1},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: the listed operations over every preset's ring and chain, batches 1 to 8, any level."""
    op = rng.choice(["add", "mul", "mul", "rotate", "ntt", "ntt", "mul_const", "rotate_hoisted", "invsqrt", "bootstrap"])
    if op == "bootstrap":  # the small ring, sparse or full slots
        return {"op": op, "preset": "bts12", "level": rng.randint(1, 6), "batch": _log_int(rng, 1, 8),
                "log_slots": rng.choice([0, 5, 8, 10])}
    if op == "invsqrt":
        return {"op": op, "preset": rng.choice(["toy", "n16", "n16d3"]), "level": 11, "batch": _log_int(rng, 1, 8),
                "degree": rng.choice([3, 7, 11, 15]), "iters": rng.randint(0, 3)}
    preset = rng.choice(["n10", "toy", "n12a4", "n13", "bts12", "n16", "n16", "n16d3"])
    p = inputs.PRESETS[preset]
    top = len(p["q_bits"]) - 1
    if op == "ntt":
        total = top + 1 + len(p["p_bits"])
        limbs = rng.randint(1, total)
        return {"op": op, "preset": preset, "limbs": limbs, "polys": _log_int(rng, 1, 16),
                "first": rng.randint(0, total - limbs), "inverse": rng.random() < 0.5}
    case = {"op": op, "preset": preset, "level": rng.randint(1, top), "batch": _log_int(rng, 1, 8)}
    if op == "rotate":
        case["steps"] = rng.choice([-1, 1]) << rng.randint(0, 5)
    elif op == "rotate_hoisted":
        case["count"] = rng.randint(2, 5)
    elif op == "mul_const":
        case["value"] = round(rng.uniform(-2.0, 2.0), 3)
    return case


def _residues(ctx, seed, first, limbs, parts):
    """[parts][limbs][N] uniform residues of the primes first.. (what a ciphertext's words look like)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.empty((parts, limbs, ctx.N), dtype=torch.int64, device="cuda")
    for i, q in enumerate(ctx.primes()[first:first + limbs]):
        x[:, i] = torch.randint(0, int(q), (parts, ctx.N), generator=g, device="cuda")
    return x


def _ciphertexts(ctx, seed, level, batch, scale):
    return ctx.batch_import(_residues(ctx, seed, 0, level + 1, 2 * batch), batch, level, scale)


def prepare(case, seed):
    op, ctx = case["op"], _context(case["preset"])
    st = {"op": op, "ctx": ctx, "case": case}
    if op == "ntt":
        # the transform works in place, so every pass takes the last one's output: residues as uniform as the first
        st["x"] = _residues(ctx, seed, case["first"], case["limbs"], case["polys"])
    elif op in ("invsqrt", "bootstrap"):
        # encryptions of real records: uniform in [0.01, 1] for InvSqrt, in [-1, 1] for a bootstrap
        lo = 0.01 if op == "invsqrt" else -1.0
        n = ctx.N // 2
        rep = 1 << case["log_slots"] if case.get("log_slots") else n
        vals = [np.tile(inputs.uniform_values(1000 * seed + k, rep, lo, 1.0), n // rep) for k in range(case["batch"])]
        st["a"] = ctx.pack([ctx.encrypt(v, case["level"], 1000 * seed + 7 + k) for k, v in enumerate(vals)])
        slots = case.get("log_slots") or ctx.log_n - 1
        if op == "bootstrap" and (case["preset"], slots) not in _bootstrapped:
            # rotation keys and encoded diagonals are made by the first bootstrap; a server holds them
            ctx.bootstrap_scaled_slots(ctx.unpack(st["a"], 0), 1, slots)
            _bootstrapped.add((case["preset"], slots))
    else:
        st["a"] = _ciphertexts(ctx, 2 * seed, case["level"], case["batch"], ctx.scale)
        if op in ("add", "mul"):
            st["b"] = _ciphertexts(ctx, 2 * seed + 1, case["level"], case["batch"], ctx.scale)
        if op == "rotate":
            ctx.gen_galois_key(ctx.galois_of_rotation(case["steps"]))
        if op == "rotate_hoisted":
            st["steps"] = list(range(1, case["count"] + 1))
            for s in st["steps"]:
                ctx.gen_galois_key(ctx.galois_of_rotation(s))
    torch.cuda.synchronize()
    return st


def _words(ctx, ct, batch):
    """The whole residue array of a batch, on the device."""
    out = torch.empty((batch, 2, ct.level + 1, ctx.N), dtype=torch.int64, device="cuda")
    ctx.batch_export(ct, out)
    return out


def run(st):
    op, ctx, case = st["op"], st["ctx"], st["case"]
    if op == "ntt":
        return ctx.ntt_batch(st["x"], case["limbs"], case["first"], inverse=case["inverse"])
    n = case["batch"]
    if op == "add":
        return _words(ctx, ctx.add(st["a"], st["b"]), n)
    if op == "mul":
        return _words(ctx, ctx.mul(st["a"], st["b"]), n)
    if op == "mul_const":
        return _words(ctx, ctx.mul_const(st["a"], case["value"], ctx.scale), n)
    if op == "rotate":
        return _words(ctx, ctx.rotate(st["a"], case["steps"]), n)
    if op == "rotate_hoisted":
        return [_words(ctx, c, n) for c in ctx.rotate_hoisted(st["a"], st["steps"])]
    if op == "invsqrt":
        return _words(ctx, ctx.invsqrt(st["a"], 0.01, 1.0, 1.0, case["degree"], case["iters"]), n)
    if case.get("log_slots"):
        return _words(ctx, ctx.bootstrap_scaled_slots(st["a"], 1, case["log_slots"]), n)
    return _words(ctx, ctx.bootstrap_scaled(st["a"], 1), n)


# ---------------------------------------------------------------- what a pass cannot do without
def _shape(preset):
    p = inputs.PRESETS[preset]
    return 1 << p["log_n"], p["log_n"], len(p["q_bits"]), len(p["p_bits"]), p["alpha"]


def _key_bytes(preset, l):
    n, _, _, k, a = _shape(preset)
    return 16.0 * n * -(-(l + 1) // a) * (l + 1 + k)


def _switch_ops(preset, l, batch):
    """Word operations (a modular product or sum is one) of a hybrid key switch at level l: the transforms (three
    a butterfly), the basis conversions and the key products."""
    n, log_n, _, k, a = _shape(preset)
    dn, ext = -(-(l + 1) // a), l + 1 + k
    new = dn * ext - (l + 1)
    limbs = (l + 1) + new + 2 * k + 2 * (l + 1)  # a rescale shares ModDown's transform and adds its last limb's
    return batch * n * (1.5 * log_n * limbs + 2.0 * a * new + 4.0 * dn * ext + 4.0 * k * (l + 1))


def work(case):
    op = case["op"]
    n, log_n, n_q, k, a = _shape(case["preset"])
    if op == "ntt":
        limbs = case["limbs"] * case["polys"]
        return {"bytes": 16.0 * n * limbs, "flops": 1.5 * n * log_n * limbs}
    l, b = case["level"], case["batch"]
    ct = 16.0 * n * (l + 1) * b
    if op == "add":
        return {"bytes": 3 * ct, "flops": ct / 8}
    if op == "mul_const":
        return {"bytes": ct + ct * l / (l + 1), "flops": 2 * b * n * (1.5 * log_n * (l + 1) + 3.0 * l)}
    if op == "mul":
        return {"bytes": 2 * ct + ct * l / (l + 1) + _key_bytes(case["preset"], l),
                "flops": 5.0 * b * n * (l + 1) + _switch_ops(case["preset"], l, b)}
    if op == "rotate":
        return {"bytes": 2 * ct + _key_bytes(case["preset"], l), "flops": _switch_ops(case["preset"], l, b)}
    if op == "rotate_hoisted":
        c = case["count"]
        dn, ext = -(-(l + 1) // a), l + 1 + k
        up = b * n * (1.5 * log_n * dn * ext + 2.0 * a * (dn * ext - l - 1))
        each = b * n * (1.5 * log_n * 2 * (l + 1 + k) + 4.0 * dn * ext + 4.0 * k * (l + 1))
        return {"bytes": ct * (1 + c) + c * _key_bytes(case["preset"], l), "flops": up + c * each}
    if op == "invsqrt":
        # products: baby steps and giant steps of the interpolant and three a Newton step, one level apart
        m = max(1, math.ceil(math.log2(case["degree"] + 1)))
        products = 2 * m - 1 + 3 * case["iters"]
        ops = sum(_switch_ops(case["preset"], max(1, l - 1 - i * (m + 2 * case["iters"]) // products), b)
                  for i in range(products))
        return {"bytes": ct + _key_bytes(case["preset"], l), "flops": ops}
    # a bootstrap: six grouped factors (about four giant steps and the shared ModUps of fifteen baby steps each), the
    # interpolant of degree 31 and four squarings; levels from the top of the chain down
    top = n_q - 1
    ops = sum(5 * _switch_ops(case["preset"], top - g, b) for g in range(3))
    ops += sum(2 * _switch_ops(case["preset"], top - 3 - i // 2, b) for i in range(14))
    ops += sum(5 * _switch_ops(case["preset"], top - 12 - g, b) for g in range(3))
    return {"bytes": ct + 16.0 * n * b * 12 + 30 * _key_bytes(case["preset"], top), "flops": ops}


def exact(case, seed):
    """Every output is an array of residues, whole numbers that must be equal: there is no rounded value to compare."""
    return None
