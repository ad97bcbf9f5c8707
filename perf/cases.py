"""Timed cases of the library's public calls.

Every case is work that a program built on this library does: one
homomorphic multiplication or rotation as a request arrives, batches of
them, the encrypted-query server, the client's encode and decode.  Parameter
sets are the library's own presets (workloads.PRESETS) and, for the ring
degrees between them, the headline chain on one shared prime list (as the
uneven mix of the benchmark uses it).

Contexts, keys, the resident table and its engine are kept per parameter
set, as a program keeps them; ciphertexts are uniform limbs (every residue
of a fresh or computed ciphertext is uniform mod its prime), drawn from the
seed.
"""
from __future__ import annotations

import hashlib
import math

import numpy as np
import torch

from paper_2503_22227_gb300 import api, encoding, roofline, serving
from paper_2503_22227_gb300 import workloads as W

ROTATIONS = 16
MIX_DEGREES = (13, 14, 15, 16)
MIX_LANES = 8
SERVE_BUDGET = 200 << 30

_contexts: dict = {}
_server: dict = {}


def listed() -> list:
    return [
        # the smallest call: one product at N = 2^12, as a gate of a circuit
        # that waits for it; latency, launches and host time
        {"name": "mul_n12_single", "kind": "mul", "params": "ckks_n12", "level": 3, "count": 1,
         "rescale": True},
        # one rotation of a rotate-and-add reduction, at an odd level
        {"name": "rotate_n13_single", "kind": "rotate", "params": "chain_n13", "level": 7,
         "count": 1},
        # rescale of a few results at once (after plaintext products)
        {"name": "rescale_n15_x3", "kind": "rescale", "params": "chain_n15", "level": 13,
         "count": 3},
        # a ragged product: a partly used second digit and halves of 3 and 2
        {"name": "mul_n15_x5", "kind": "mul", "params": "chain_n15", "level": 13, "count": 5,
         "rescale": True},
        # BGV and BFV batches of the paper's integer schemes
        {"name": "bgv_n14_x16", "kind": "mul", "params": "bgv_n14", "level": 8, "count": 16,
         "rescale": False},
        {"name": "bfv_n14_x16", "kind": "mul", "params": "bfv_n14", "level": 8, "count": 16,
         "rescale": False},
        # one full-size product: a request that is served alone
        {"name": "mul_n16_single", "kind": "mul", "params": "ckks_n16", "level": 24, "count": 1,
         "rescale": True},
        # the headline batch
        {"name": "mul_n16_x8", "kind": "mul", "params": "ckks_n16", "level": 24, "count": 8,
         "rescale": True},
        # the same batch rotated by 1 .. 16 (a convolution or a matrix product
        # reads all of them), the lifted digits shared
        {"name": "rotations_n16_x8", "kind": "hoist", "params": "ckks_n16", "level": 24,
         "count": 8, "rotations": 16},
        # many users' independent operations of four ring degrees and any
        # level, captured once and replayed
        {"name": "mix_256", "kind": "mix", "ops": 256},
        # eight encrypted range queries arriving together at the server, from
        # the uploads of their bounds to the encrypted answers in host memory
        {"name": "queries_8", "kind": "queries", "requests": 8},
        # the client's side: one message encoded, one answer decrypted and
        # decoded, both full size
        {"name": "client_n16", "kind": "client", "params": "ckks_n16", "level": 24},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng) -> dict:
    kind = rng.choice(["mul", "mul", "mul", "mul", "rotate", "rotate", "rescale", "hoist", "mix",
                       "queries", "client"])
    if kind == "mix":
        return {"kind": kind, "ops": _log_int(rng, 8, 256)}
    if kind == "queries":
        return {"kind": kind, "requests": rng.randint(1, 8)}
    params = rng.choice(["ckks_n12", "chain_n12", "chain_n13", "chain_n14", "chain_n15",
                         "ckks_n16", "ckks_n16_k8"])
    if kind in ("mul", "rotate") and rng.random() < 0.3:
        params = rng.choice(["bgv_n14", "bfv_n14"])
    pr = _preset(params)
    level = rng.randint(2, pr.L)
    if kind == "client":
        return {"kind": kind, "params": params, "level": level}
    case = {"kind": kind, "params": params, "level": level,
            "count": _log_int(rng, 1, 8 if pr.log_n == 16 else 16)}
    if kind == "mul":
        case["rescale"] = pr.scheme == W.CKKS and rng.random() < 0.7
    if kind == "hoist":
        case["count"] = min(case["count"], 8)
        case["rotations"] = rng.randint(2, ROTATIONS)
    return case


# ------------------------------------------------------------------ kept handles
def _preset(params: str) -> W.Preset:
    if params in W.PRESETS:
        return W.PRESETS[params]
    base = W.PRESETS["ckks_n16"]
    return W.Preset(params, W.CKKS, int(params[len("chain_n"):]), base.q_bits, base.p_bits,
                    base.dnum, log_n_max=16, log_scale=base.log_scale)


def _context(params: str):
    got = _contexts.get(params)
    if got is None:
        ctx = api.Context(_preset(params))
        keys = ctx.keygen(W.seed_for(f"cases-keys-{params}"))
        steps = [ctx.galois_elt(r) for r in range(1, ROTATIONS + 1)]
        for g in steps:
            keys.gen_galois(g)
        got = _contexts[params] = (ctx, keys, steps)
    return got


def _table():
    if not _server:
        table = serving.Table()
        _server["table"] = table
        _server["engine"] = serving.GpuEngine(table, lanes=8)
    return _server["table"], _server["engine"]


def _generator(seed: int):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(ctx, gen, count: int, level: int):
    ct = ctx.empty_ct(count, level)
    for i in range(level):
        ct[:, :, i].random_(0, int(ctx.q[i]), generator=gen)
    return ct


def _mix_entries(ops: int):
    """(log N, level, kind, rotation) of each entry, the same for every seed."""
    rng = W.rng_for(f"cases-mix-{ops}")
    kinds = (api.OP_MUL_RELIN, api.OP_ROTATE, api.OP_RESCALE)
    return [(int(rng.choice(MIX_DEGREES)), int(rng.integers(2, 25)), kinds[int(rng.integers(0, 3))],
             int(rng.integers(0, ROTATIONS))) for _ in range(ops)]


def _chain(log_n: int) -> str:
    return "ckks_n16" if log_n == 16 else f"chain_n{log_n}"


def _message(case: dict, seed: int, what: str) -> np.ndarray:
    rng = W.rng_for(f"cases-{what}-{seed}")
    return W.complex_slots(rng, _preset(case["params"]).n)


# ------------------------------------------------------------------ a case
def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    if kind == "mix":
        return _prepare_mix(case, seed)
    if kind == "queries":
        table, engine = _table()
        return {"kind": kind, "table": table, "engine": engine, "seed": f"cases-requests-{seed}",
                "requests": case["requests"]}
    ctx, keys, steps = _context(case["params"])
    st = {"kind": kind, "ctx": ctx, "keys": keys}
    level = case["level"]
    if kind == "client":
        pr = _preset(case["params"])
        st["scale"] = 2.0 ** pr.log_scale
        st["message"] = _message(case, seed, "encode")
        answer = encoding.encode(_message(case, seed, "decode"), ctx.n, st["scale"])
        ct = ctx.encrypt(keys, answer, hashlib.sha256(f"cases-{seed}".encode()).digest())
        st["answer"] = ctx.drop_level(ct, level) if level < ctx.L else ct
        st["level"] = level
        return st
    gen = _generator(seed)
    count = case["count"]
    st["a"] = _uniform(ctx, gen, count, level)
    if kind == "mul":
        st["b"] = _uniform(ctx, gen, count, level)
        st["rescale"] = case["rescale"]
        st["out"] = ctx.empty_ct(count, level - 1 if case["rescale"] else level)
    elif kind == "rotate":
        st["g"] = steps[int(torch.randint(0, ROTATIONS, (1,), generator=gen, device="cuda"))]
        st["out"] = ctx.empty_ct(count, level)
    elif kind == "rescale":
        st["out"] = ctx.empty_ct(count, level - 1)
    elif kind == "hoist":
        st["g"] = steps[: case["rotations"]]
        st["out"] = torch.empty((case["rotations"], count, 2, level, ctx.n), dtype=torch.int64,
                                device="cuda")
    return st


def _prepare_mix(case: dict, seed: int) -> dict:
    """The captured graph of a set of entries; all results lie in one buffer."""
    gen = _generator(seed)
    entries = _mix_entries(case["ops"])
    handles = {log_n: _context(_chain(log_n)) for log_n in MIX_DEGREES}
    sizes = [2 * (level - (op == api.OP_RESCALE)) << log_n for log_n, level, op, _ in entries]
    results = torch.empty(sum(sizes), dtype=torch.int64, device="cuda")
    ops, keep, at = [], [], 0
    for (log_n, level, op, r), size in zip(entries, sizes):
        ctx, keys, steps = handles[log_n]
        a = _uniform(ctx, gen, 1, level)
        b = _uniform(ctx, gen, 1, level) if op == api.OP_MUL_RELIN else None
        out = results[at:at + size].view(1, 2, -1, ctx.n)
        at += size
        ops.append(api.make_op(op, ctx, a, out, keys=keys, b=b, galois_elt=steps[r]))
        keep.append((a, b))
    return {"kind": "mix", "graph": api.Graph(ops, lanes=MIX_LANES), "inputs": keep,
            "out": results}


def run(st: dict):
    kind = st["kind"]
    if kind == "mix":
        st["graph"].launch()
        return st["out"]
    if kind == "queries":
        requests = serving.make_requests(st["table"], st["requests"], 0.0, st["seed"])
        serving.serve(requests, st["engine"], SERVE_BUDGET)
        return [r.result for r in requests]
    ctx, keys = st["ctx"], st["keys"]
    if kind == "mul":
        call = ctx.mul_relin_rescale if st["rescale"] else ctx.mul_relin
        return call(keys, st["a"], st["b"], out=st["out"])
    if kind == "rotate":
        return ctx.rotate(keys, st["a"], st["g"], out=st["out"])
    if kind == "rescale":
        return ctx.rescale(st["a"], out=st["out"])
    if kind == "hoist":
        return ctx.rotate_hoisted(keys, st["a"], st["g"], out=st["out"])
    return {"plain": ctx.encode_ckks(st["message"], st["scale"], st["level"]),
            "slots": ctx.decode_ckks(keys, st["answer"], st["scale"])}


def exact(case: dict, seed: int):
    """Ciphertexts are whole numbers and have one right value; the decoded
    slots are the message that was encrypted."""
    if case["kind"] != "client":
        return None
    return {"plain": None, "slots": _message(case, seed, "decode")}


# ------------------------------------------------------------------ work
def _alpha(pr: W.Preset) -> int:
    return -(-pr.L // pr.dnum)


def _key_bytes(pr: W.Preset, level: int) -> float:
    """One switching key's limbs that a call at `level` reads."""
    digits = len(roofline.digits(level, _alpha(pr)))
    return digits * 2 * (level + pr.K) * pr.n * 8


def _rescale_products(n: int, level: int) -> float:
    return level * n * int(math.log2(n)) + 4 * level * n


def _query_work() -> tuple:
    """(bytes, products) of one query's circuit."""
    table, _ = _table()
    pr = W.PRESETS["ckks_n16_k8"]
    nodes = table.circuit.nodes
    products = 0.0
    for i in table.circuit.live():
        nd = nodes[i]
        if nd.kind == "mul":
            products += roofline.ckks_mul_relin_rescale(pr.n, nd.level + 1, pr.K, _alpha(pr)).modmuls
        elif nd.kind == "rotate":
            products += roofline.ckks_rotate(pr.n, nd.level, pr.K, _alpha(pr)).modmuls
        elif nd.kind == "rescale":
            products += _rescale_products(pr.n, nd.level + 1)
        elif nd.kind == "mul_int":
            products += 2 * nd.level * pr.n
    out = nodes[table.circuit.outputs["sum"]]
    # two bounds and two columns read, the answer written
    return (4 * 2 * pr.L + 2 * out.level) * pr.n * 8.0, products


def work(case: dict) -> dict:
    """bytes: inputs read and outputs written once, each switching key once a
    pass.  flops: modular products (a 64-bit product and its reduction each)."""
    kind = case["kind"]
    if kind == "queries":
        nbytes, products = _query_work()
        return {"bytes": nbytes * case["requests"], "flops": products * case["requests"]}
    if kind == "mix":
        nbytes = products = 0.0
        used = {}
        for log_n, level, op, r in _mix_entries(case["ops"]):
            pr = _preset(_chain(log_n))
            limb = pr.n * 8.0
            if op == api.OP_RESCALE:
                nbytes += (2 * level + 2 * (level - 1)) * limb
                products += _rescale_products(pr.n, level)
                continue
            mul = op == api.OP_MUL_RELIN
            count = roofline.ckks_mul_relin if mul else roofline.ckks_rotate
            products += count(pr.n, level, pr.K, _alpha(pr)).modmuls
            nbytes += (6 if mul else 4) * level * limb
            key = (log_n, -1 if mul else r)
            used[key] = max(used.get(key, 0.0), _key_bytes(pr, level))
        return {"bytes": nbytes + sum(used.values()), "flops": products}
    pr = _preset(case["params"])
    n, level, alpha = pr.n, case["level"], _alpha(pr)
    limb = n * 8.0
    if kind == "client":
        # encode: slots read, one transform per limb, the plaintext written;
        # decode: the ciphertext and the secret read, the slots written
        fft = 2 * 5 * n * pr.log_n
        conv = level + level * level
        return {"bytes": (2 * limb + level * limb) + (3 * level + 1) * limb,
                "flops": 2 * level * n / 2 * pr.log_n + (conv + level) * n + fft}
    count = case["count"]
    if kind == "rescale":
        return {"bytes": count * (4 * level - 2) * limb, "flops": count * _rescale_products(n, level)}
    if kind == "hoist":
        rot = case["rotations"]
        per = roofline.ckks_rotate_hoisted(n, level, pr.K, alpha, rot).modmuls
        return {"bytes": count * (1 + rot) * 2 * level * limb + rot * _key_bytes(pr, level),
                "flops": count * rot * per}
    if kind == "rotate":
        per, limbs = roofline.ckks_rotate(n, level, pr.K, alpha).modmuls, 4 * level
    elif pr.scheme == W.BFV:
        bound = 2 * pr.t * n * 2 ** sum(pr.q_bits)
        nb = next(k for k in range(1, 33) if 2 ** (pr.b_bits * k) > bound)
        per, limbs = roofline.bfv_mul_relin(n, level, pr.K, alpha, nb).modmuls, 6 * level
    elif pr.scheme == W.BGV:
        per, limbs = roofline.bgv_mul_relin(n, level, pr.K, alpha).modmuls, 6 * level
    elif case["rescale"]:
        per = roofline.ckks_mul_relin_rescale(n, level, pr.K, alpha).modmuls
        limbs = 6 * level - 2
    else:
        per, limbs = roofline.ckks_mul_relin(n, level, pr.K, alpha).modmuls, 6 * level
    return {"bytes": count * limbs * limb + _key_bytes(pr, level), "flops": count * per}
