"""Performance cases of the multi-key TFHE library: what a program of its users has it do.

Every case goes through the package's Python binding (Context, Server), with the library's default
product form unless the case names another one.  Parameter sets, key seeds and request streams are
the repository's own (workloads.py); bits, gate types, operands and encryption randomness come from
the case's seed.  Outputs are ciphertexts (32-bit torus words as int32), which every exact form
determines bit for bit, so there is no floating-point reference to compare them with.

The evaluation keys of a parameter set are generated once per process and the context that holds
them on the device is kept, as a server keeps the keys of its parties; a state holds its own
ciphertexts and outputs.
"""
import math

import numpy as np
import torch

from paper_2205_05825_gb300 import binding as B
from paper_2205_05825_gb300 import workloads as W

SETS = {"full": W.full_params, "toy": W.toy_params}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # One gate at a time: a client's interactive request, or a netlist level of one gate.
        dict(name="gate_1_k2", kind="gates", set="full", k=2, count=1, form="ntt2"),
        # A narrow netlist level or a small request, odd size.
        dict(name="gates_37_k2", kind="gates", set="full", k=2, count=37, form="ntt2"),
        # The benchmark batch: random gates of two parties.
        dict(name="gates_4096_k2", kind="gates", set="full", k=2, count=4096, form="ntt2"),
        # A few gates of four parties: a narrow level of the serving workload.
        dict(name="gates_5_k4", kind="gates", set="full", k=4, count=5, form="ntt2"),
        # The 4-party half of the metric, a ragged batch.
        dict(name="gates_1001_k4", kind="gates", set="full", k=4, count=1001, form="ntt2"),
        # Eight parties, the largest count the library takes (the precision sweep's last row).
        dict(name="gates_96_k8", kind="gates", set="full", k=8, count=96, form="ntt2"),
        # The toy configuration: all gate types on all input pairs, then four NOTs.
        dict(name="toy_24_not_4", kind="gates", set="toy", k=2, count=24, nots=4, form="ntt2"),
        # The exact tensor-core form on a batch below one full wave.
        dict(name="gates_300_k2_tc", kind="gates", set="full", k=2, count=300, form="tc"),
        # An operator over several operand pairs: every level is a middle-sized batch.
        dict(name="add_8bit_16_pairs", kind="operator", op="add", k=2, bits=8, pairs=16, style="array"),
        # One multiplication as fast as it goes: narrow levels of a shallow netlist.
        dict(name="mul_8bit_1_pair", kind="operator", op="mul", k=2, bits=8, pairs=1, style="shallow"),
        # Continuous batching of mixed requests of four parties until all are done.
        dict(name="serve_6_requests_k4", kind="serve", k=4, bits=8, requests=6, style="shallow"),
        # The per-party key switch by itself, the second stage of every gate, at the benchmark batch.
        dict(name="keyswitch_4096_k2", kind="keyswitch", set="full", k=2, count=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: gate batches of 2 to 8 parties (the largest no dearer than 4096 gates of two),
    operators of 2 to 8 bits, requests, key switches, the toy set; sizes spread over their logarithm."""
    kind = rng.choice(["gates"] * 6 + ["operator"] * 2 + ["serve", "keyswitch", "toy"])
    if kind == "gates":
        k = rng.choice([2, 2, 2, 3, 4, 4, 5, 8])
        most = 4096 * 8 // (k * (k + 2))
        form = "tc" if k <= 4 and rng.random() < 0.1 else "ntt2"
        return dict(kind="gates", set="full", k=k, count=_log_int(rng, 1, most // (3 if form == "tc" else 1)), form=form)
    if kind == "toy":
        return dict(kind="gates", set="toy", k=rng.choice([2, 3]), count=_log_int(rng, 2, 2000), nots=_log_int(rng, 1, 500),
                    form="ntt2")
    if kind == "keyswitch":
        return dict(kind="keyswitch", set="full", k=rng.choice([2, 4]), count=_log_int(rng, 1, 4096))
    if kind == "serve":
        return dict(kind="serve", k=4, bits=rng.choice([6, 7, 8]), requests=rng.randint(2, 6), style="shallow")
    op = rng.choice(["add", "sub", "mul"])
    bits = rng.randint(2, 8) if op != "mul" else rng.randint(2, 6)
    return dict(kind="operator", op=op, k=rng.choice([2, 4]), bits=bits, pairs=_log_int(rng, 1, 24),
                style=rng.choice(["array", "shallow"]))


# ------------------------------------------------------------------ states
_contexts = {}


def _params(case):
    return SETS[case.get("set", "full")](case["k"])


def _context(case):
    """The kept context of a parameter set, product form and netlist family, its keys on the device."""
    key = (case.get("set", "full"), case["k"], case.get("form", "ntt2"), case.get("style", "array"))
    if key not in _contexts:
        ctx = B.Context(_params(case), W.CRS_SEED, device=0)
        held = next((c for (s, k, _, _), c in _contexts.items() if (s, k) == key[:2]), None)
        if held is None:
            for party, seed in enumerate(W.party_seeds(case["k"])):
                ctx.keygen(party, seed)
        else:
            ctx.load_keys(held.save_keys())
        ctx.set_form(key[2])
        ctx.set_circuit_style(key[3])
        ct = _device(ctx.encrypt(0, np.array([1], np.uint8), 1))
        ctx.gate("AND", ct, ct, torch.empty_like(ct))  # lays the keys out on the device
        ctx.sync()
        _contexts[key] = ctx
    return _contexts[key]


def _device(words):
    return torch.from_numpy(np.ascontiguousarray(words).view(np.int32)).cuda()


def _encrypt_seed(seed, stream):
    return W.INPUT_SEED_BASE + 16 * (seed + 1) + stream


def _encrypt_pair(ctx, k, b1, b2, seed):
    """Operands as the benchmark has them: two parties' own bits, or every party's block in use."""
    if k == 2:
        return ctx.encrypt(0, b1, _encrypt_seed(seed, 0)), ctx.encrypt(1, b2, _encrypt_seed(seed, 1))
    return ctx.encrypt_joint(b1, _encrypt_seed(seed, 0)), ctx.encrypt_joint(b2, _encrypt_seed(seed, 1))


def _operands(ctx, bits, values, party, seed):
    planes = W.int_to_bits(values, bits)
    return _device(ctx.encrypt(party, planes.reshape(-1), seed).reshape(len(values), bits, ctx.W))


def _empty(*shape):
    return torch.zeros(shape, dtype=torch.int32, device="cuda")


def _requests(case, seed):
    """Operator names and operands of the served requests: add, sub and mul in turn."""
    r = np.random.default_rng(seed)
    half = 1 << (case["bits"] - 1)
    return [(("mul", "add", "sub")[i % 3], r.integers(-half, half, 1), r.integers(-half, half, 1))
            for i in range(case["requests"])]


def prepare(case, seed):
    ctx = _context(case)
    r = np.random.default_rng(seed)
    state = dict(case=case, ctx=ctx)
    if case["kind"] == "gates":
        n = case["count"]
        if case.get("set") == "toy" and n == 24:
            types, b1, b2 = W.truth_table_inputs()
        else:
            types, b1, b2 = (r.integers(0, hi, n) for hi in (6, 2, 2))
        a, b = _encrypt_pair(ctx, case["k"], b1.astype(np.uint8), b2.astype(np.uint8), seed)
        state.update(types=torch.from_numpy(types.astype(np.uint8)).cuda(), a=_device(a), b=_device(b), out=_empty(n, ctx.W))
        if case.get("nots"):
            bits = r.integers(0, 2, case["nots"]).astype(np.uint8)
            state.update(c=_device(ctx.encrypt(0, bits, _encrypt_seed(seed, 2))), nout=_empty(case["nots"], ctx.W))
    elif case["kind"] == "keyswitch":
        # Extracted samples of a blind rotation: every word of the torus occurs.
        gen = torch.Generator(device="cuda").manual_seed(seed)
        ext = torch.randint(-(1 << 31), 1 << 31, (case["count"], ctx.E), generator=gen, device="cuda", dtype=torch.int64)
        state.update(ext=ext.to(torch.int32), out=_empty(case["count"], ctx.W))
    elif case["kind"] == "operator":
        half, bits, pairs = 1 << (case["bits"] - 1), case["bits"], case["pairs"]
        state.update(a=_operands(ctx, bits, r.integers(-half, half, pairs), 0, _encrypt_seed(seed, 0)),
                     b=_operands(ctx, bits, r.integers(-half, half, pairs), 1, _encrypt_seed(seed, 1)),
                     out=_empty(pairs, bits * (2 if case["op"] == "mul" else 1), ctx.W))
    else:
        bits = case["bits"]
        state["server"] = B.Server(ctx, wave_gates=4096, pool_rows=1 << 14)
        state["requests"] = [
            (op, _operands(ctx, bits, x, i % 4, _encrypt_seed(seed, 2 * i)),
             _operands(ctx, bits, y, (i + 1) % 4, _encrypt_seed(seed, 2 * i + 1)),
             _empty(1, bits * (2 if op == "mul" else 1), ctx.W)) for i, (op, x, y) in enumerate(_requests(case, seed))]
    return state


# ------------------------------------------------------------------ one pass
def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "gates":
        ctx.gates(state["types"], state["a"], state["b"], state["out"])
        if "c" in state:
            ctx.mk_not(state["c"], state["nout"])
            return {"gates": state["out"], "not": state["nout"]}
        return state["out"]
    if case["kind"] == "keyswitch":
        return ctx.stage_keyswitch(state["ext"], state["out"])
    if case["kind"] == "operator":
        call = {"add": ctx.add_kbit, "sub": ctx.sub_kbit, "mul": ctx.mul_kbit}[case["op"]]
        return call(case["bits"], state["a"], state["b"], state["out"])
    server = state["server"]
    for op, a, b, out in state["requests"]:
        server.submit(op, case["bits"], a, b, out)
    left = len(state["requests"])
    while left:
        left -= server.step()
    return [out for _, _, _, out in state["requests"]]


# ------------------------------------------------------------------ what a pass cannot do without
def _gate_ops(P, parties):
    """Ring operations of one bootstrapped gate whose input has `parties` nonzero party blocks: the
    (k+2)(d+1) transforms and (2k+4)d pointwise products of each CMux step, and the key switch's row
    additions (three digits in four are nonzero)."""
    n, N, k, d, t = P["n"], P["N"], P["k"], P["d"], P["t"]
    step = 3 * (k + 2) * (d + 1) * (N // 2) * int(math.log2(N)) + 2 * (2 * k + 4) * d * N
    return parties * (n * step + N * t * 3 // 4 * (n + 1))


def _key_bytes(P, parties):
    """Bootstrapping, public and key-switching keys that such gates read, as torus words."""
    n, N, k, d, t = P["n"], P["N"], P["k"], P["d"], P["t"]
    return 4 * (parties * (n * 3 * d * N + N * t * ((1 << P["ks_bit"]) - 1) * (n + 1)) + (k + 1) * d * N)


def work(case):
    P = _params(case)
    row = 4 * (P["k"] * P["n"] + 1)
    if case["kind"] == "gates":
        nots = case.get("nots", 0)
        return {"bytes": case["count"] * (3 * row + 1) + 2 * nots * row + _key_bytes(P, P["k"]),
                "flops": case["count"] * _gate_ops(P, P["k"]) + nots * row // 4}
    if case["kind"] == "keyswitch":
        rows = P["N"] * P["t"] * ((1 << P["ks_bit"]) - 1) * (P["n"] + 1)
        return {"bytes": case["count"] * (4 * (P["k"] * P["N"] + 1) + row) + 4 * P["k"] * rows,
                "flops": case["count"] * P["k"] * P["N"] * P["t"] * 3 // 4 * (P["n"] + 1)}
    # Operators and requests: the operands come from two parties, whose blocks alone are nonzero.
    if case["kind"] == "operator":
        jobs = [(case["op"], case["pairs"])]
    else:
        jobs = [(op, 1) for op, _, _ in _requests(case, 0)]
    gates = rows = 0
    for op, pairs in jobs:
        net = B.circuit_netlist(op, case["bits"], case["style"])
        gates += pairs * len(net["gates"])
        rows += pairs * case["bits"] * (4 if op == "mul" else 3)
    return {"bytes": rows * row + _key_bytes(P, 2 if case["kind"] == "operator" else P["k"]), "flops": gates * _gate_ops(P, 2)}


def exact(case, seed):
    """Ciphertext words are whole numbers, compared word for word: there is no rounding to measure."""
    return None
