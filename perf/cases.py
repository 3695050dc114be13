"""Performance cases of the framework: the calls a program that serves or trains a KLA model makes, over the sizes it makes them at.

    listed()            the named cases
    draw(rng)           one more case of the ranges they stand for (rng: a random.Random)
    prepare(case, seed) what a program holds on the GPU before the call
    run(state)          one pass through the public entry points; returns every output whole
    work(case)          bytes and operations that one pass cannot do without
    tolerance(case)     how far another correct implementation of the same precision may be off

A case names an operation and its sizes:
    op      "forward" (kla_chunk_fwd), "backward" (kla_bwd), "dg_forward" (kla_dg_fwd: one decay per key dimension),
            "decode" (kla_decode_step, or kla_decode_steps where steps > 1), "dg_decode" (kla_dg_decode_step)
    B, T, H, d          sequences, tokens per sequence, heads, head dimension (d_k = d_v)
    n_seq, max_len      packed input instead of B, T: that many sequences, lengths drawn uniformly in [1, max_len] (lens_seed)
    dtype               "bf16" or "f32": q, k, v and the output
    state               whether the call starts from a given state (the continuation of a prompt)

Value distributions are those of the package's synthetic workloads: q, k ~ N(0, 1/d) with per-token log-normal norms (heavy
tails and near-zero keys in packed input), v ~ N(0, 1), eta = sigmoid(N(0, 1)), log alpha = -softplus(N(0, 1)) / 8.
"""
import math
import random

import torch

from paper_2605_08587_b200 import kla_bwd, kla_chunk_fwd, kla_decode_step, kla_decode_steps, kla_dg_decode_step, kla_dg_fwd

EPS = 1e-6


def listed():
    return [
        # decoding: one user; a full serving batch (the state fits the L2 cache); a batch whose states live in HBM, four tokens
        dict(name="decode B1", op="decode", B=1, H=8, d=128, steps=1, dtype="bf16"),
        dict(name="decode B64", op="decode", B=64, H=8, d=128, steps=1, dtype="bf16"),
        dict(name="decode B512 x4", op="decode", B=512, H=8, d=128, steps=4, dtype="bf16"),
        # prefill: one prompt of ragged length, and a context of 65 536 tokens that continues from a state
        dict(name="prefill 777", op="forward", B=1, T=777, H=8, d=128, dtype="bf16", state=False),
        dict(name="long context 65536", op="forward", B=1, T=65536, H=8, d=128, dtype="bf16", state=True),
        # the forward of a training step: fixed length, and packed sequences of all lengths
        dict(name="forward B8 T4096", op="forward", B=8, T=4096, H=8, d=128, dtype="bf16", state=False),
        dict(name="forward packed 32", op="forward", n_seq=32, max_len=8192, lens_seed=1004, H=16, d=64, dtype="bf16", state=False),
        # full precision: the small fp32 configuration
        dict(name="forward fp32 T256", op="forward", B=1, T=256, H=2, d=64, dtype="f32", state=False),
        # the backward of a training step: fixed length, and packed
        dict(name="backward B8 T4096", op="backward", B=8, T=4096, H=8, d=128, dtype="bf16", state=False),
        dict(name="backward packed 16", op="backward", n_seq=16, max_len=4096, lens_seed=1005, H=16, d=64, dtype="bf16", state=False),
        # diagonal gates: a layer's forward, and decoding
        dict(name="diagonal B8 T4096", op="dg_forward", B=8, T=4096, H=8, d=128, dtype="bf16", state=False),
        dict(name="diagonal decode B64", op="dg_decode", B=64, H=8, d=128, steps=1, dtype="bf16"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["forward", "forward", "forward", "backward", "backward", "dg_forward", "decode", "decode", "dg_decode"])
    d = rng.choice([64, 128, 128])
    H = rng.choice([2, 4, 8, 16])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    if op in ("decode", "dg_decode"):
        steps = rng.choice([1, 1, 4]) if op == "decode" and H >= 4 else 1   # (per-step gate rows stay 16-byte aligned)
        B = _log_int(rng, 1, 4096 // H)
        return dict(op=op, B=B, H=H, d=d, steps=steps, dtype=dtype)
    # tokens x heads x head dimension of the whole call: up to those of the largest listed case of the operation
    most = {"forward": 65536 * 8 * 128, "backward": 32768 * 8 * 128, "dg_forward": 32768 * 8 * 128}[op]
    if dtype == "f32":
        most //= 8
    tokens = most // (H * d)
    state = rng.random() < 0.5
    if op != "dg_forward" and rng.random() < 0.35:
        n_seq = _log_int(rng, 2, 64)
        max_len = _log_int(rng, 16, max(17, min(8192, tokens // n_seq)))
        return dict(op=op, n_seq=n_seq, max_len=max_len, lens_seed=rng.randrange(1 << 20), H=H, d=d, dtype=dtype, state=state)
    B = _log_int(rng, 1, 16)
    T = _log_int(rng, 16, tokens // B)
    return dict(op=op, B=B, T=T, H=H, d=d, dtype=dtype, state=state)


def _lengths(case):
    r = random.Random(case["lens_seed"])
    return [r.randint(1, case["max_len"]) for _ in range(case["n_seq"])]


def _shape(case):
    """(B, T, n_seq, lengths or None) of a sequence operation."""
    if "n_seq" in case:
        lens = _lengths(case)
        return 1, sum(lens), len(lens), lens
    return case["B"], case["T"], case["B"], None


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    op, H, d = case["op"], case["H"], case["d"]

    def randn(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    packed = "n_seq" in case
    if op in ("decode", "dg_decode"):
        lead, n_seq, lens = (case["steps"], case["B"], H), case["B"], None
    else:
        B, T, n_seq, lens = _shape(case)
        lead = (B, T, H)
    q = randn(*lead, d) / d ** 0.5 * torch.exp(0.5 * randn(*lead, 1))
    k = randn(*lead, d) / d ** 0.5 * torch.exp((1.5 if packed else 0.5) * randn(*lead, 1))
    if packed:   # stress eps: 1 % of the keys near zero, 0.1 % exactly zero
        u = torch.rand((*lead, 1), generator=g, device="cuda")
        k = torch.where(u < 0.01, k * 1e-4, k)
        k = torch.where(u < 0.001, torch.zeros_like(k), k)
    s = dict(op=op, q=q.to(dt), k=k.to(dt), v=randn(*lead, d).to(dt), eta=torch.sigmoid(randn(*lead)),
             log_alpha=-torch.nn.functional.softplus(randn(*lead, d) if op.startswith("dg_") else randn(*lead)) / 8.0)
    if op in ("decode", "dg_decode"):
        s["state"] = 0.02 * randn(n_seq, H, d, d)
        if case["steps"] == 1:
            for name in ("q", "k", "v", "eta", "log_alpha"):
                s[name] = s[name][0].contiguous()
        return s
    s["init"] = 0.02 * randn(n_seq, H, d, d) if case["state"] else None
    s["cu"] = s["host"] = None
    if packed:
        s["host"] = torch.tensor([0] + torch.tensor(lens).cumsum(0).tolist(), dtype=torch.int32)
        s["cu"] = s["host"].cuda()
    if op == "backward":
        s["d_out"] = randn(*lead, d).to(dt)
        s["d_final"] = randn(n_seq, H, d, d) if case["state"] else None
    return s


def run(s):
    a = (s["q"], s["k"], s["v"], s["log_alpha"], s["eta"], EPS)
    op = s["op"]
    if op == "forward":
        out, fin = kla_chunk_fwd(*a, init_state=s["init"], cu_seqlens=s["cu"], host_seqlens=s["host"])
        return {"out": out, "final_state": fin}
    if op == "backward":
        return kla_bwd(*a, s["d_out"], init_state=s["init"], d_final_state=s["d_final"], cu_seqlens=s["cu"], host_seqlens=s["host"])
    if op == "dg_forward":
        out, fin = kla_dg_fwd(*a, init_state=s["init"])
        return {"out": out, "final_state": fin}
    step = kla_dg_decode_step if op == "dg_decode" else kla_decode_step if s["q"].dim() == 3 else kla_decode_steps
    out = step(*a, s["state"])   # the state is updated in place
    return {"out": out, "state": s["state"]}


def work(case):
    H, d, io = case["H"], case["d"], 2 if case["dtype"] == "bf16" else 4
    gate = d if case["op"].startswith("dg_") else 1   # decays per token and head
    if case["op"] in ("decode", "dg_decode"):
        units = case["B"] * H
        # the state is carried through all steps of a call: read once, written once
        return {"bytes": units * (2 * d * d * 4 + case["steps"] * (4 * d * io + 4 * gate + 4)), "flops": case["steps"] * units * 8 * d * d}
    B, T, n_seq, _ = _shape(case)
    tokens, C = B * T * H, 64
    # Algorithm 1 (right) with its triangular factors counted as such
    flops = tokens * (4 * C * d + 6 * d * d + C * C / 3)
    state = n_seq * H * d * d * 4
    if case["op"] == "backward":
        # the states are recomputed (one forward), and every product of the forward has two in the derivative
        return {"bytes": tokens * (4 * d * io + 8 + 3 * d * 4 + 8) + state * (3 if case["state"] else 1), "flops": 3 * flops}
    return {"bytes": tokens * (4 * d * io + 4 * gate + 4) + state * (2 if case["state"] else 1), "flops": flops}


def tolerance(case):
    if case["op"] == "backward":   # gradients in fp32 from fp32 arithmetic; dependent sums over whole sequences
        return {"rel": 2e-5, "max": 1e-3}
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 5e-3, "max": 1e-2}   # outputs rounded to bf16
