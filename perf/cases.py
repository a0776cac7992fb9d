"""The calls that users of the library make, as cases for timing: training steps (forward and
backward) of one attention layer, inference forwards and prefill, segments of long sequences,
blocks of new tokens and single decode steps.

``listed()`` names the fixed cases, ``draw(rng)`` gives another one of the same ranges,
``prepare(case, seed)`` makes the tensors a program holds before the call, ``run(state)`` is one
pass through the public binding, ``work(case)`` the bytes and operations the method cannot do
without, ``tolerance(case)`` how far another correct implementation may be off.

Sizes are those of the workload recipes in ``paper_2409_18747_b200/synth.py`` (BERT-base and
GPT-2-small layers, the long causal step, the long-context sweep, the decode batch), of
``bench.py`` (packed batches, token blocks) and ragged relatives of them.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2409_18747_b200 as cott

# A case, whichever the operation:
#   op       train   cott.fwd, then cott.bwd on the same tensors
#            forward cott.fwd; with "state" it also returns the state that decoding continues from
#            segment cott.fwd_stateful on a state from earlier tokens; with "grad" cott.bwd_stateful after it
#            packed  cott.fwd_varlen on sequences of lo..hi tokens, then cott.bwd_varlen
#            decode  cott.decode_step: one token per sequence on a state, updated in place
#   B, H     sequences, heads;  N: tokens per sequence;  dk, dv: head sizes of keys and values
#   dtype    bf16 | f32;  causal;  zero: share of key rows that are exactly zero (padding)
#   layout   dense [B,H,N,d] | bnhd ([B,N,H,d] in memory) | fused (slices of a [B,N,3,H,d] projection output)
#   keep     train: both workspaces belong to the program, and the backward is given the forward's
_DEFAULTS = dict(op="train", B=1, H=1, N=1, dk=64, dv=64, dtype="bf16", causal=True, layout="dense",
                 zero=0.0, keep=False, state=False, grad=False, lo=1, hi=1)
_LONG = 8192.0   # scaling base of decode steps and segments: the length of the whole sequence


def _case(**kw):
    return {**_DEFAULTS, **kw}


def listed():
    return [
        # one user's token through one layer of a GPT-2-small: nothing but latency
        _case(name="decode-single", op="decode", B=1, H=12),
        # a serving batch's token: 67 MB of fp32 state read and written
        _case(name="decode-batch", op="decode", B=64, H=16, dk=128, dv=128),
        # sixteen new tokens per sequence on the same states (speculative decoding, short prompts)
        _case(name="block-16", op="segment", B=64, H=16, N=16, dk=128, dv=128, state=True),
        # a batch of sentences through a BERT-base layer at inference: ragged and shorter than a tile
        _case(name="forward-sentences", op="forward", B=64, H=12, N=77, causal=False),
        # a small single-precision layer, as one trains to check a model
        _case(name="train-fp32", op="train", B=2, H=8, N=509, dtype="f32"),
        # BERT-base pre-training step: q, k, v are slices of the projection's output
        _case(name="train-bert", op="train", B=32, H=12, N=512, causal=False, layout="fused"),
        # GPT-2-small training step, some keys padded with zeros
        _case(name="train-gpt2", op="train", B=8, H=12, N=1024, layout="fused", zero=0.05),
        # the long causal training step the headline figure is quoted on
        _case(name="train-long", op="train", B=4, H=16, N=4096, keep=True),
        # heads of 128, a sequence length that no tile divides
        _case(name="train-d128", op="train", B=3, H=16, N=2999, dk=128, dv=128, layout="bnhd"),
        # training through chunked prefill: one segment in the middle of long sequences
        _case(name="train-segment", op="segment", B=4, H=16, N=2048, state=True, grad=True),
        # sequences of 512 to 2048 tokens packed without padding
        _case(name="train-packed", op="packed", B=64, H=16, dk=128, dv=128, lo=512, hi=2048, grad=True),
        # prefill of a very long context, the state kept for decoding
        _case(name="prefill-long", op="forward", B=1, H=16, N=131072, dk=128, dv=128, state=True),
    ]


def _log(rng, lo, hi):
    """A whole number from lo to hi, spread evenly over its logarithm; about half of them odd."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        op = rng.choice(("train", "train", "train", "forward", "forward", "segment", "packed", "decode"))
        d = rng.choice((64, 64, 64, 128, 128, 128, 32, 96))
        c = _case(op=op, H=rng.choice((1, 4, 8, 12, 12, 16, 16, 32)), dk=d, dv=d)
        if op == "decode":
            c.update(B=_log(rng, 1, 96))
        elif op == "packed":
            hi = _log(rng, 64, 4096)
            c.update(B=_log(rng, 2, 128), hi=hi, lo=max(1, hi // rng.choice((2, 4, 16))), causal=rng.random() < 0.6,
                     grad=rng.random() < 0.6)
        elif op == "segment":
            grad = rng.random() < 0.3
            c.update(B=_log(rng, 1, 64), N=_log(rng, 128 if grad else 2, 4096), state=True, grad=grad)
        else:
            causal = rng.random() < 0.6
            c.update(B=_log(rng, 1, 64), N=_log(rng, 16, 131072 if op == "forward" and causal else 8192), causal=causal,
                     layout=rng.choice(("dense", "bnhd", "fused")), zero=rng.choice((0.0, 0.0, 0.05)),
                     keep=op == "train" and rng.random() < 0.3, state=op == "forward" and causal and rng.random() < 0.5)
            if rng.random() < 0.15 and d in (32, 64, 128):
                c.update(dtype="f32", zero=0.0)
            elif rng.random() < 0.1 and c["layout"] == "dense":   # key and value sizes of their own
                c.update(dk=64, dv=128, keep=False)
        w = work(c)
        # no dearer than the largest listed ones; single precision runs on the plain multiply-add units
        if w["bytes"] <= 2.0e9 and (c["dtype"] == "bf16" or w["flops"] <= 2.0e9):
            return c


def _lengths(case):
    r = random.Random(case["B"] * 65537 + case["hi"])
    return [r.randint(case["lo"], case["hi"]) for _ in range(case["B"])]


def _rows(case):
    """Tokens of the whole batch."""
    return sum(_lengths(case)) if case["op"] == "packed" else case["B"] * (1 if case["op"] == "decode" else case["N"])


def work(case):
    dk, dv, size = case["dk"], case["dv"], 2 if case["dtype"] == "bf16" else 4
    units = _rows(case) * case["H"]                      # rows of one head
    state = case["B"] * case["H"] * dk * dv * 4
    fwd, bwd = units * 2 * (dk + dv) * size, units * (4 * dk + 3 * dv) * size
    # the state form of the method, or the score form where the sequence is shorter than the head
    n = max(_lengths(case)) if case["op"] == "packed" else case["N"]
    per = min(4 * dk * dv, 2 * n * (dk + dv)) if case["op"] in ("train", "forward", "packed") else 4 * dk * dv
    nbytes, flops = fwd, units * per
    if case["op"] == "train" or case["grad"]:
        nbytes, flops = nbytes + bwd, flops + units * per * 5 // 2
    if case["op"] in ("decode", "segment"):
        nbytes += 2 * state + (3 * state if case["grad"] else 0)
    elif case["state"]:
        nbytes += state
    return {"bytes": nbytes, "flops": flops}


def _heads(shape, mean, gen, dtype, head_dim):
    """Normal rows around a direction of the head's own, as the activations of a layer are."""
    x = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    view = [1] * len(shape)
    view[head_dim], view[-1] = shape[head_dim], shape[-1]
    return x.add_(mean.view(view)).to(dtype)


def prepare(case, seed):
    B, H, N, dk, dv = (case[x] for x in ("B", "H", "N", "dk", "dv"))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    rand = lambda *shape: torch.randn(shape, generator=gen, device="cuda")
    m, key_mean, value_mean = rand(H), 0.5 * rand(H, dk), 0.5 * rand(H, dv)
    s = {"case": case, "m": m}
    op = case["op"]
    if op == "packed":
        lens = _lengths(case)
        T, edges = sum(lens), [0]
        for n in lens:
            edges.append(edges[-1] + n)
        s["cu"], s["longest"] = torch.tensor(edges, dtype=torch.int32, device="cuda"), max(lens)
        s["q"], s["k"] = (_heads((T, H, dk), key_mean, gen, dtype, 1) for _ in range(2))
        s["v"] = _heads((T, H, dv), value_mean, gen, dtype, 1)
        if case["grad"]:
            s["d_o"] = _heads((T, H, dv), value_mean, gen, dtype, 1)
        return s
    if op == "decode":
        s["q"], s["k"] = (_heads((B, H, dk), key_mean, gen, dtype, 1) for _ in range(2))
        s["v"] = _heads((B, H, dv), value_mean, gen, dtype, 1)
    elif case["layout"] == "dense":
        s["q"], s["k"] = (_heads((B, H, N, dk), key_mean, gen, dtype, 1) for _ in range(2))
        s["v"] = _heads((B, H, N, dv), value_mean, gen, dtype, 1)
        if op == "train" or case["grad"]:
            s["d_o"] = _heads((B, H, N, dv), value_mean, gen, dtype, 1)
    else:
        q, k, v = (_heads((B, N, H, dk), x, gen, dtype, 2) for x in (key_mean, key_mean, value_mean))
        if case["layout"] == "fused":
            s["qkv"] = torch.stack((q, k, v), dim=2)
            q, k, v = s["qkv"].unbind(2)
        s["q"], s["k"], s["v"] = (x.permute(0, 2, 1, 3) for x in (q, k, v))
        if op == "train":
            s["d_o"] = _heads((B, N, H, dv), value_mean, gen, dtype, 2).permute(0, 2, 1, 3)
    if case["zero"] > 0:
        s["k"].masked_fill_(torch.rand((B, H, N, 1), generator=gen, device="cuda") < case["zero"], 0.0)
    if op in ("decode", "segment"):
        # what about a thousand earlier tokens leave behind: sums of entries of unit keys times c v
        scale = math.sqrt(1000.0 / dk) * _LONG ** -torch.sigmoid(m)
        s["state"] = rand(B, H, dk, dv) * scale.view(1, H, 1, 1)
        if case["grad"]:
            s["d_state"] = rand(B, H, dk, dv) * math.sqrt(1000.0 / dk)
    if case["keep"]:
        dt = cott.cott.BF16 if case["dtype"] == "bf16" else cott.cott.F32
        s["ws"], s["ws_bwd"] = (torch.empty(cott.workspace_bytes(x, dt, B, H, N, dk, case["causal"]) or 256, dtype=torch.uint8,
                                            device="cuda") for x in (cott.cott.OP_FWD, cott.cott.OP_BWD))
    return s


def _like(x):
    """An output tensor in the memory layout of the layer's activations, [B,N,H,d]."""
    B, H, N, d = x.shape
    return torch.empty((B, N, H, d), dtype=x.dtype, device=x.device).permute(0, 2, 1, 3)


def run(s):
    case, q, k, v, m = s["case"], s["q"], s["k"], s["v"], s["m"]
    op, causal = case["op"], case["causal"]
    if op == "decode":
        return {"o": cott.decode_step(q, k, v, s["state"], m, _LONG), "state": s["state"]}
    if op == "packed":
        o = cott.fwd_varlen(q, k, v, m, s["cu"], s["longest"], causal=causal)
        if not case["grad"]:
            return {"o": o}
        return {"o": o, "grads": cott.bwd_varlen(q, k, v, s["d_o"], m, s["cu"], s["longest"], causal=causal)}
    if op == "segment":
        o, state = cott.fwd_stateful(q, k, v, m, _LONG, state_in=s["state"])
        if not case["grad"]:
            return {"o": o, "state": state}
        return {"o": o, "state": state,
                "grads": cott.bwd_stateful(q, k, v, s["d_o"], m, _LONG, state_in=s["state"], d_state_out=s["d_state"])}
    dense = case["layout"] == "dense"
    out = None if dense else _like(v)
    if op == "forward":
        return {"o": cott.fwd(q, k, v, m, causal=causal, return_state=case["state"], out=out)}
    o = cott.fwd(q, k, v, m, causal=causal, out=out, workspace=s.get("ws"))
    grads = None
    if case["layout"] == "fused":      # the gradient of the projection's output, written in place
        d_qkv = torch.empty_like(s["qkv"])
        grads = tuple(x.permute(0, 2, 1, 3) for x in d_qkv.unbind(2))
    elif not dense:
        grads = tuple(_like(x) for x in (q, k, v))
    return {"o": o, "grads": cott.bwd(q, k, v, s["d_o"], m, causal=causal, out=grads, workspace=s.get("ws_bwd"),
                                      fwd_workspace=s.get("ws"))}


def tolerance(case):
    # against the quadratic definition in 64 bits: bf16 outputs and gradients are off by 1.7e-3 to 2.4e-3 (the rounding
    # of the outputs and of the tensor-core operands), single precision by 1e-7 to 2e-7 at up to 500 tokens; four times
    # that, and room for the longer sums of single-precision sequences of thousands of tokens
    return {"rel": 1e-2} if case["dtype"] == "bf16" else {"rel": 2e-6}
