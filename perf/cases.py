"""The work this library is used for, as measured cases.

A pass is what one attention layer of a training or evaluation step asks of the library: forward (and
backward) over one packed batch of sequences of widely varying length, through the public calls of
`binding` and, where a plan splits the batch, of `stream`.  The length mixes are those of `inputs`
(text, video clips, one extreme sequence, the two axes of a 2-D model) and a plain log-uniform one; head
counts and head dimensions are those of the benchmark and the tests (64, 72, 128; 72 is a 2-D model's).
"""
from __future__ import annotations

import math
import random

import torch

from paper_2608_07524_b200 import binding as B
from paper_2608_07524_b200 import inputs
from paper_2608_07524_b200.stream import StreamRunner, plan_batch


def _log_uniform(lo, hi, n, seed):
    g = inputs.SplitMix64(seed)
    return [int(math.floor(lo * (hi / lo) ** g.uniform())) for _ in range(n)]


def _lengths(case):
    mix, n, seed = case["mix"], case["n"], case["mix_seed"]
    if mix == "log":
        return _log_uniform(case["lo"], case["hi"], n, seed)
    if mix == "tiny":
        return list(inputs.config(1).lengths)
    if mix == "video":
        return inputs.video_lengths(n, seed)
    if mix == "long":
        return inputs.extreme_lengths(n, seed, case["long"])
    if mix in ("spatial", "temporal"):
        return inputs.short2d_lengths(mix, n, seed)
    raise ValueError(f"unknown mix {mix!r}")


def listed():
    return [
        # The smallest call of the tests: four sequences of 17-255 tokens, 2 heads of 64 (a small model, or the last
        # few sequences of an epoch).  Launches and the host side count.
        {"name": "tiny_train", "call": "train", "mix": "tiny", "n": 4, "mix_seed": 0, "heads": 2, "head_dim": 64, "causal": True},
        # One forward of a caller that must not allocate: a few short requests, outputs and scratch supplied beforehand.
        {"name": "noalloc_forward", "call": "noalloc", "mix": "log", "lo": 24, "hi": 1500, "n": 5, "mix_seed": 7, "heads": 8,
         "head_dim": 128, "causal": True},
        # Many short texts: 512 sequences of 16-200 tokens, most of which share a 128-row tile with their neighbours.
        {"name": "short_text_train", "call": "train", "mix": "log", "lo": 16, "hi": 200, "n": 512, "mix_seed": 9, "heads": 16,
         "head_dim": 64, "causal": True},
        # The benchmark's text batch: 32 sequences, log-uniform in [512, 8192), causal.
        {"name": "text_train", "call": "train", "mix": "log", "lo": 512, "hi": 8192, "n": 32, "mix_seed": 2, "heads": 16,
         "head_dim": 128, "causal": True},
        # Evaluation on the same kind of text: forward only, fewer sequences.
        {"name": "text_forward", "call": "forward", "mix": "log", "lo": 300, "hi": 6000, "n": 12, "mix_seed": 12, "heads": 16,
         "head_dim": 128, "causal": True},
        # The benchmark's default, the video batch: 24 clips of 256-46800 tokens, bidirectional.
        {"name": "video_train", "call": "train", "mix": "video", "n": 24, "mix_seed": 3, "heads": 16, "head_dim": 128, "causal": False},
        # The benchmark's extreme imbalance: one sequence of 131072 tokens beside 64 of 128-2048, causal.
        {"name": "extreme_train", "call": "train", "mix": "long", "long": 131072, "n": 64, "mix_seed": 4, "heads": 8,
         "head_dim": 128, "causal": True},
        # A 2-D model's spatial axis: every latent frame of the video batch attends over its 256-3600 tokens.
        {"name": "spatial_train", "call": "train", "mix": "spatial", "n": 24, "mix_seed": 3, "heads": 16, "head_dim": 128, "causal": False},
        # The same axis at that model's own width, 16 heads of 72.
        {"name": "spatial_d72_train", "call": "train", "mix": "spatial", "n": 24, "mix_seed": 3, "heads": 16, "head_dim": 72,
         "causal": False},
        # Its temporal axis: every spatial position attends over its 1-13 frames (20384 sequences).
        {"name": "temporal_train", "call": "train", "mix": "temporal", "n": 24, "mix_seed": 3, "heads": 16, "head_dim": 128,
         "causal": False},
        # One rank's share of sequence parallelism: 4 heads inside tensors of 16, strided entry points.
        {"name": "head_group_train", "call": "head_group", "mix": "video", "n": 10, "mix_seed": 6, "heads": 16, "group": 4,
         "head_dim": 128, "causal": False},
        # A batch of the stream whose plan (28 layers, 16 GB) splits it into micro-batches and recomputes in some: plan, gather,
        # forward, recompute, backward, scatter.
        {"name": "stream_split", "call": "stream", "mix": "video", "n": 12, "mix_seed": 16, "heads": 16, "head_dim": 128,
         "causal": False, "layers": 28, "budget_gb": 16.0},
    ]


def draw(rng: random.Random):
    def log_int(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    kind = rng.choice(["small", "short", "text", "text", "video", "long", "spatial", "temporal", "head_group", "stream"])
    c = {"call": "train", "mix_seed": rng.randrange(1 << 20), "heads": rng.choice([4, 8, 12, 16]),
         "head_dim": rng.choice([64, 72, 128, 128]), "causal": rng.random() < 0.5}
    if kind == "small":
        lo = log_int(1, 60)
        c.update(mix="log", lo=lo, hi=lo * 4 + rng.randrange(600), n=rng.randint(1, 9), heads=rng.choice([2, 3, 8]),
                 call=rng.choice(["train", "noalloc", "forward"]))
    elif kind == "short":
        c.update(mix="log", lo=log_int(2, 40), hi=rng.randint(60, 400), n=log_int(64, 2000))
    elif kind == "text":
        lo = log_int(200, 1000)
        c.update(mix="log", lo=lo, hi=lo * rng.randint(2, 16), n=rng.randint(4, 32), causal=True, call=rng.choice(["train", "forward"]))
    elif kind == "video":
        c.update(mix="video", n=rng.randint(3, 20), causal=False)
    elif kind == "long":
        c.update(mix="long", long=log_int(8192, 98304), n=rng.randint(0, 64), heads=rng.choice([4, 8]), causal=True)
    elif kind in ("spatial", "temporal"):
        c.update(mix=kind, n=rng.randint(4, 24), causal=False)
    elif kind == "head_group":
        c.update(call="head_group", mix=rng.choice(["video", "spatial"]), n=rng.randint(4, 16), heads=16, group=rng.choice([2, 4, 8]),
                 causal=False)
    else:
        c.update(call="stream", mix="video", n=rng.randint(6, 12), head_dim=128, heads=16, causal=False, layers=28,
                 budget_gb=rng.choice([16.0, 20.0, 40.0]))
    return c


class _State:
    pass


def prepare(case, seed):
    lengths, H, d = _lengths(case), case["heads"], case["head_dim"]
    T = sum(lengths)
    s = _State()
    s.case, s.call, s.lengths, s.T, s.causal = case, case["call"], lengths, T, case["causal"]
    s.max_seqlen = max(lengths)
    if s.call == "stream":
        # the runner owns the batch's and the micro-batches' buffers; its values come from the seed
        s.runner = StreamRunner(T, len(lengths), H, d, s.causal, "cuda", value_seed=4 * seed)
        return s
    s.q, s.k, s.v, s.g = inputs.make_qkvg_device(T, H, d, 4 * seed, "cuda")
    cu = [0]
    for length in lengths:
        cu.append(cu[-1] + length)
    s.cu = torch.tensor(cu, dtype=torch.int32, device="cuda")
    if s.call == "noalloc":
        s.o = torch.empty_like(s.q)
        s.lse = torch.empty((H, T), dtype=torch.float32, device="cuda")
    elif s.call == "head_group":
        h = slice(case["group"], 2 * case["group"])          # the second rank's heads
        s.q, s.k, s.v, s.g = (x[:, h, :] for x in (s.q, s.k, s.v, s.g))
        s.o, s.dq, s.dk, s.dv = (torch.zeros((T, H, d), dtype=torch.bfloat16, device="cuda")[:, h, :] for _ in range(4))
        s.ws = B.alloc_workspace(T, len(lengths), case["group"], d, True, "cuda")
    else:
        s.ws = B.alloc_workspace(T, len(lengths), H, d, s.call == "train", "cuda")
    return s


def run(s):
    c = s.case
    if s.call == "stream":
        plan = plan_batch(s.lengths, int(c["budget_gb"] * 10 ** 9), c["heads"], c["head_dim"], n_layers=c["layers"])
        s.runner.run_batch(plan, s.T)
        r = s.runner
        return {"o": r.o, "lse": r.lse, "dq": r.dq, "dk": r.dk, "dv": r.dv}
    if s.call == "noalloc":
        o, lse = B.dcp_varlen_attn_fwd_noalloc(s.q, s.k, s.v, s.cu, s.max_seqlen, s.causal, s.o, s.lse)
        return {"o": o, "lse": lse}
    if s.call == "head_group":
        o, lse = B.dcp_varlen_attn_fwd_strided(s.q, s.k, s.v, s.cu, s.max_seqlen, s.causal, s.o, workspace=s.ws)
        dq, dk, dv = B.dcp_varlen_attn_bwd_strided(s.q, s.k, s.v, o, s.g, lse, s.cu, s.max_seqlen, s.causal, s.dq, s.dk, s.dv,
                                                   workspace=s.ws)
        return {"o": o, "lse": lse, "dq": dq, "dk": dk, "dv": dv}
    o, lse = B.dcp_varlen_attn_fwd(s.q, s.k, s.v, s.cu, s.max_seqlen, s.causal, workspace=s.ws)
    if s.call == "forward":
        return {"o": o, "lse": lse}
    dq, dk, dv = B.dcp_varlen_attn_bwd(s.q, s.k, s.v, o, s.g, lse, s.cu, s.max_seqlen, s.causal, workspace=s.ws)
    return {"o": o, "lse": lse, "dq": dq, "dk": dk, "dv": dv}


def work(case):
    """Forward: q, k, v read, o and lse written.  A training pass also reads dO and writes dq, dk, dv, and does 2.5 times
    the forward's products besides; a causal mask halves them.  (A stream's recomputed forwards and copies are not counted.)"""
    lengths, d = _lengths(case), case["head_dim"]
    heads = case.get("group", case["heads"])
    backward = case["call"] in ("train", "head_group", "stream")
    flops = 4.0 * sum(float(x) * x for x in lengths) * d * heads * (0.5 if case["causal"] else 1.0)
    rows = float(sum(lengths)) * heads
    return {"bytes": rows * ((8 if backward else 4) * d * 2 + 4), "flops": flops * (3.5 if backward else 1.0)}


def tolerance(case):
    # bf16 operands, probabilities and results with 32-bit sums: each output is within 3e-3 (2-norm) of the 64-bit
    # result on every mix, so two correct implementations differ by at most about the same; four times that is stated
    return {"rel": 1.2e-2}
