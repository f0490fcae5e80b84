"""Performance cases of the dual-state linear attention (DSLA) layer.

Each case is one call of a public entry point on inputs that are already on the GPU, at sizes that an
inference server of Llama2-7B-shaped layers (32 heads of 128) meets: prompts from a few tokens to 64K, single
requests and packed batches, fresh prompts and continued ones, decode batches from one row to a full
batch.  The fp32 layer with heads of 64 and the wider forms of the layer (gates per key channel, n states,
masked rows, the gate producer) are there with the sizes they have in this repository's benchmark and tests.

A caller keeps its output buffer, its workspace and its state store between calls, as a serving loop does.
"""
from __future__ import annotations

import math

import torch

import paper_2506_09316_b200 as dsla
from paper_2506_09316_b200 import inputs as gen

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
D_MODEL = 4096


def _decode(name, B, H=32, d=128, dtype="bf16", n=2, channel=False, masked=False):
    return dict(name=name, kind="decode", B=B, H=H, d=d, dtype=dtype, n=n, channel=channel, masked=masked)


def _prefill(name, lens, H=32, d=128, dtype="bf16", n=2, channel=False, resume=False):
    """``lens``: prompt lengths as text, or "lo:hi:count:seed" for lengths drawn log-uniformly from [lo, hi]."""
    return dict(name=name, kind="prefill", lens=lens, H=H, d=d, dtype=dtype, n=n, channel=channel, resume=resume)


def listed():
    return [
        # one chat user: the next token of one sequence in one layer; what the serving loop calls most often
        _decode("decode_1", 1),
        # a full decode batch of one layer: 128 sequences, 537 MB of states
        _decode("decode_128", 128),
        # a mixed batch in which about half of the rows belong to this layer, gates per key channel
        _decode("decode_channel_mask", 45, channel=True, masked=True),
        # a short chat prompt of odd length
        _prefill("prefill_777", "777"),
        # the Llama2-7B-shaped layer on a 4K prompt (the benchmark's default workload)
        _prefill("prefill_4k", "4096"),
        # one long document: 64K tokens
        _prefill("prefill_64k", "65536"),
        # a packed batch of 16 fresh prompts, log-uniform in [1K, 64K], 335K tokens
        _prefill("prefill_ragged", "1024:65536:16:1005"),
        # pieces of 8 prompts of odd lengths that continue from the states in their slots (prompts fed piece by piece)
        _prefill("prefill_resume", "301,512,77,1000,643,129,850,64", resume=True),
        # the small fp32 layer: 4 heads of 64, 512 tokens
        _prefill("prefill_f32", "512", H=4, d=64, dtype="f32"),
        # gates per key channel (the gated-linear-attention form) on the 4K prompt
        _prefill("prefill_channel", "4096", channel=True),
        # four states per head (the number-of-states ablation) on the 4K prompt
        _prefill("prefill_n4", "4096", n=4),
        # the gates of a 4K prompt from the layer's input
        dict(name="gates_4k", kind="gates", T=4096, H=32, D=D_MODEL),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "prompt", "prompt", "packed", "resume", "f32", "channel", "nstate", "gates"])
    H = rng.choice([8, 16, 24, 32, 32, 40])
    if kind == "decode":
        n = rng.choice([2, 2, 2, 1, 4])
        c = _decode("", _log_int(rng, 1, 200), H=H, d=rng.choice([64, 128, 128]), dtype=rng.choice(["bf16", "bf16", "f32"]), n=n,
                    channel=rng.random() < 0.3, masked=rng.random() < 0.3)
    elif kind == "prompt":
        c = _prefill("", str(_log_int(rng, 16, 65536)), H=rng.choice([8, 16, 24, 32]))
    elif kind == "packed":
        count = rng.randint(2, 24)
        hi = _log_int(rng, 512, min(65536, 200000 // count))
        c = _prefill("", "%d:%d:%d:%d" % (max(16, hi // 64), hi, count, rng.randrange(1 << 20)), H=rng.choice([8, 16, 24, 32]))
    elif kind == "resume":
        lens = [_log_int(rng, 16, 2048) for _ in range(rng.randint(1, 12))]
        c = _prefill("", ",".join(str(x) for x in lens), H=H, resume=True)
    elif kind == "f32":
        c = _prefill("", str(_log_int(rng, 32, 2048)), H=rng.randint(2, 16), d=rng.choice([64, 128]), dtype="f32", resume=rng.random() < 0.3)
    elif kind == "channel":
        c = _prefill("", str(_log_int(rng, 64, 4096)), H=rng.choice([8, 16, 32]), channel=True, resume=rng.random() < 0.3)
    elif kind == "nstate":
        c = _prefill("", str(_log_int(rng, 64, 8192)), H=rng.choice([8, 16, 32]), n=rng.choice([1, 4, 8]), resume=rng.random() < 0.3)
    else:
        c = dict(kind="gates", T=_log_int(rng, 1, 65536), H=rng.choice([16, 32, 32, 40]), D=rng.choice([2048, 4096, 5120]))
    c.pop("name", None)
    return c


def _lengths(case):
    if ":" in case["lens"]:
        lo, hi, count, seed = (int(x) for x in case["lens"].split(":"))
        return [int(x) for x in gen.ragged_lengths(seed, count, lo, hi)]
    return [int(x) for x in case["lens"].split(",")]


def _gate_means(n):
    """Pre-activation means of the states' gates, slow to fast: (6, 1) for the dual state."""
    return [6.0] if n == 1 else [6.0 - 5.0 * i / (n - 1) for i in range(n)]


class _Draw:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def normal(self, shape, scale, dtype):
        out = torch.empty(shape, dtype=dtype, device="cuda")
        rows = max(1, (1 << 28) // max(1, math.prod(shape[1:])))
        for r in range(0, shape[0], rows):
            e = min(shape[0], r + rows)
            out[r:e] = torch.randn((e - r,) + tuple(shape[1:]), generator=self.g, device="cuda") * scale
        return out

    def gates(self, shape, mean):
        return torch.sigmoid(torch.randn(shape, generator=self.g, device="cuda") * 0.5 + mean)

    def uniform(self, shape):
        return torch.rand(shape, generator=self.g, device="cuda")

    def permutation(self, n):
        return torch.randperm(n, generator=self.g, device="cuda").to(torch.int32)


def prepare(case, seed):
    r = _Draw(seed)
    if case["kind"] == "gates":
        T, H, D = case["T"], case["H"], case["D"]
        return dict(kind="gates", x=r.normal((T, D), 1.0, torch.bfloat16), w=r.normal((2 * H, D), 1.0 / math.sqrt(D), torch.bfloat16),
                    bias=r.uniform((2 * H,)) * 6.0, g_hist=torch.empty(T, H, device="cuda"), g_rec=torch.empty(T, H, device="cuda"))
    H, d, n, dtype = case["H"], case["d"], case["n"], DTYPES[case["dtype"]]
    lens = _lengths(case) if case["kind"] == "prefill" else None
    rows = sum(lens) if lens else case["B"]
    seqs = len(lens) if lens else case["B"]
    s = dict(kind=case["kind"], n=n)
    for name in ("q", "k", "v"):
        s[name] = r.normal((rows, H, d), 1.0 / math.sqrt(d), dtype)
    gates = [r.gates((rows, H, d) if case["channel"] else (rows, H), m) for m in _gate_means(n)]
    if n == 2:
        s["g_hist"], s["g_rec"], s["gamma"] = gates[0], gates[1], r.uniform((H,))
        s["st"] = dsla.dsla_state_alloc(seqs, H, d, d)
    else:
        w = r.uniform((H, n))
        s["gates"], s["weights"] = torch.stack(gates), (w / w.sum(1, keepdim=True)).contiguous()
        s["st"] = dsla.dsla_state_alloc_n(seqs, n, H, d, d)
    for slot in range(seqs):
        s["st"].tensor[slot].normal_(0.0, 0.02, generator=r.g)
    s["o"] = torch.zeros_like(s["v"])
    s["slots"] = r.permutation(seqs) if seqs > 1 else None
    if case["kind"] == "decode":
        s["mask"] = (r.uniform((seqs,)) < 0.5).to(torch.uint8) if case["masked"] else None
        return s
    s["resume"] = bool(case["resume"])
    s["cu"] = None
    s["longest"] = max(lens)
    if seqs > 1:
        s["cu"] = torch.tensor([0] + lens, device="cuda").cumsum(0).to(torch.int32)
    if n == 2:
        need = dsla.dsla_prefill_workspace_bytes(rows, seqs, s["longest"], H, d, dtype, dense_T=None if seqs > 1 else s["longest"])
    else:
        need = dsla.dsla_nstate_prefill_workspace_bytes(s["q"], s["k"], s["v"], s["gates"], s["weights"], cu_seqlens=s["cu"],
                                                        max_seqlen=s["longest"])
    s["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda") if need else None
    return s


def run(s):
    if s["kind"] == "gates":
        return dsla.dsla_gate_project(s["x"], s["w"], s["bias"], g_hist=s["g_hist"], g_rec=s["g_rec"])
    if s["kind"] == "decode":
        if s["n"] == 2:
            o = dsla.dsla_decode_step(s["q"], s["k"], s["v"], s["g_hist"], s["g_rec"], s["gamma"], s["st"], o=s["o"], slots=s["slots"],
                                      row_mask=s["mask"])
        else:
            o = dsla.dsla_nstate_decode_step(s["q"], s["k"], s["v"], s["gates"], s["weights"], s["st"], o=s["o"], slots=s["slots"],
                                             row_mask=s["mask"])
    elif s["n"] == 2:
        o = dsla.dsla_prefill(s["q"], s["k"], s["v"], s["g_hist"], s["g_rec"], s["gamma"], s["st"], o=s["o"], cu_seqlens=s["cu"],
                              slots=s["slots"], max_seqlen=s["longest"], use_initial_state=s["resume"], workspace=s["ws"])
    else:
        o = dsla.dsla_nstate_prefill(s["q"], s["k"], s["v"], s["gates"], s["weights"], s["st"], o=s["o"], cu_seqlens=s["cu"],
                                     slots=s["slots"], max_seqlen=s["longest"], use_initial_state=s["resume"], workspace=s["ws"])
    return o, s["st"].tensor


def work(case):
    """q, k, v, o and the gates once; the states read where the call starts from them and written once.  Operations of the
    recurrence: per state, token and head one rank-1 update and one readout of a d x d state."""
    if case["kind"] == "gates":
        T, H, D = case["T"], case["H"], case["D"]
        return {"bytes": 2 * T * D + 4 * H * D + 8 * H + 8 * T * H, "flops": 4.0 * T * H * D}
    H, d, n = case["H"], case["d"], case["n"]
    es = 2 if case["dtype"] == "bf16" else 4
    gate = n * 4 * (d if case["channel"] else 1)
    state = n * d * d * 4
    if case["kind"] == "decode":
        rows = case["B"] * (0.5 if case["masked"] else 1.0)
        return {"bytes": rows * H * (2 * state + 4 * d * es + gate), "flops": rows * H * n * 4.0 * d * d}
    lens = _lengths(case)
    tokens = sum(lens)
    return {"bytes": tokens * H * (4 * d * es + gate) + len(lens) * H * state * (2 if case["resume"] else 1),
            "flops": tokens * H * n * 4.0 * d * d}


def tolerance(case):
    """bf16 results of fp32 arithmetic differ by their last rounding (2^-9 each); the bf16 prompt kernels round their products'
    factors to bf16 as well; everything else is a 32-bit sum."""
    if case["kind"] == "gates" or case["dtype"] == "f32":
        return {"rel": 1e-5}
    if case["kind"] == "decode" or case["channel"]:
        return {"rel": 4e-3}
    return {"rel": 1e-2}
