"""What a user of the layer has it do, as cases that can be timed and compared.

The layer is called in four ways, all on two model shapes (32 query / 8 key-value heads of width 64, hidden width 2048,
and the same heads of width 128, hidden width 4096): prefill of a prompt or of a piece of one, one decode step per
generated token, the gate function in front of either, and the distillation step (forward, then the gradients of the
whole layer). Sizes and options are those of the benchmark configurations and tests of this repository.

A case is a dict of plain values: `kind` (decode | gate | prefill | packed | train) and the shape and options of the call.
"""
import math
import random

import torch

from paper_2509_18467_b200 import api

SMALL = dict(H=32, H_kv=8, d=64)    # the 1B shape
LARGE = dict(H=32, H_kv=8, d=128)   # the 7B shape
CONV_K = 4


def listed():
    return [
        # one sequence being generated, one token: the smallest call there is, all launches and latency
        dict(name="decode-one", kind="decode", B=1, dtype="bf16", tau=16.0, **SMALL),
        # one token for each of a serving batch of 64 sequences: the fp32 states go through memory once
        dict(name="decode-batch", kind="decode", B=64, dtype="bf16", tau=16.0, **LARGE),
        # the gate function for that batch's tokens
        dict(name="gate-decode", kind="gate", tokens=64, d_model=4096, n_out=4096, rank=32),
        # the gate function over a whole long prompt
        dict(name="gate-prompt", kind="gate", tokens=32768, d_model=4096, n_out=4096, rank=32),
        # a turn of a conversation: an odd number of tokens behind a past, whose state and conv caches come in and go out
        dict(name="prefill-turn", kind="prefill", B=1, T=1223, dtype="bf16", tau=16.0, carry=True, **LARGE),
        # the headline: a 32K-token prompt on the 7B shape
        dict(name="prefill-long", kind="prefill", B=1, T=32768, dtype="bf16", tau=16.0, carry=False, **LARGE),
        # an 8K-token prompt on the 1B shape
        dict(name="prefill-1b", kind="prefill", B=1, T=8192, dtype="bf16", tau=16.0, carry=False, **SMALL),
        # the plain sigmoid gate (no power 1/tau), as the paper writes it
        dict(name="prefill-plain-gate", kind="prefill", B=1, T=4096, dtype="bf16", tau=1.0, carry=False, **LARGE),
        # 32-bit storage, the small verification shape
        dict(name="prefill-fp32", kind="prefill", B=1, T=512, dtype="f32", tau=16.0, carry=False, H=4, H_kv=4, d=64),
        # a serving loop's batch of prompts of different lengths, packed
        dict(name="prefill-packed", kind="packed", nseq=16, T=8192, **LARGE),
        # the distillation step on the 1B shape
        dict(name="train-1b", kind="train", B=8, T=1024, **SMALL),
        # the distillation step on the 7B shape, at a length of the paper's distillation data
        dict(name="train-7b", kind="train", B=4, T=1300, **LARGE),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.499)))))))


def draw(rng):
    """One of the listed uses at another size of its range; a drawn case is never larger than the listed one of its use."""
    use = rng.choice(["decode", "decode", "gate", "gate", "prefill", "prefill", "prefill", "plain", "fp32", "packed", "packed",
                      "train-1b", "train-1b", "train-7b", "train-7b"])
    shape = rng.choice([SMALL, LARGE])
    if use == "decode":
        return dict(kind="decode", B=_log_int(rng, 1, 64), dtype="bf16", tau=16.0, **shape)
    if use == "gate":
        width = shape["H"] * shape["d"]
        return dict(kind="gate", tokens=_log_int(rng, 1, 32768), d_model=width, n_out=width, rank=rng.choice([16, 32, 64, 128]))
    if use == "prefill":
        B = rng.choice([1, 1, 1, 2, 4])
        return dict(kind="prefill", B=B, T=_log_int(rng, 4, 32768 // B), dtype="bf16", tau=rng.choice([8.0, 16.0, 16.0]),
                    carry=rng.random() < 0.5, **shape)
    if use == "plain":
        return dict(kind="prefill", B=1, T=_log_int(rng, 16, 4096), dtype="bf16", tau=1.0, carry=rng.random() < 0.5, **shape)
    if use == "fp32":
        H = rng.choice([2, 4])
        return dict(kind="prefill", B=1, T=_log_int(rng, 4, 512), dtype="f32", tau=16.0, carry=rng.random() < 0.5, H=H,
                    H_kv=rng.choice([1, 2, H]), d=64)
    if use == "packed":
        T = _log_int(rng, 256, 8192)
        return dict(kind="packed", nseq=_log_int(rng, 2, min(32, T // 64)), T=T, **shape)
    if use == "train-1b":
        T = _log_int(rng, 64, 2048)
        return dict(kind="train", B=rng.randint(1, max(1, min(8, 8192 // T))), T=T, **SMALL)
    return dict(kind="train", B=rng.randint(1, 4), T=_log_int(rng, 64, 1300), **LARGE)


class _Maker:
    """Tensors of one seed, drawn on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(self, *shape, scale=1.0, dtype=torch.bfloat16):
        x = torch.randn(*shape, generator=self.g, device="cuda", dtype=torch.float32)
        return (x if scale == 1.0 else x.mul_(scale)).to(dtype)

    def uniform(self, *shape, lo, hi):
        return torch.rand(*shape, generator=self.g, device="cuda", dtype=torch.float32).mul_(hi - lo).add_(lo)


def _state(m, c, n, dt):
    """State and conv caches of n sequences with some hundred tokens behind them: the softmax features average 1/d and a
    decay of 2^-1/tau or so per token leaves about twice tau tokens in sight."""
    H, H_kv, d = c["H"], c["H_kv"], c["d"]
    seen = 2.0 * c.get("tau", 16.0)
    return dict(S=m.normal(n, H, d, d, scale=math.sqrt(seen) / d, dtype=torch.float32),
                z=m.uniform(n, H, d, lo=0.5 * seen / d, hi=1.5 * seen / d),
                cache_q=m.normal(n, CONV_K - 1, H * d, dtype=dt), cache_k=m.normal(n, CONV_K - 1, H_kv * d, dtype=dt))


def _params(c, B, T):
    return api.params(B, T, c["H"], c["H_kv"], c["d"], c["d"], conv_k=CONV_K, dtype=c.get("dtype", "bf16"),
                      gate_tau=c.get("tau", 16.0))


def _lengths(seed, nseq, T):
    """nseq prompt lengths that add up to T, spread over about a factor of ten."""
    r = random.Random(seed)
    w = [math.exp(r.uniform(0.0, math.log(10.0))) for _ in range(nseq)]
    ends = [round(T * sum(w[:i + 1]) / sum(w)) for i in range(nseq)]
    return [0] + ends[:-1] + [T]


def prepare(case, seed):
    c, m = case, _Maker(seed)
    dt = torch.float32 if c.get("dtype") == "f32" else torch.bfloat16
    if c["kind"] == "gate":
        n, dm, no, r = c["tokens"], c["d_model"], c["n_out"], c["rank"]
        d = 64 if dm == 2048 else 128
        return dict(case=c, p=api.params(1, n, no // d, no // d, d, d),
                    x=m.normal(1, n, dm), A1=m.normal(r, dm, scale=dm ** -0.5), A2=m.normal(no, r, scale=r ** -0.5),
                    bias=m.normal(no, scale=0.5))
    H, H_kv, d = c["H"], c["H_kv"], c["d"]
    s = dict(case=c, w_q=m.normal(H * d, CONV_K, scale=CONV_K ** -0.5, dtype=dt),
             w_k=m.normal(H_kv * d, CONV_K, scale=CONV_K ** -0.5, dtype=dt), W=m.normal(H, d, d, scale=d ** -0.5, dtype=dt))
    if c["kind"] == "decode":
        B = c["B"]
        s.update(p=_params(c, B, 1), q=m.normal(B, H, d, dtype=dt), k=m.normal(B, H_kv, d, dtype=dt),
                 v=m.normal(B, H_kv, d, dtype=dt), gate=m.normal(B, H, d, dtype=dt), **_state(m, c, B, dt))
        return s
    B, T = c.get("B", 1), c["T"]
    s.update(p=_params(c, B, T), q=m.normal(B, T, H, d, dtype=dt), k=m.normal(B, T, H_kv, d, dtype=dt),
             v=m.normal(B, T, H_kv, d, dtype=dt), gate=m.normal(B, T, H, d, dtype=dt))
    if c["kind"] == "train":
        s["dO"] = m.normal(B, T, H, d, dtype=dt)
    elif c["kind"] == "packed":
        s["cu_seqlens"] = _lengths(seed, c["nseq"], T)
    elif c["carry"]:
        s.update(_state(m, c, B, dt))
    return s


def run(state):
    s = state
    kind, p = s["case"]["kind"], s["p"]
    if kind == "gate":
        return api.lawcat_gate_fn_fwd(p, s["case"]["d_model"], s["case"]["rank"], s["x"], s["A1"], s["A2"], s["bias"])
    layer = (s["q"], s["k"], s["v"], s["gate"], s["w_q"], s["w_k"], s["W"])
    if kind == "decode":  # the state and the caches advance in place
        o = api.lawcat_decode_step(p, *layer, s["S"], s["z"], s["cache_q"], s["cache_k"])
        return dict(o=o, S=s["S"], z=s["z"], cache_q=s["cache_q"], cache_k=s["cache_k"])
    if kind == "packed":
        return api.lawcat_layer_fwd_varlen(p, s["cu_seqlens"], *layer)
    if kind == "train":
        out = api.lawcat_layer_fwd(p, *layer, want_state=False, want_cache=False)
        return dict(api.lawcat_layer_bwd(p, *layer, s["dO"]), o=out["o"])
    return api.lawcat_layer_fwd(p, *layer, s.get("cache_q"), s.get("cache_k"), s.get("S"), s.get("z"))


def work(case):
    c = case
    if c["kind"] == "gate":
        n, dm, no, r = c["tokens"], c["d_model"], c["n_out"], c["rank"]
        return dict(bytes=2 * (n * dm + n * no + r * dm + no * r + no), flops=2 * n * r * (dm + no))
    H, H_kv, d = c["H"], c["H_kv"], c["d"]
    es = 4 if c.get("dtype") == "f32" else 2
    seqs = c.get("nseq", c.get("B", 1))
    tokens = {"decode": c.get("B"), "packed": c.get("T")}.get(c["kind"], c.get("B", 1) * c.get("T", 1))
    weights = es * ((H + H_kv) * d * CONV_K + H * d * d)
    state, caches = 4 * seqs * H * (d * d + d), es * seqs * (CONV_K - 1) * (H + H_kv) * d
    per_token_in, per_token_out = es * (2 * H + 2 * H_kv) * d, es * H * d
    # conv, the shared linear layer on both streams, state update and read-out with their normalizer
    flops = tokens * H * (2 * CONV_K * d * (1 + H_kv / H) + 4 * d * d + 4 * d * (d + 1))
    if c["kind"] == "decode":
        return dict(bytes=tokens * (per_token_in + per_token_out) + weights + 2 * state + 2 * caches, flops=flops)
    if c["kind"] == "train":
        # forward: inputs in, o out; backward: inputs and dO in, their gradients out, the weights' gradients out in fp32
        moved = tokens * (per_token_in + per_token_out + per_token_in + per_token_out + per_token_in)
        return dict(bytes=moved + 2 * weights + 2 * weights, flops=3 * flops)
    moved = tokens * (per_token_in + per_token_out) + weights + state + caches
    return dict(bytes=moved + (state + caches if c.get("carry") else 0), flops=flops)


def tolerance(case):
    """bf16 storage with 16-bit tensor-core operands: 1e-2 (a value stored in bf16 alone is off by up to 2^-8 of itself);
    32-bit storage: what fp32 sums in another order show."""
    if case.get("dtype") == "f32":
        return dict(rel=1e-5, max=1e-3)
    return dict(rel=1e-2, max=0.03)
