"""Batches of so many short sequences that (sequences x heads) passes 65 535, the limit of a launch's second and third axis.
The batch repeats five sequences, so the oracle runs on those alone and every repetition has to agree with the first bit for
bit; weight gradients are the sum over all of them."""
import numpy as np
import pytest

from helpers import check, oracle_params
from oracle import lawcat_oracle as O
from paper_2509_18467_b200 import inputs as I
from test_layer_bwd import oracle_layer_gradients

pytestmark = pytest.mark.gpu

NAMES = ["q", "k", "v", "gate", "w_q", "w_k", "W"]
PER_TOKEN = ("q", "k", "v", "gate", "dO", "d_qdot", "d_kdot")
BASE, REP, H = 5, 205, 64   # 1025 sequences of 64 heads: 65 600


def setup(T, d, names, **kw):
    import torch
    from paper_2509_18467_b200 import api
    s = I.LayerShape(BASE, T, H, H, d, d, dtype="bf16", config_id=130, **kw)
    x = I.make(s, names)
    t = {n: api.to_device(v, "bf16") for n, v in x.items()}
    t = {n: v.repeat(REP, *[1] * (v.dim() - 1)) if n in PER_TOKEN else v for n, v in t.items()}
    assert BASE * REP * H > 65535 and torch.cuda.is_available()
    return api, s, x, t, api.params(BASE * REP, T, H, H, d, d, gate_tau=s.gate_tau)


def check_repeats(y, ref, what):
    import torch
    check(y[:BASE], ref, "bf16", what)
    assert torch.equal(y.view(REP, BASE, *y.shape[1:]), y[:BASE].expand(REP, *y[:BASE].shape)), what


@pytest.mark.parametrize("T,tau", [(4, 16.0), (20, 1.0)])
def test_layer_forward_of_the_exact_path(T, tau):
    api, s, x, t, p = setup(T, 64, NAMES, gate_tau=tau)
    r = api.lawcat_layer_fwd(p, *[t[n] for n in NAMES], want_state=False, want_cache=False)
    check_repeats(r["o"], O.layer_fwd(oracle_params(s), *[x[n] for n in NAMES])["o"], "o")


@pytest.mark.parametrize("d", [64, 128])
def test_layer_backward(d):
    api, s, x, t, p = setup(16, d, NAMES + ["dO"])
    g = api.lawcat_layer_bwd(p, *[t[n] for n in NAMES], t["dO"])
    ref = oracle_layer_gradients(s, x)
    for n in ("dq", "dk", "dv", "dgate"):
        check_repeats(g[n], ref[n], n)
    for n in ("dw_q", "dw_k", "dW"):
        check(g[n], REP * np.asarray(ref[n]), "bf16", n, f32_store=True)


def test_conv_and_mix_forward_and_backward():
    api, s, x, t, p = setup(4, 64, NAMES + ["d_qdot", "d_kdot"])
    qd, kd = api.lawcat_conv_fwd(p, t["q"], t["k"], t["w_q"], t["w_k"], t["W"])
    ref = O.layer_fwd(oracle_params(s), *[x[n] for n in NAMES])
    check_repeats(qd, ref["qdot"], "qdot")
    check_repeats(kd, ref["kdot"], "kdot")
    g = api.lawcat_conv_bwd(p, t["q"], t["k"], t["w_q"], t["w_k"], t["W"], t["d_qdot"], t["d_kdot"])
    ref = O.conv_bwd(oracle_params(s), x["q"], x["k"], x["w_q"], x["w_k"], x["W"], x["d_qdot"], x["d_kdot"])
    for n in ("dq", "dk"):
        check_repeats(g[n], ref[n], n)
    for n in ("dw_q", "dw_k", "dW"):
        check(g[n], REP * np.asarray(ref[n]), "bf16", n, f32_store=True)
