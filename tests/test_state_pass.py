"""Sequences that are cut into segments: the start states come from the state-only pass, whose pieces of one or a few chunks
meet behind a scan. Against the fp64 oracle at the sizes and options where that pass takes a path of its own: pieces of one and
two chunks, two 64-wide heads per block and one (odd groups, one decay per head), the conv's halo in front of a piece, given
states, log-decay gates, and mix outputs too large to be exponentiated without the row's maximum."""
import numpy as np
import pytest

from helpers import check, oracle_params
from oracle import lawcat_oracle as O
from paper_2509_18467_b200 import inputs as I

pytestmark = pytest.mark.gpu

NAMES = ["q", "k", "v", "gate", "w_q", "w_k", "W"]


@pytest.mark.parametrize("d,H,Hkv,gate_dim", [(128, 2, 1, 0), (128, 2, 2, 1), (64, 4, 2, 0), (64, 3, 1, 0), (64, 2, 1, 1)])
@pytest.mark.parametrize("T,opt", [(512, ""), (577, "state"), (1300, "logdecay"), (1300, "large"), (2049, "state conv2")])
def test_cut_sequences(d, H, Hkv, gate_dim, T, opt):
    import torch
    from paper_2509_18467_b200 import api
    conv_k = 2 if "conv2" in opt else 4
    s = I.LayerShape(1, T, H, Hkv, d, d, conv_k=conv_k, gate_dim=gate_dim or d, dtype="bf16", config_id=94)
    x = I.make(s, NAMES + (["S0", "z0", "cache_q", "cache_k"] if "state" in opt else []))
    kw = {}
    if "logdecay" in opt:
        x["gate"] = I.round_to_bf16(-np.abs(x["gate"]) / 16)
        kw = dict(gate_mode=1)
    if "large" in opt:  # (every fifth key ten times as large: |y| up to about 40; beyond, the fp16 conv output is what the error is)
        x["k"] = I.round_to_bf16(x["k"] * np.where(np.arange(T) % 5 == 0, 10.0, 1.0)[None, :, None, None].astype(np.float32))
    t = {n: api.to_device(v, "f32" if n in ("S0", "z0") else "bf16") for n, v in x.items()}
    p = api.params(1, T, H, Hkv, d, d, conv_k=conv_k, gate_dim=gate_dim, **kw)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.trace_begin()
    r = api.lawcat_layer_fwd(p, *[t[n] for n in NAMES], t.get("cache_q"), t.get("cache_k"), t.get("S0"), t.get("z0"),
                             dev_status=status)
    assert "layer_tc_state" in api.trace_end() and int(status.item()) == 0
    ref = O.layer_fwd(oracle_params(s, **kw), *[x[n] for n in NAMES], x.get("cache_q"), x.get("cache_k"), x.get("S0"), x.get("z0"))
    for n in ("S_T", "z_T"):
        check(r[n], ref[n], "bf16", n, f32_store=True)
    check(r["o"], ref["o"], "bf16", "o")
