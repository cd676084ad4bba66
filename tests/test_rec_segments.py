"""The exact recurrence cut into segments along T (lawcat_gla_fwd / lawcat_layer_fwd outside the chunkwise kernels): lengths
at the edges of its 16-token batches and of its segments, carried states, and gates so sharp that a batch's decay leaves
the range in which the state is kept divided by it."""
import numpy as np
import pytest

from helpers import check, oracle_params
from oracle import lawcat_oracle as O
from paper_2509_18467_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,dk,dv", [("f32", 64, 64), ("f32", 128, 128), ("f32", 16, 128), ("bf16", 128, 64), ("f32", 32, 16)])
@pytest.mark.parametrize("T,sharp", [(15, 0), (16, 0), (17, 1), (63, 0), (65, 1), (257, 1), (1000, 0)])
def test_gla_fwd_segments(dtype, dk, dv, T, sharp):
    import torch
    from paper_2509_18467_b200 import api
    s = I.LayerShape(2, T, 4, 2, dk, dv, dtype=dtype, config_id=120)
    x = I.make(s, ["q", "k", "v", "gate", "S0", "z0"])
    x["q"], x["k"] = (I.round_to_bf16(np.abs(x["q"])), I.round_to_bf16(np.abs(np.repeat(x["k"], 2, axis=2))))
    x["gate"] = I.round_to_bf16(-np.abs(x["gate"]) * (np.float32(1.0) if sharp else np.float32(0.05)))
    if sharp:  # some channels lose e^-7 per token: 2^-160 over a batch
        x["gate"][:, T // 3:, :, ::3] = -7.0
    d = {n: api.to_device(v, "f32" if n in ("S0", "z0") else dtype) for n, v in x.items()}
    p = api.params(s.B, T, 4, 2, dk, dv, dtype=dtype, gate_mode=1)
    r = api.lawcat_gla_fwd(p, d["q"], d["k"], d["v"], d["gate"], d["S0"], d["z0"])
    torch.cuda.synchronize()
    ref = O.gla_fwd(oracle_params(s, gate_mode=1), x["q"], x["k"], x["v"], x["gate"], x["S0"], x["z0"])
    check(r["o"], ref["o"], dtype, "o")
    for n in ("den", "S_T", "z_T"):
        check(r[n], ref[n], dtype, n, f32_store=True)


@pytest.mark.parametrize("T", [16, 129, 700])
@pytest.mark.parametrize("d", [64, 128])
def test_plain_sigmoid_gate_layer(T, d):
    """tau = 1 on bf16 storage: features in fp32 between the stages, so the states stay close to the oracle's."""
    import torch
    from paper_2509_18467_b200 import api
    names = ["q", "k", "v", "gate", "w_q", "w_k", "W"]
    s = I.LayerShape(1, T, 4, 2, d, d, dtype="bf16", gate_tau=1.0, config_id=121)
    x = I.make(s, names + ["S0", "z0", "cache_q", "cache_k"])
    t = {n: api.to_device(v, "f32" if n in ("S0", "z0") else "bf16") for n, v in x.items()}
    r = api.lawcat_layer_fwd(api.params(1, T, 4, 2, d, d, gate_tau=1.0), *[t[n] for n in names], t["cache_q"], t["cache_k"],
                             t["S0"], t["z0"])
    torch.cuda.synchronize()
    ref = O.layer_fwd(oracle_params(s), *[x[n] for n in names], x["cache_q"], x["cache_k"], x["S0"], x["z0"])
    check(r["o"], ref["o"], "bf16", "o")
    check(r["S_T"], ref["S_T"], "f32", "S_T")
    check(r["z_T"], ref["z_T"], "f32", "z_T")
