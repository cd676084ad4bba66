"""The exact recurrence has two forms of its loop over a batch of sixteen tokens: a short one, and one written out that calls of at
least 128 batches take. Both against the fp64 oracle on either side of that line, and what the compiler reports of their registers."""
import os
import re

import numpy as np
import pytest

from helpers import check, oracle_params
from oracle import lawcat_oracle as O
from paper_2509_18467_b200 import build as B
from paper_2509_18467_b200 import inputs as I


def test_no_form_of_the_recurrence_lives_in_local_memory():
    """The state of a head lies in registers: a form that spills more than a few values pays for it in every batch."""
    report = os.path.join(B.OBJ, "gla_rec.ptxas")
    if not os.path.exists(report):
        pytest.skip("the library was not built here")
    text = open(report).read()
    kernels = re.findall(r"Compiling entry function '(\S*gla_fwd_rec_kernel\S*)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", text, re.S)
    assert len(kernels) >= 24
    for name, stores, loads in kernels:
        assert int(stores) <= 128 and int(loads) <= 192, (name, stores, loads)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,d,Hkv", [("f32", 128, 2), ("f32", 64, 4), ("f32", 16, 1), ("bf16", 128, 2), ("bf16", 64, 1)])
@pytest.mark.parametrize("T", [496, 497, 512, 530])
def test_both_sides_of_the_line(dtype, d, Hkv, T):
    """4 heads: 31 batches each are below it, 32 are on it. Some channels lose e^-7 per token, so that batches of both kinds occur (the
    state kept divided by its decay, and plainly)."""
    from paper_2509_18467_b200 import api
    names = ["q", "k", "v", "gate", "w_q", "w_k", "W"]
    s = I.LayerShape(1, T, 4, Hkv, d, d, dtype=dtype, config_id=122)
    x = I.make(s, names + ["S0", "z0"])
    x["gate"] = I.round_to_bf16(-np.abs(x["gate"]) * np.float32(0.05))
    x["gate"][:, T // 2:T // 2 + 40, :, ::3] = -7.0
    t = {n: api.to_device(v, "f32" if n in ("S0", "z0") else dtype) for n, v in x.items()}
    r = api.lawcat_layer_fwd(api.params(1, T, 4, Hkv, d, d, dtype=dtype, gate_mode=1, chunk=1), *[t[n] for n in names], None, None,
                             t["S0"], t["z0"])
    ref = O.layer_fwd(oracle_params(s, gate_mode=1), *[x[n] for n in names], None, None, x["S0"], x["z0"])
    check(r["o"], ref["o"], dtype, "o")
    for n in ("S_T", "z_T"):
        check(r[n], ref[n], "f32", n)
