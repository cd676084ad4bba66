"""A bounded device-side wait that runs out: the tensor-core layer kernel and the streaming decode kernel report
LAWCAT_ERR_TIMEOUT through dev_status, return, and leave the device usable (the next ordinary call is parity-green).

Nothing is made to fault or hang. The test only shortens the bound of the kernel's waits, through the library's test hook,
to a few hundred clock cycles, less than any copy or product takes, so the first wait that is not already satisfied gives
up. The kernel itself is the one every other test runs."""
import pytest

from helpers import check, oracle_params
from oracle import lawcat_oracle as O
from paper_2509_18467_b200 import inputs as I

pytestmark = pytest.mark.gpu

NAMES = ["q", "k", "v", "gate", "w_q", "w_k", "W"]


@pytest.mark.parametrize("T", [40, 700])
def test_wait_that_runs_out_is_reported_and_the_device_stays_usable(T):
    import torch
    from paper_2509_18467_b200 import api
    s = I.LayerShape(1, T, 2, 1, 128, 128, dtype="bf16", config_id=91)
    x = I.make(s, NAMES)
    d = {n: api.to_device(v, s.dtype) for n, v in x.items()}
    p = api.params(s.B, s.T, s.H, s.H_kv, s.d_k, s.d_v)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    try:
        api.test_set_wait_limit(300)
        api.trace_begin()
        api.lawcat_layer_fwd(p, *[d[n] for n in NAMES], dev_status=status)
        kernels = api.trace_end()   # (waits for the kernel: it must return by itself)
    finally:
        api.test_set_wait_limit(0)
    assert any(k.startswith("layer_tc") for k in kernels)
    torch.cuda.synchronize()
    assert int(status.item()) == 5, int(status.item())          # LAWCAT_ERR_TIMEOUT
    assert api.status_string(5) == "bounded device wait ran out"
    # the same call with the default bound: no status, parity with the oracle
    status.zero_()
    r = api.lawcat_layer_fwd(p, *[d[n] for n in NAMES], dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = O.layer_fwd(oracle_params(s), *[x[n] for n in NAMES])
    check(r["o"], ref["o"], "bf16", "o")
    check(r["S_T"], ref["S_T"], "bf16", "S_T", f32_store=True)


@pytest.mark.parametrize("d", [128, 64])
def test_wait_of_a_packed_launch_that_runs_out(d):
    """(the last chunk of a packed sequence passes through barriers of its own)"""
    import torch
    from paper_2509_18467_b200 import api
    cu = [0, 40, 170, 234, 934]
    s = I.LayerShape(1, cu[-1], 2, 1, d, d, dtype="bf16", config_id=93)
    t = [api.to_device(v, "bf16") for v in I.make(s, NAMES).values()]
    p = api.params(1, s.T, 2, 1, d, d)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref = api.lawcat_layer_fwd_varlen(p, cu, *t)
    try:
        api.test_set_wait_limit(300)
        api.lawcat_layer_fwd_varlen(p, cu, *t, dev_status=status)
        torch.cuda.synchronize()
    finally:
        api.test_set_wait_limit(0)
    assert int(status.item()) == 5
    status.zero_()
    r = api.lawcat_layer_fwd_varlen(p, cu, *t, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and torch.equal(r["o"], ref["o"]) and torch.equal(r["S_T"], ref["S_T"])


@pytest.mark.parametrize("d,B", [(128, 16), (64, 48)])
def test_wait_of_the_streaming_decode_step_that_runs_out(d, B):
    import torch
    from paper_2509_18467_b200 import api
    s = I.LayerShape(B, 1, 32, 8, d, d, dtype="bf16", config_id=92)
    x = I.make(s, NAMES + ["S0", "z0", "cache_q", "cache_k"])
    p = api.params(B, 1, 32, 8, d, d)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def step():
        t = {n: api.to_device(v, "f32" if n in ("S0", "z0") else "bf16") for n, v in x.items()}
        t.update({n: t[n][:, 0].contiguous() for n in ("q", "k", "v", "gate")})
        api.trace_begin()
        o = api.lawcat_decode_step(p, *[t[n] for n in NAMES], t["S0"], t["z0"], t["cache_q"], t["cache_k"], dev_status=status)
        kernels = api.trace_end()   # (waits for the kernel: it must return by itself)
        assert "decode_stream" in kernels
        torch.cuda.synchronize()
        return o, t

    try:
        api.test_set_wait_limit(300)
        step()
    finally:
        api.test_set_wait_limit(0)
    assert int(status.item()) == 5          # LAWCAT_ERR_TIMEOUT
    status.zero_()
    o, t = step()
    assert int(status.item()) == 0
    ref = O.decode_step(oracle_params(s), *[x[n] for n in NAMES], x["S0"], x["z0"], x["cache_q"], x["cache_k"])
    check(o, ref["o"], "bf16", "o")
    check(t["S0"], ref["S"], "bf16", "S", f32_store=True)
    check(t["z0"], ref["z"], "bf16", "z", f32_store=True)
