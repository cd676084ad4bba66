"""Packed variable-length sequences (lawcat_layer_fwd_varlen): every sequence of the pack against the oracle run on that
sequence alone (so the state and the conv are reset at every boundary), with and without carried-in states and caches, on
the tensor-core path (bf16, d = 128) and on the exact path (fp32)."""
import numpy as np
import pytest

from helpers import check, oracle_params
from oracle import lawcat_oracle as O
from paper_2509_18467_b200 import inputs as I



NAMES = ["q", "k", "v", "gate", "w_q", "w_k", "W"]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 64), ("f32", 32)])
@pytest.mark.parametrize("with_state", [False, True])
def test_packed_sequences_match_the_oracle_one_by_one(dtype, d, with_state):
    import dataclasses
    import torch
    from paper_2509_18467_b200 import api
    lens = [1, 63, 0, 200, 700, 64]
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    s = I.LayerShape(1, cu[-1], 4, 2, d, d, dtype=dtype, config_id=95)
    x = I.make(s, NAMES)
    st = I.make(dataclasses.replace(s, B=len(lens)), ["S0", "z0", "cache_q", "cache_k"]) if with_state else {}
    dv = {n: api.to_device(v, dtype) for n, v in x.items()}
    ds = {n: api.to_device(v, "f32" if n in ("S0", "z0") else dtype) for n, v in st.items()}
    p = api.params(1, s.T, s.H, s.H_kv, d, d, dtype=dtype)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    r = api.lawcat_layer_fwd_varlen(p, cu, *[dv[n] for n in NAMES], ds.get("cache_q"), ds.get("cache_k"), ds.get("S0"),
                                    ds.get("z0"), dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for i, n in enumerate(lens):
        lo, hi = cu[i], cu[i + 1]
        sub = dataclasses.replace(s, T=n)
        init = {k2: (v[i:i + 1] if k2 in st else None) for k2, v in st.items()}
        if n == 0:  # an empty sequence hands its state through
            want_S = st["S0"][i] if with_state else np.zeros_like(r["S_T"][i].cpu().numpy())
            assert np.array_equal(r["S_T"][i].cpu().numpy(), want_S)
            continue
        ref = O.layer_fwd(oracle_params(sub), *[x[m][:, lo:hi] for m in NAMES[:4]], *[x[m] for m in NAMES[4:]],
                          init.get("cache_q"), init.get("cache_k"), init.get("S0"), init.get("z0"))
        check(r["o"][:, lo:hi], ref["o"], dtype, f"o of sequence {i}")
        check(r["S_T"][i:i + 1], ref["S_T"], dtype, f"S_T of sequence {i}", f32_store=True)
        check(r["z_T"][i:i + 1], ref["z_T"], dtype, f"z_T of sequence {i}", f32_store=True)
        assert np.array_equal(r["cache_q"][i:i + 1].float().cpu().numpy(), ref["cache_q"].astype(np.float32))
        assert np.array_equal(r["cache_k"][i:i + 1].float().cpu().numpy(), ref["cache_k"].astype(np.float32))


@pytest.mark.gpu
@pytest.mark.parametrize("d,gate_dim", [(128, 0), (64, 0), (128, 1)])
def test_many_sequences_share_the_launches(d, gate_dim):
    """More sequences than one launch's table holds, one long enough to be cut into segments, the others around the chunk
    length and too short for the chunkwise kernel."""
    import dataclasses
    import torch
    from paper_2509_18467_b200 import api
    lens = [16, 64, 65, 20 if gate_dim else 1, 0, 2100, 127, 128, 129] + [17 + 5 * (i % 13) for i in range(66)]
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    s = I.LayerShape(1, cu[-1], 4, 2, d, d, gate_dim=gate_dim, dtype="bf16", config_id=96)
    x = I.make(s, NAMES)
    st = I.make(dataclasses.replace(s, B=len(lens)), ["S0", "z0", "cache_q", "cache_k"])
    dv = {n: api.to_device(v, "bf16") for n, v in x.items()}
    ds = {n: api.to_device(v, "f32" if n in ("S0", "z0") else "bf16") for n, v in st.items()}
    p = api.params(1, s.T, s.H, s.H_kv, d, d, gate_dim=gate_dim)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    n0 = api.launch_count()
    r = api.lawcat_layer_fwd_varlen(p, cu, *[dv[n] for n in NAMES], ds["cache_q"], ds["cache_k"], ds["S0"], ds["z0"],
                                    dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and api.launch_count() - n0 <= 14
    for i in [0, 1, 2, 3, 5, 6, 7, 8, 9, 40, 73, 74]:
        lo, hi = cu[i], cu[i + 1]
        ref = O.layer_fwd(oracle_params(dataclasses.replace(s, T=hi - lo)), *[x[m][:, lo:hi] for m in NAMES[:4]],
                          *[x[m] for m in NAMES[4:]], *[st[m][i:i + 1] for m in ("cache_q", "cache_k", "S0", "z0")])
        check(r["o"][:, lo:hi], ref["o"], "bf16", f"o of sequence {i}")
        check(r["S_T"][i:i + 1], ref["S_T"], "bf16", f"S_T of sequence {i}", f32_store=True)
        check(r["z_T"][i:i + 1], ref["z_T"], "bf16", f"z_T of sequence {i}", f32_store=True)
        assert np.array_equal(r["cache_q"][i:i + 1].float().cpu().numpy(), ref["cache_q"].astype(np.float32))
        assert np.array_equal(r["cache_k"][i:i + 1].float().cpu().numpy(), ref["cache_k"].astype(np.float32))


@pytest.mark.gpu
@pytest.mark.parametrize("d,H,H_kv,gate_dim", [(128, 4, 2, 0), (64, 4, 2, 0), (64, 2, 2, 0), (128, 2, 1, 1)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), 1.0e5, 3.0e38])
def test_a_sequence_does_not_reach_its_neighbours(d, H, H_kv, gate_dim, bad):
    """Every token of one sequence of the pack is not finite, or beyond the range of fp16: the sequences in front of it (whose
    last chunk it shares) and behind it keep their outputs and states bit for bit."""
    import torch
    from paper_2509_18467_b200 import api
    lens = [100, 80, 65, 17, 700, 90, 130]
    cu = np.concatenate([[0], np.cumsum(lens)]).tolist()
    s = I.LayerShape(1, cu[-1], H, H_kv, d, d, gate_dim=gate_dim, dtype="bf16", config_id=97)
    t = {n: api.to_device(v, "bf16") for n, v in I.make(s, NAMES).items()}
    p = api.params(1, s.T, H, H_kv, d, d, gate_dim=gate_dim)
    ref = api.lawcat_layer_fwd_varlen(p, cu, *[t[n] for n in NAMES])
    poisoned = (1, 3, 5)
    for i in poisoned:
        for n in ("q", "k", "v") + (("gate",) if bad != bad else ()):
            t[n][:, cu[i]:cu[i + 1]] = bad
    r = api.lawcat_layer_fwd_varlen(p, cu, *[t[n] for n in NAMES])
    torch.cuda.synchronize()
    for i in set(range(len(lens))) - set(poisoned):
        assert torch.equal(r["o"][:, cu[i]:cu[i + 1]], ref["o"][:, cu[i]:cu[i + 1]]), f"o of sequence {i}"
        for n in ("S_T", "z_T"):
            assert bool(torch.isfinite(ref[n][i]).all()) and torch.equal(r[n][i], ref[n][i]), f"{n} of sequence {i}"


def test_bad_offsets_are_refused_on_the_host():
    import ctypes
    from paper_2509_18467_b200 import api
    L = api.lib()
    p = api.params(1, 10, 2, 1, 64, 64)
    ok = ctypes.c_void_p(0x1000)
    f = L.lawcat_layer_fwd_varlen
    f.restype = ctypes.c_int
    f.argtypes = [ctypes.POINTER(api.Params), ctypes.c_void_p, ctypes.c_int] + [ctypes.c_void_p] * 17 + \
                 [ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p]
    args = [ok] * 7 + [None] * 4 + [ok] + [None] * 4 + [ok, 1 << 30, None, None]
    for bad in ([0, 4, 9], [1, 4, 10], [0, 6, 4, 10]):
        cu = (ctypes.c_int32 * len(bad))(*bad)
        assert f(ctypes.byref(p), cu, len(bad) - 1, *args) == 1
    p2 = api.params(2, 10, 2, 1, 64, 64)
    cu = (ctypes.c_int32 * 2)(0, 10)
    assert f(ctypes.byref(p2), cu, 1, *args) == 1
