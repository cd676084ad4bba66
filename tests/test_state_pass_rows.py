"""The state-only pass in front of a cut sequence, and conv + mix, at rows that the ordinary inputs do not have: mix outputs that overflow
unless the row's maximum is taken off, rows and parts of rows whose maximum is negative, keys that are not finite, a decay of zero; and
a batch whose sequences are all cut. The segments of a call of 1300 tokens and few heads are 320 tokens long."""
import numpy as np
import pytest

from helpers import oracle_params
from oracle import lawcat_oracle as O
from paper_2509_18467_b200 import inputs as I

pytestmark = pytest.mark.gpu

NAMES = ["q", "k", "v", "gate", "w_q", "w_k", "W"]
SHAPES = [(128, 2, 1, 0), (128, 2, 2, 1), (64, 4, 2, 0), (64, 3, 1, 0), (64, 2, 1, 1)]  # d, H, Hkv, gate_dim
SEG = 320


def layer(s, x, status=None, **kw):
    from paper_2509_18467_b200 import api
    t = {n: api.to_device(v, "f32" if n in ("S0", "z0") else "bf16") for n, v in x.items()}
    p = api.params(s.B, s.T, s.H, s.H_kv, s.d_k, s.d_v, gate_dim=s.gate_dim, gate_tau=s.gate_tau, **kw)
    api.trace_begin()
    r = api.lawcat_layer_fwd(p, *[t[n] for n in NAMES], t.get("cache_q"), t.get("cache_k"), t.get("S0"), t.get("z0"), dev_status=status)
    return {n: v.float().cpu().numpy() for n, v in r.items()}, api.trace_end()


def oracle(s, x):
    return O.layer_fwd(oracle_params(s), *[x[n] for n in NAMES], x.get("cache_q"), x.get("cache_k"), x.get("S0"), x.get("z0"))


def mix_of_keys(s, x):
    """The key stream's mix outputs per query head, and the sums of their terms' magnitudes."""
    u = np.asarray(O.conv(x["k"], x["w_k"], x.get("cache_k"), s.conv_k)).reshape(s.B, s.T, s.H_kv, s.d_k)
    u = np.repeat(u, s.H // s.H_kv, axis=2)
    W = x["W"].astype(np.float64)
    return np.einsum("bthc,hce->bthe", u, W), np.einsum("bthc,hce->bthe", np.abs(u), np.abs(W))


def state_bound(s, x, e):
    """Elementwise bounds of S_T and z_T when the mix outputs are off by at most e: a feature is then off by expm1(2 e) of itself, a key
    by 2^-11 more (its fp16 rounding, 2^-12, and the fp32 exponents of its decay), or by 2^-25 where it is an fp16 subnormal."""
    a = dict(x, v=np.abs(x["v"]))
    if "S0" in a:
        a["S0"] = np.abs(a["S0"])
    r = oracle(s, a)
    rel = np.expm1(2 * e) + 2.0 ** -11
    return rel * r["S_T"] + 2.0 ** -25 * s.T * np.abs(x["v"]).max(), rel * r["z_T"] + 2.0 ** -25 * s.T


@pytest.mark.parametrize("d,H,Hkv,gate_dim", SHAPES)
def test_rows_that_need_their_maximum(d, H, Hkv, gate_dim):
    """Keys with 200 or -200 in one of two channels whose rows of W are +1 throughout, and +1 in one half, -1 in the other. The taps pass
    the current token on, so conv output and W are exact in 16 bits and y is off only by its fp32 sum of d exact products: by at most
    2^-16 of the sum of their magnitudes."""
    import torch
    s = I.LayerShape(1, 1300, H, Hkv, d, d, gate_dim=gate_dim or d, dtype="bf16", config_id=95)
    x = I.make(s, NAMES)
    x["w_k"][:] = np.array([1.0, 0.0, 0.0, 0.0], np.float32)
    x["W"][:, 0, :] = 1.0
    x["W"][:, 1, :d // 2], x["W"][:, 1, d // 2:] = 1.0, -1.0
    t = np.arange(s.T)
    x["k"][:, t % 7 == 1, :, 0] = -200.0
    x["k"][:, t % 7 == 3, :, 0] = 200.0
    x["k"][:, t % 7 == 5, :, 1] = 200.0
    y, mag = mix_of_keys(s, x)
    early = y[:, :s.T - SEG]
    parts = early.reshape(1, s.T - SEG, H, d // 32, 32).max(-1)
    assert (early.max(-1) > 89).mean() > 0.2                                    # overflow without the row's maximum
    assert (early.max(-1) < -104).mean() > 0.1                                  # nothing but zeros without it
    assert ((parts.max(-1) > 89) & (parts.min(-1) < 0)).mean() > 0.1           # warps whose part of the row is all negative
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    r, kernels = layer(s, x, status)
    assert "layer_tc_state" in kernels and int(status.item()) == 0
    ref = oracle(s, x)
    bS, bz = state_bound(s, x, 2.0 ** -16 * mag.max())
    assert (np.abs(r["S_T"] - ref["S_T"]) <= bS).all() and (np.abs(r["z_T"] - ref["z_T"]) <= bz).all()
    assert np.isfinite(r["o"]).all()
    assert np.linalg.norm(r["o"] - ref["o"]) <= (2.0 ** -8 + 2 * np.expm1(2.0 ** -15 * mag.max())) * np.linalg.norm(ref["o"])


@pytest.mark.parametrize("tau", [16.0, 1.0])
@pytest.mark.parametrize("d,H,Hkv,gate_dim", SHAPES[:4])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_key_that_is_not_finite(d, H, Hkv, gate_dim, bad, tau):
    """One entry of one key: from its token on nothing of its heads is finite, and nothing else is touched. (tau = 1: features from conv
    + mix in fp32, and the exact recurrence; rows of an infinite key's tile are then formed with their maximum taken off.)"""
    s = I.LayerShape(1, 1300, H, Hkv, d, d, gate_dim=gate_dim or d, gate_tau=tau, dtype="bf16", config_id=96)
    x = I.make(s, NAMES)
    clean, kernels = layer(s, x)
    assert ("layer_tc_state" if tau == 16.0 else "gla_fwd_rec_state") in kernels and ("convmix_tc_fwd" in kernels) == (tau == 1.0)
    t0, j, G = SEG + 70, Hkv - 1, H // Hkv
    x["k"][0, t0, j, 5] = bad
    r, _ = layer(s, x)
    ref = oracle(s, x)
    hit = np.arange(H) // G == j
    for n in ("o", "S_T", "z_T"):
        assert (np.isfinite(r[n]) == np.isfinite(ref[n])).all(), n
    assert not np.isfinite(r["o"][:, t0:, hit]).any() and not np.isfinite(r["S_T"][:, hit]).any() and not np.isfinite(r["z_T"][:, hit]).any()
    same = np.array_equal if tau == 16.0 or np.isnan(bad) else lambda a, b: np.allclose(a, b, rtol=2.0 ** -7, atol=2.0 ** -7)
    assert same(r["o"][:, :t0], clean["o"][:, :t0]) and same(r["o"][:, :, ~hit], clean["o"][:, :, ~hit])
    for n in ("S_T", "z_T"):
        assert same(r[n][:, ~hit], clean[n][:, ~hit]), n


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_conv_and_mix_of_a_row_that_is_not_finite(d, bad):
    """The rows that the conv spreads it over, of the heads that it belongs to; the other rows are as they were, but for the maximum that
    an infinite row's tile takes off: the bounds of the ordinary test."""
    from paper_2509_18467_b200 import api
    s = I.LayerShape(1, 300, 4, 2, d, d, dtype="bf16", config_id=97)
    names = ["q", "k", "w_q", "w_k", "W"]
    x = I.make(s, names)

    def run():
        return [v.float().cpu().numpy() for v in
                api.lawcat_conv_fwd(api.params(1, 300, 4, 2, d, d), *[api.to_device(x[n], "bf16") for n in names])]

    cq, ck = run()
    x["k"][0, 140, 1, 3] = x["q"][0, 7, 2, 9] = bad
    q, k = run()
    bq, bk = np.zeros(q.shape, bool), np.zeros(k.shape, bool)
    bq[0, 7:11, 2], bk[0, 140:144, 2:4] = True, True
    for got, was, out in ((q, cq, bq), (k, ck, bk)):
        assert not np.isfinite(got[out]).any() and np.isfinite(got[~out]).all()
        if np.isnan(bad):
            assert np.array_equal(got[~out], was[~out])
        else:
            assert np.allclose(got[~out], was[~out], rtol=2.0 ** -7, atol=0.0)


@pytest.mark.parametrize("d,H,Hkv,gate_dim", SHAPES)
def test_a_decay_of_zero_clears_the_state(d, H, Hkv, gate_dim):
    """Logits of -inf (and +inf: no decay at all) in the first segment. The chunks around them run with clamped exponents, which the
    status reports; the state behind them, which the other segments start from, holds to its ordinary bounds."""
    import torch
    s = I.LayerShape(1, 1300, H, Hkv, d, d, gate_dim=gate_dim or d, dtype="bf16", config_id=99)
    x = I.make(s, NAMES + ["S0", "z0"])
    x["gate"][:, [100, 230, 231]] = -np.inf
    x["gate"][:, [40, 150, 300, 600, 1299]] = np.inf
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    r, kernels = layer(s, x, status)
    assert "layer_tc_state" in kernels and int(status.item()) == 6  # LAWCAT_ERR_NUMERIC
    ref = oracle(s, x)
    assert all(np.isfinite(v).all() for v in r.values())
    _, mag = mix_of_keys(s, x)
    bS, bz = state_bound(s, x, 2.0 ** -11 * mag.max())
    assert (np.abs(r["S_T"] - ref["S_T"]) <= bS).all() and (np.abs(r["z_T"] - ref["z_T"]) <= bz).all()
    err = np.linalg.norm(r["o"][:, SEG:] - ref["o"][:, SEG:])
    assert err <= (2.0 ** -8 + 2 * np.expm1(2.0 ** -10 * mag.max())) * np.linalg.norm(ref["o"][:, SEG:])


@pytest.mark.parametrize("d,H,Hkv,gate_dim", SHAPES)
def test_a_batch_whose_sequences_are_cut(d, H, Hkv, gate_dim):
    import torch
    s = I.LayerShape(2, 1300, H, Hkv, d, d, gate_dim=gate_dim or d, dtype="bf16", config_id=100)
    x = I.make(s, NAMES + ["S0", "z0", "cache_q", "cache_k"])
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    r, kernels = layer(s, x, status)
    assert "layer_tc_state" in kernels and int(status.item()) == 0
    ref = oracle(s, x)
    _, mag = mix_of_keys(s, x)
    bS, bz = state_bound(s, x, 2.0 ** -11 * mag.max())
    assert (np.abs(r["S_T"] - ref["S_T"]) <= bS).all() and (np.abs(r["z_T"] - ref["z_T"]) <= bz).all()
    for b in range(2):
        err = np.linalg.norm(r["o"][b] - ref["o"][b])
        assert err <= (2.0 ** -8 + 2 * np.expm1(2.0 ** -10 * mag.max())) * np.linalg.norm(ref["o"][b])
