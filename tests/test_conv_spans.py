"""The conv's backward walks spans of 16 to 64 tokens, by a rule on the size of the call, in two forms of the kernel. Against the fp64
oracle at sizes that the rule gives spans of 16, 24, 32 (known to the compiler) and 32, 48, 56, 64 tokens on 148 SMs, with ragged last
spans and conv caches in front."""
import pytest

from helpers import check
from oracle import lawcat_oracle as O
from paper_2509_18467_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T", [(1, 703), (1, 1001), (3, 501), (3, 821), (3, 1303), (3, 1500), (4, 1300)])
def test_spans(B, T):
    from paper_2509_18467_b200 import api
    s = I.LayerShape(B, T, 32, 8, 64, 64, dtype="bf16", config_id=75)
    names = ["q", "k", "w_q", "w_k", "W", "d_qdot", "d_kdot", "cache_q", "cache_k"]
    x = I.make(s, names)
    d = {n: api.to_device(v, "bf16") for n, v in x.items()}
    api.trace_begin()
    g = api.lawcat_conv_bwd(api.params(B, T, 32, 8, 64, 64), *[d[n] for n in names])
    assert "conv_bwd4" in api.trace_end()
    ref = O.conv_bwd(O.OracleParams(B, T, 32, 8, 64, 64), *[x[n] for n in names])
    for n in ("dq", "dk"):
        check(g[n], ref[n], "bf16", n)
    for n in ("dw_q", "dw_k", "dW"):
        check(g[n], ref[n], "bf16", n, f32_store=True)
