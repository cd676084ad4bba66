"""The mix backward walks the heads of a group in one block, or in two where that fills the GPU better: on 148 SMs one block per group
takes calls of 75 to 148 (sequence, key/value head, tile of 128 tokens) at width 128 and of 149 to 296 at width 64, smaller ones two.
Every gradient of the layer against the fp64 oracle at sizes of either kind."""
import numpy as np
import pytest

from helpers import check
from paper_2509_18467_b200 import inputs as I
from test_layer_bwd import NAMES, P, oracle_layer_gradients, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2509_18467_b200 import api as A
    return A


@pytest.mark.parametrize("d,B,T,G", [(128, 10, 20, 2), (128, 5, 150, 3), (128, 10, 33, 4), (64, 20, 20, 2), (64, 10, 150, 3), (64, 20, 33, 4)])
def test_one_block_walks_a_group(api, d, B, T, G):
    run(api, I.LayerShape(B, T, 8 * G, 8, d, d, dtype="bf16", config_id=101), False, True)


@pytest.mark.parametrize("d,B,Hkv", [(128, 10, 8), (64, 20, 8), (128, 1, 1), (64, 1, 1)])
def test_scales_that_rise_and_fall_along_a_group(api, d, B, Hkv):
    """Eight heads a group, in one block or as four and four, whose upstream gradients go up and down by up to 2^30 from head to head: the
    key stream's du is rescaled in place several times, by steps of either sign."""
    s = I.LayerShape(B, 24, 8 * Hkv, Hkv, d, d, dtype="bf16", config_id=102)
    x = I.make(s, NAMES + ["dO"])
    f = np.float32([2.0 ** -14, 2.0 ** -30, 1.0, 2.0 ** -26, 2.0 ** -6, 2.0 ** -13, 2.0 ** -29, 2.0 ** -3])
    x["dO"] = x["dO"] * np.tile(f, Hkv)[:, None]
    t = {n: api.to_device(v, s.dtype) for n, v in x.items()}
    g = api.lawcat_layer_bwd(P(api, s), *[t[n] for n in NAMES], t["dO"])
    ref = oracle_layer_gradients(s, x)
    for h in range(8):  # (all groups' heads of one scale together)
        for n in ("dq", "dgate"):
            check(g[n][:, :, h::8], ref[n][:, :, h::8], "bf16", f"{n} of heads {h}")
        check(g["dW"][h::8], ref["dW"][h::8], "bf16", f"dW of heads {h}", f32_store=True)
    for n in ("dk", "dv"):
        check(g[n], ref[n], "bf16", n)
    for n in ("dw_q", "dw_k"):
        check(g[n], ref[n], "bf16", n, f32_store=True)
