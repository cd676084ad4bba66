"""The native module that turns tensors into the pointers of a C entry point: what is not a tensor is a Python error, and other
Python threads run while the library does (no GPU: nothing is launched there); scratch of a call on a stream of its own."""
import ctypes
import threading
import time

import pytest

from paper_2509_18467_b200 import api, build


@pytest.fixture(scope="module")
def binding():
    build.build()
    return api._bind()


ARGS = [None] * 12   # of a decode step, all NULL: refused by the library before anything is launched


def call(b, args=ARGS, ws=None, dev_status=None, nint=None):
    p = api.params(1, 1, 4, 2, 64, 64)
    extra = () if nint is None else (nint,)
    return b.call(api._addr["lawcat_decode_step"], ctypes.addressof(p), 0, -1, tuple(args), ws, None, dev_status, *extra)


def test_null_tensors_reach_the_library(binding):
    assert call(binding) == 1   # LAWCAT_ERR_INVALID_ARG


@pytest.mark.parametrize("bad", [16, 0, True, 1.5, "ws", [0]])
@pytest.mark.parametrize("where", ["ws", "dev_status", "first", "last"])
def test_what_is_not_a_tensor_is_a_python_error(binding, bad, where):
    args = list(ARGS)
    kw = {}
    if where in ("ws", "dev_status"):
        kw[where] = bad
    else:
        args[0 if where == "first" else -1] = bad
    with pytest.raises(TypeError):
        call(binding, args, **kw)


@pytest.mark.parametrize("nint", [-1, 13, "2"])
def test_number_of_leading_integers(binding, nint):
    with pytest.raises(TypeError):
        call(binding, nint=nint)
    with pytest.raises(TypeError):
        call(binding, [None] * 12, nint=1)   # (an integer is expected in front)


def test_other_threads_run_during_a_call(binding):
    """usleep stands in for an entry point that waits for room in the launch queue (it reads its first argument only)."""
    usleep = ctypes.cast(ctypes.CDLL(None).usleep, ctypes.c_void_p).value
    stamps, stop = [], threading.Event()

    def tick():
        while not stop.is_set():
            stamps.append(time.perf_counter())
            time.sleep(0.005)

    t = threading.Thread(target=tick)
    t.start()
    try:
        time.sleep(0.05)
        t0 = time.perf_counter()
        assert binding.call(usleep, 500_000, 0, -1, (None,), None, None, None) == 0
        t1 = time.perf_counter()
    finally:
        stop.set()
        t.join()
    assert t1 - t0 >= 0.5
    assert sum(t0 + 0.02 < s < t1 - 0.02 for s in stamps) >= 10


@pytest.mark.gpu
def test_scratch_of_a_call_on_another_stream_is_not_handed_on_early():
    """The call's kernels wait behind a delay on a side stream while the current stream allocates and fills blocks of the
    scratch's size: the result is that of a call on the current stream."""
    import torch
    from paper_2509_18467_b200 import inputs as I
    names = ["q", "k", "v", "gate", "w_q", "w_k", "W"]
    s = I.LayerShape(1, 300, 4, 2, 64, 64, dtype="bf16", gate_tau=1.0, config_id=131)
    t = [api.to_device(v, "bf16") for v in I.make(s, names).values()]
    p = api.params(1, 300, 4, 2, 64, 64, gate_tau=1.0)   # (served by the kernels that keep features in scratch)
    need = api.workspace_bytes(p, api.OP_LAYER_FWD)
    assert need > 0
    ref = api.lawcat_layer_fwd(p, *t)["o"]
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)   # about 10 ms
    r = api.lawcat_layer_fwd(p, *t, stream=side)["o"]
    junk = [torch.full((need,), 255, dtype=torch.uint8, device="cuda") for _ in range(4)]
    torch.cuda.synchronize()
    assert torch.equal(r, ref) and len(junk) == 4
