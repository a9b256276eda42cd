"""A bounded wait that expired in a call that only enqueues work (als_sweep_async, a batch sweep,
an MTTKRP into device memory) is reported by the next call that waits for the handle's stream,
whichever that is, once, and not by a later call as its own."""
import ctypes as ct

import numpy as np
import pytest

from paper_2112_03985_gb300 import _lib, api

pytestmark = pytest.mark.gpu

DIMS, RANKS = (40, 33, 61), [5] * 41

WAITING = {
    "sync": lambda h: h.sync(),
    "get_factors": lambda h: h.get_factors(),
    "set_factors": lambda h: h.set_factors([np.ones((I, sum(RANKS))) for I in DIMS]),
    "block_status": lambda h: h.block_status(),
    "loss_history": lambda h: h.loss_history(1),
    "jackknife_se": lambda h: h.jackknife_se(ref_block=0),
    "als_sweep": lambda h: h.als_sweep(1),
    "grad": lambda h: h.grad(),
    "mttkrp": lambda h: h.mttkrp(0),
    "run": lambda h: h.run(1),
}


def _handle(**kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(1)
    left = [[p] for p in range(40)] + [[]]
    return api.JKCALS(rng.random(DIMS), 0, RANKS, left, [rng.random((I, sum(RANKS))) for I in DIMS], **kw)


@pytest.mark.parametrize("precision", ["fp64", "exact_bf16"])
@pytest.mark.parametrize("call", WAITING)
def test_reported_once_by_the_next_call_that_waits(call, precision):
    lib = _lib.load()
    with _handle(precision=precision) as h:
        h.als_sweep_async(1)
        h.sync()
        assert lib.jkcals_selftest_expired_wait(h._h, 5) == 0
        with pytest.raises(Exception, match="code 5"):
            WAITING[call](h)
        WAITING[call](h)
        h.sync()


def test_arguments():
    lib = _lib.load()
    with _handle(precision="exact_bf16") as h:
        assert lib.jkcals_selftest_expired_wait(h._h, 0) == 1       # ERR_ARG
    with _handle(max_device_bytes=1 << 46) as h:                    # FP64 on the CUDA cores
        assert lib.jkcals_selftest_expired_wait(h._h, 5) == 6       # ERR_STATE
        h.sync()
    assert lib.jkcals_selftest_expired_wait(ct.c_void_p(None), 5) == 1
