"""Sample orders of training (sp_model_train) against copies that are carried
out as late as CUDA allows: the host values that an asynchronous copy reads
have to stand until the stream has been waited for."""
import ctypes

import numpy as np
import pytest

import fake_cuda
from paper_1011_4046_gb300 import inputs, sp


@pytest.fixture(scope="module")
def lib():
    return fake_cuda.load()


@pytest.mark.parametrize("own_orders", [False, True])
@pytest.mark.parametrize("fails", [False, True])
def test_every_epoch_trains_on_its_own_order(lib, own_orders, fails):
    """Four epochs: what arrives on the device for each is that epoch's
    order, made by the library or passed in; also where the call gives up
    after the training (no memory for the predictions), and then before it
    returns."""
    n, epochs, seed = 137, 4, 9
    steps = epochs * -(-n // 16)
    lib.fake_reset(1 << 30, 1, 0)
    m = ctypes.c_void_p()
    assert lib.sp_model_create(3, None, ctypes.byref(m)) == sp.SP_OK
    want = inputs.epoch_orders(seed, n, epochs)
    order = None
    if own_orders:
        flat = np.ascontiguousarray(np.concatenate(want), dtype=np.int32)
        order = flat.ctypes.data_as(ctypes.POINTER(ctypes.c_int32))
    x, y = np.zeros((n, sp.SP_MODEL_FEATURES), np.float32), np.zeros(n, np.float32)
    losses = np.zeros(steps, np.float32)
    if fails:  # room for the orders, losses and bias corrections only
        lib.fake_set_capacity(lib.fake_used() + 4 * n * epochs + 12 * steps)
    try:
        rc = lib.sp_model_train(m, x.ctypes.data, y.ctypes.data, n, epochs, 16, 1e-3, seed, order,
                                losses.ctypes.data_as(ctypes.POINTER(ctypes.c_float)))
        assert rc == (sp.SP_ENOMEM if fails else sp.SP_OK)
        dst = (ctypes.c_void_p * 16)()
        assert lib.fake_copies(4 * n, dst, 16) >= epochs
        got = [np.ctypeslib.as_array(ctypes.cast(dst[e], ctypes.POINTER(ctypes.c_int32)), (n,)).copy()
               for e in range(epochs)]
    finally:
        lib.sp_model_destroy(m)
    for e in range(epochs):
        assert np.array_equal(got[e], want[e]), f"epoch {e}"
