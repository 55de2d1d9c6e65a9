"""The size of the training cluster (sp_model_train) where a device takes none
of 16 CTAs, or none at all: training goes on with what fits and reports no
error of the query."""
import ctypes

import numpy as np
import pytest

import fake_cuda
from paper_1011_4046_gb300 import sp


@pytest.mark.parametrize("refused", [0, 16, 8])
def test_refused_cluster_size_is_no_error(refused):
    lib = fake_cuda.load()
    lib.fake_reset(1 << 30, 0, refused)
    m = ctypes.c_void_p()
    assert lib.sp_model_create(3, None, ctypes.byref(m)) == sp.SP_OK
    n = 64
    x, y = np.zeros((n, sp.SP_MODEL_FEATURES), np.float32), np.zeros(n, np.float32)
    try:
        for _ in range(2):
            assert lib.sp_model_train(m, x.ctypes.data, y.ctypes.data, n, 1, 16, 1e-3, 0, None, None) == sp.SP_OK
    finally:
        lib.sp_model_destroy(m)
