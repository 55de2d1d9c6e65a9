"""Which grids sweep two levels a pass (columns_pay, csrc/sp_columns.cu), seen
by the copy of (pi, c) that such a call takes: grids that leave most of a tile
or of a chunk empty do not (measured 1.3 to 2.7 times slower that way), others
beyond L2 do."""
import ctypes

import pytest

import fake_cuda
from paper_1011_4046_gb300 import sp


@pytest.mark.parametrize("n, pays", [
    ((512, 512, 64), True), ((160, 160, 160), True), ((173, 292, 207), True), ((1024, 1024, 4), True), ((58, 26, 1700), True),
    ((128, 128, 128), False),   # on L2
    ((1024, 4, 1024), False), ((4, 1024, 1024), False), ((4, 16384, 64), False), ((64, 16384, 4), False),
    ((16, 512, 512), False), ((20, 512, 512), False), ((17, 343, 494), False), ((137, 137, 137), False),
    ((61, 27, 2048), False), ((27, 2048, 61), False),  # just over a tile's width or rows
])
def test_shapes_that_take_level_pairs(n, pays):
    lib = fake_cuda.load()
    sites = n[0] * n[1] * n[2]
    lib.fake_reset(1 << 40, 0, 0)
    before = lib.fake_used()
    h = ctypes.c_void_p()
    p = sp.make_params(n, nu=2.0, tau0=10.0, tau_ref=20.0)
    assert lib.sp_grid_create(ctypes.byref(p), 1, None, 16, ctypes.byref(h)) == sp.SP_OK
    try:
        assert lib.sp_evolve(h, 4, sp.SP_MONOLITHIC) == sp.SP_OK
        assert (lib.fake_used() - before > (24 + 8 + 15) * sites) == pays
    finally:
        assert lib.sp_destroy(h) == sp.SP_OK
