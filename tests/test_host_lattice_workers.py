"""Default workers of a lattice launch (plan_lattice, csrc/sp_api.cu) by the
regions that its own simulations have in a layer, whatever else the batch
holds: edges 8 and 12 take 128 where a layer has few regions (up to 6 and 11
per SM), else 64."""
import ctypes

import pytest

import fake_cuda
from paper_1011_4046_gb300 import sp


@pytest.mark.parametrize("sides, workers, base", [
    ([24], {8: 128}, 0), ([128 + 8], {8: 64}, 0), ([24] * 3 + [128] * 4, {8: 128, 16: 128}, 0), ([24] * 41, {8: 64}, 0),
    ([136] + [32] * 2, {8: 64, 16: 128}, 0), ([48], {8: 128}, 8), ([56], {8: 64}, 8), ([84], {12: 128}, 12),
    ([96], {12: 64}, 12), ([160], {20: 256}, 20), ([32], {16: 128}, 16), ([8], {4: 64}, 4),
])
def test_workers_by_the_launch_of_each_edge(sides, workers, base):
    lib = fake_cuda.load()
    lib.fake_reset(1 << 40, 0, 0)
    before = lib.fake_used()
    params = (sp.sp_params * len(sides))(*[sp.make_params(n) for n in sides])
    h = ctypes.c_void_p()
    assert lib.sp_grid_create(params, len(sides), None, 16, ctypes.byref(h)) == sp.SP_OK
    try:
        assert lib.sp_set_option(h, sp.SP_OPT_REGION_SHAPE, sp.SP_SHAPE_LATTICE) == sp.SP_OK
        assert lib.sp_region_plan(h, base, 0, 0, None) == sp.SP_OK
        for s, n in enumerate(sides):
            info = sp.sp_plan_info()
            assert lib.sp_read_surface(h, s, sp.SP_SURF_PLAN, ctypes.addressof(info), ctypes.sizeof(info), 0) == sp.SP_OK
            assert info.base_B == (base or (16 if n % 16 == 0 else 8))
            assert info.threads == workers[info.base_B], n
    finally:
        assert lib.sp_destroy(h) == sp.SP_OK
    assert lib.fake_used() == before
