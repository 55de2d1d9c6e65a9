"""Diagnostics of grids narrower than a warp (diag_flat, csrc/sp_diag.cu), whose
planes go to the threads site by site: widths that divide a warp and do not,
planes that end inside a block, on the fields of test_gpu_diag.py."""
import pytest

torch = pytest.importorskip("torch")

import test_gpu_diag as diag  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(4, 67, 9), (31, 33, 6), (16, 16, 70), (32, 20, 8)])
@pytest.mark.parametrize("kind", ["normal", "ties", "mixed", "tiny"])
def test_narrow_grids(kind, n):
    diag.test_diagnostics_equal_fp64(kind, n)
