"""Two-level sweep passes (csrc/sp_columns.cu) at the edges of the shapes that
take them: rows narrower than a tile, fewer rows than a tile, odd rows, as few
planes as a grid can have.  Compared as in test_gpu_columns.py, and that the
call did take passes by the copy of (pi, c) that it holds afterwards."""
import pytest

torch = pytest.importorskip("torch")

import test_gpu_columns as columns  # noqa: E402
from paper_1011_4046_gb300 import sp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(30, 260, 409), (511, 21, 400), (1024, 1024, 4), (173, 292, 207)])
def test_edges_of_the_rule(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sites = n[0] * n[1] * n[2]
    phi, pic = columns._state(n, 1)
    g = sp.Grid([sp.make_params(n, nu=2.0, tau0=10.0, tau_ref=20.0)], states=[(phi, pic)])
    try:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        g.evolve(4, sp.SP_MONOLITHIC)
        assert free - torch.cuda.mem_get_info()[0] > 24 * sites * 9 // 10
    finally:
        g.close()
    columns.test_level_pairs_equal_single_levels(n, 6, 2, 0)
