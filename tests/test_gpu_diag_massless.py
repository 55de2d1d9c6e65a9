"""Potential energy without a vacuum value (eta = 0, csrc/sp_diag.cu): fields
whose squares fall below the FP32 range still have a fourth power in FP64, and
only a field that is zero gives zero (also a uniform field, which has no other
energy).  The reference and the bound are those of
test_gpu_diag.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import test_gpu_diag as diag  # noqa: E402
from accuracy_bars import energy_tol  # noqa: E402
from paper_1011_4046_gb300 import sp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(4, 4, 4), (33, 9, 5), (70, 17, 131)])
@pytest.mark.parametrize("kind, scale", [("normal", 1.0), ("ties", 1.0), ("tiny", 1.0), ("tiny", 1e-2), ("tiny", 1e-18),
                                         ("mixed", 1.0), ("mixed", 1e-20), ("normal", 0.0),
                                         ("uniform", 1.0), ("uniform", 1e-12), ("uniform", 1e-23), ("uniform", 1e-40)])
def test_potential_without_vacuum_value(kind, scale, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    phi = diag._field(kind, n, 1) * np.float32(scale)
    if kind == "uniform":
        phi[:] = np.complex64(0.75 - 2.0j) * np.float32(scale)
    pi = np.zeros_like(phi)
    g = sp.Grid([sp.make_params(n, lam=2.0, eta=0.0, nu=0.0)])
    try:
        g.write_state(0, phi, pi, pi)
        d = g.diag(0)
    finally:
        g.close()
    kin, grad, pot, _ = diag._reference(phi, pi, 0.0, 1.0)
    assert (pot > 0) == (scale > 0)
    for got, want in ((d["kinetic"], kin), (d["gradient"], grad), (d["potential"], pot)):
        assert np.isclose(got, float(want), rtol=energy_tol(phi.size), atol=0.0), (kind, got, want)
