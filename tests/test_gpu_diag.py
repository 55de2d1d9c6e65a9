"""Energy terms and windings (csrc/sp_diag.cu) against plain numpy in extended
precision (in FP64 the potential of a vacuum field is itself 1e-10 off, from
the cancellation in |phi|^2 - eta^2), on fields where the FP32 words and edge
tests can go wrong: values that tie on every edge, zeros, values so small or
large that FP32 squares leave their range, infinities and NaN, and grids whose
chunks of planes and blocks end unevenly.  The tolerance is the bound of two
FP64 sums in different orders (accuracy_bars.energy_tol); windings are equal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from accuracy_bars import energy_tol  # noqa: E402
from paper_1011_4046_gb300 import sp  # noqa: E402

pytestmark = pytest.mark.gpu


def _field(kind, n, seed):
    r = np.random.RandomState(seed)
    shape = (n[2], n[1], n[0])
    z = (r.randn(*shape) + 1j * r.randn(*shape)).astype(np.complex64)
    if kind == "ties":
        z = (r.randint(-1, 2, shape) + 1j * r.randint(-1, 2, shape)).astype(np.complex64)
        z[r.rand(*shape) < 0.2] *= -1.0  # signed zeros
    elif kind == "tiny":
        z *= np.float32(1e-22)
    elif kind == "mixed":  # a few columns out of range, the others not
        z[:, :2, :3] *= np.float32(3e-25)
        z[:, 3, 1] *= np.float32(1e21)
    elif kind == "vacuum":
        z /= np.abs(z)
    return z


def _reference(phi, pi, eta2, half):
    f, v = phi.astype(np.clongdouble), pi.astype(np.clongdouble)
    with np.errstate(all="ignore"):
        kin = np.sum(v.real ** 2 + v.imag ** 2)
        grad = sum(np.sum((np.roll(f.real, -1, ax) - f.real) ** 2 + (np.roll(f.imag, -1, ax) - f.imag) ** 2)
                   for ax in range(3))
        pot = half * np.sum((f.real ** 2 + f.imag ** 2 - eta2) ** 2)

        def crossing(u, v):
            cr = u.real * v.imag - u.imag * v.real
            ua, va = u.imag >= 0, v.imag >= 0
            return (~ua & va & (cr >= 0)).astype(np.int64) - (ua & ~va & (cr <= 0)).astype(np.int64)

        w = []
        for k in range(3):
            a, b = 2 - (k + 1) % 3, 2 - (k + 2) % 3
            p1 = np.roll(f, -1, a)
            p2, p3 = np.roll(p1, -1, b), np.roll(f, -1, b)
            w.append(crossing(f, p1) + crossing(p1, p2) + crossing(p2, p3) + crossing(p3, f))
    return kin, grad, pot, np.stack(w)


@pytest.mark.parametrize("n", [(4, 4, 4), (33, 9, 5), (70, 17, 131), (8, 100, 300)])
@pytest.mark.parametrize("kind", ["normal", "ties", "tiny", "mixed", "vacuum", "zero", "inf", "nan"])
def test_diagnostics_equal_fp64(kind, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    phi, pi = _field(kind, n, 1), _field(kind, n, 2)
    if kind == "zero":
        phi, pi = np.zeros_like(phi), np.zeros_like(pi)
    elif kind in ("inf", "nan"):
        phi[1, 2, 3] = np.inf if kind == "inf" else np.nan
        pi[0, 1, 2] = 1e30
    p = sp.make_params(n, lam=2.0, eta=1.0, nu=0.0)
    g = sp.Grid([p])
    try:
        g.write_state(0, phi, pi, np.zeros_like(pi))
        d, w = g.diag(0), g.winding(0)
    finally:
        g.close()
    kin, grad, pot, ref = _reference(phi, pi, 1.0, 1.0)
    assert np.array_equal(w, ref)
    assert d["pierced"] == [int((ref[k] != 0).sum()) for k in range(3)]
    assert d["net_winding"] == [int(ref[k].sum()) for k in range(3)]
    assert d["abs_winding"] == int(np.abs(ref).sum())
    tol = energy_tol(phi.size)
    for got, want in ((d["kinetic"], kin), (d["gradient"], grad), (d["potential"], pot)):
        assert np.isclose(got, float(want), rtol=tol, atol=0.0, equal_nan=True) or got == want, (kind, got, want)
