"""Lattice regions on a state whose phi starts on 8 bytes but not on 16 (the
library asks for 8): imports then take no 16-byte site pairs.  Bit-exact with
the sweep, as on an aligned state, for a size whose imports come as slot pairs
and one whose do not."""
import pytest

torch = pytest.importorskip("torch")

from paper_1011_4046_gb300 import sp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, n", [(16, (32, 48, 16)), (8, (16, 24, 8)), (24, (24, 24, 48))])
def test_phi_off_16_byte_alignment(B, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    steps, sites = 37, n[0] * n[1] * n[2]
    p = sp.make_params(n, nu=2.0, tau0=10.0, tau_ref=10.0 + steps * 0.25)
    runs = []
    for offset, mono in ((1, False), (0, False), (0, True)):
        gen = torch.Generator(device="cuda").manual_seed(9)
        theta = torch.rand(sites, generator=gen, device="cuda") * 6.2831853
        phi = torch.empty(sites + offset, dtype=torch.complex64, device="cuda")[offset:]
        phi.copy_(torch.polar(torch.ones_like(theta), theta))
        pic = torch.zeros(sites, 2, dtype=torch.complex64, device="cuda")
        assert phi.data_ptr() % 16 == 8 * offset
        torch.cuda.synchronize()
        g = sp.Grid([p], states=[(phi, pic)], stream=torch.cuda.Stream())
        try:
            if not mono:
                g.plan(base_B=B, shape=sp.SP_SHAPE_LATTICE)
            g.evolve(steps, sp.SP_MONOLITHIC if mono else 0)
        finally:
            g.close()
        runs.append([torch.view_as_real(t).view(torch.int32) for t in (phi, pic)])
    for run in runs[:2]:
        assert torch.equal(run[0], runs[2][0]) and torch.equal(run[1], runs[2][1])
