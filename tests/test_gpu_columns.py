"""The two-level sweep pass (csrc/sp_columns.cu) against one level at a time.

A whole-grid call of four or more steps on a grid beyond L2 takes its levels
two at a time; a call of one step never does.  The same steps made by one call
and by one-step calls must agree bit for bit, at the sizes where the pass can
go wrong: tiles and halos wider than the grid, odd rows (no aligned pairs of
sites), chunks of few planes, an odd number of level pairs or steps, and a
state whose phi is not 16-byte aligned.
"""
import pytest

torch = pytest.importorskip("torch")

from paper_1011_4046_gb300 import sp  # noqa: E402

pytestmark = pytest.mark.gpu


def _state(n, seed, offset=0):
    """Random-phase phi and small velocities and carries; phi starts ``offset``
    sites into its allocation."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    sites = n[0] * n[1] * n[2]
    theta = torch.rand(sites, generator=gen, device="cuda") * 6.2831853
    phi = torch.empty(sites + offset, dtype=torch.complex64, device="cuda")[offset:]
    phi.copy_(torch.polar(torch.ones_like(theta), theta))
    pic = torch.view_as_complex(torch.randn(sites, 2, 2, generator=gen, device="cuda") * torch.tensor(
        [[[0.1], [1e-8]]], device="cuda"))
    return phi, pic.contiguous()


@pytest.mark.parametrize("n, steps, damp, offset", [
    ((144, 144, 144), 8, 0, 0),       # whole tiles and chunks
    ((151, 145, 131), 4, 0, 0),       # odd rows
    ((150, 145, 131), 7, 3, 1),       # phi off 16-byte alignment, odd steps, damped levels
    ((16, 400, 400), 6, 0, 0),        # rows narrower than a tile: its halo wraps several times
    ((1024, 5, 500), 5, 0, 0),        # fewer rows than a tile
    ((1250, 511, 4), 9, 0, 0),        # fewer planes than the halo of a chunk
])
def test_level_pairs_equal_single_levels(n, steps, damp, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = sp.make_params(n, dx=1.0, dt=0.25, lam=2.0, eta=1.0, nu=2.0, tau0=10.0, tau_ref=10.0 + steps * 0.25,
                       damp_steps=damp)
    assert n[0] * n[1] * n[2] >= 2500000
    runs = []
    for calls in ([steps], [1] * steps, [4] + [1] * (steps - 4)):
        phi, pic = _state(n, 3, offset)
        assert phi.data_ptr() % 16 == 8 * (offset % 2)
        g = sp.Grid([p], states=[(phi, pic)], stream=torch.cuda.Stream())
        torch.cuda.synchronize()
        try:
            for k in calls:
                g.evolve(k, sp.SP_MONOLITHIC)
            assert g.level(0) == steps
        finally:
            g.close()
        runs.append((torch.view_as_real(phi).view(torch.int32), torch.view_as_real(pic).view(torch.int32)))
    assert torch.isfinite(torch.view_as_real(phi)).all()
    for phi, pic in runs[1:]:
        assert torch.equal(phi, runs[0][0]), "phi differs"
        assert torch.equal(pic, runs[0][1]), "(pi, c) differ"
