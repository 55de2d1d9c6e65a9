"""Split-tiling regions handed out in ticket order (static order, bases 4 to 16),
several per CTA with 64 or 128 workers: bit-exact with the sweep at grids on
both sides of every default worker count of base 8, at the smallest grids a base
takes, for a batch whose simulations differ in size and era, over repeated
calls, and for two handles whose launches share the GPU."""
import pytest

torch = pytest.importorskip("torch")

from paper_1011_4046_gb300 import sp  # noqa: E402

pytestmark = pytest.mark.gpu


def _state(n, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    theta = torch.rand((n[2], n[1], n[0]), generator=gen, device="cuda") * 6.2831853
    return torch.polar(torch.ones_like(theta), theta), torch.zeros(theta.shape + (2,), dtype=torch.complex64, device="cuda")


def _run(sims, steps, B, mono, threads=0, handles=1):
    """Final states (bits) of the simulations (n, nu), and the plan."""
    params = [sp.make_params(n, nu=nu, tau0=10.0 if nu else 1.0, tau_ref=(10.0 if nu else 1.0) + 0.25 * steps) for n, nu in sims]
    states = [[_state(n, i) for i, (n, _) in enumerate(sims)] for _ in range(handles)]
    torch.cuda.synchronize()
    grids = [sp.Grid(params, states=s, stream=torch.cuda.Stream()) for s in states]
    info = None
    try:
        if not mono:
            for g in grids:
                g.plan(base_B=B, threads=threads)
            info = grids[0].plan_info(0)
        for _ in range(2):  # the second call's flags are of another epoch
            for g in grids:
                g.evolve(steps, sp.SP_MONOLITHIC if mono else 0)
        torch.cuda.synchronize()
    finally:
        for g in grids:
            g.close()
    return [[torch.view_as_real(t).view(torch.int32) for st in s for t in st] for s in states], info


CASES = [
    ([((16, 16, 16), 2.0)], 8, 0, 256),
    ([((32, 24, 48), 2.0)], 8, 0, 256),  # 72 regions of a type, 256 workers up to 76
    ([((40, 32, 32), 2.0)], 8, 0, 128),  # 80
    ([((72, 72, 72), 2.0)], 8, 0, 128),  # 729, 128 workers up to 760
    ([((80, 80, 64), 2.0)], 8, 0, 64),  # 800: eight regions at a time on an SM
    ([((32, 32, 32), 2.0)], 16, 0, 480),
    ([((48, 32, 80), 0.0)], 16, 256, 256),
    ([((8, 12, 16), 2.0)], 4, 0, 64),
    ([((24, 16, 40), 2.0)], 4, 128, 128),
    ([((48, 16, 24), 2.0), ((16, 16, 16), 0.0), ((24, 56, 32), 1.0), ((16, 32, 24), 2.0)], 8, 0, 128),
    ([((32, 64, 48), 1.0), ((32, 32, 32), 2.0), ((64, 48, 32), 0.0)], 16, 0, 480),
]


@pytest.mark.parametrize("sims, B, threads, workers", CASES)
def test_ticket_order(sims, B, threads, workers):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    got, info = _run(sims, 21, B, False, threads)
    assert info["base_B"] == B and info["threads"] == workers
    want, _ = _run(sims, 21, B, True)
    assert all(torch.equal(a, b) for a, b in zip(got[0], want[0]))


def test_two_handles_at_once():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sims = [((64, 64, 64), 2.0)]
    got, _ = _run(sims, 64, 8, False, threads=64, handles=3)
    want, _ = _run(sims, 64, 8, True)
    assert all(torch.equal(a, b) for run in got for a, b in zip(run, want[0]))
