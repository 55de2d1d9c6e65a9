"""Lattice calls of few steps, which small sizes run on the kernel with a region
per CTA (lattice_ring_brief, csrc/sp_lattice.cu), between longer ones that run on
the resident kernel: both share the layer numbers and done flags of the plan,
and the run equals the sweep bit for bit."""
import pytest

torch = pytest.importorskip("torch")

import test_gpu_lattice as lattice  # noqa: E402
from paper_1011_4046_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [0, 128])
@pytest.mark.parametrize("B, n, calls", [
    (4, (20, 12, 16), [8, 9, 1, 12, 3]), (8, (56, 48, 64), [4, 5, 1, 20, 3]), (8, (16, 24, 16), [1, 6, 3]),
    (12, (48, 60, 36), [16, 17, 1, 30, 12]),
])
def test_short_and_long_calls_equal_the_sweep(B, n, calls, threads):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = lattice.params_for(n, 1.0, sum(calls))
    st = inputs.initial_state(n, 8, "phase")
    reg, info = lattice.run(p, st, calls, base_B=B, threads=threads)
    assert info["base_B"] == B
    lattice.assert_bit_equal(reg, lattice.run(p, st, calls, mono=True)[0])
