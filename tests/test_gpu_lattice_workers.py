"""Worker counts and sizes on both sides of the choice between the two lattice
kernels (lattice_ring_faster, csrc/sp_lattice.cu): each equals the sweep bit
for bit, over two calls of odd step counts."""
import pytest

torch = pytest.importorskip("torch")

import test_gpu_lattice as lattice  # noqa: E402
from paper_1011_4046_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, n, threads", [
    (12, (84, 84, 84), 64), (12, (72, 84, 72), 64),       # many and few regions of a layer
    (16, (48, 32, 64), 64), (20, (40, 60, 40), 64), (20, (40, 40, 60), 128), (20, (60, 40, 40), 192), (16, (32, 48, 32), 192),
])
def test_both_kernels_equal_the_sweep(B, n, threads):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = lattice.params_for(n, 2.0, 24)
    st = inputs.initial_state(n, 4, "phase")
    reg, info = lattice.run(p, st, [17, 7], base_B=B, threads=threads)
    assert info["threads"] == threads and info["base_B"] == B
    lattice.assert_bit_equal(reg, lattice.run(p, st, [17, 7], mono=True)[0])
