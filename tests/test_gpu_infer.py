"""The cost model's outputs at the sizes where its tiles end: one sample, the
last of a block, one more, the first size of two samples per thread, a ragged
last tile, and samples that are not 16-byte aligned.  An output does not
depend on the size of the call or its place in it, and agrees with the FP64
oracle within FP32 rounding (three layers of at most 65 terms: 200 2^-24 of the
sum of absolute terms)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp  # noqa: E402
from paper_1011_4046_gb300 import inputs, sp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, offset", [(1, 0), (128, 0), (129, 1), (38912, 0), (38913, 0), (78001, 3)])
def test_outputs_at_tile_edges(n, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = np.random.RandomState(n)
    X = r.rand(n, 16).astype(np.float32)
    theta = (inputs.mlp_init(4) + 0.05 * r.randn(5313)).astype(np.float32)
    buf = torch.zeros(16 * n + offset, device="cuda")
    xd = buf[offset:]
    xd.copy_(torch.from_numpy(X).reshape(-1))
    out = torch.full((n + 1,), 7.0, device="cuda")
    m = sp.Model()
    try:
        m.set_params(theta)
        m.predict(xd.data_ptr(), n, out.data_ptr())
        one = torch.empty(1, device="cuda")
        for k in {0, n // 2, n - 1}:  # alone, through the one-sample tile
            m.predict(xd.data_ptr() + 64 * k, 1, one.data_ptr())
            assert torch.equal(one.view(torch.int32), out[k:k + 1].view(torch.int32))
    finally:
        m.close()
    got = out.cpu().numpy()
    assert got[n] == 7.0  # nothing past the last sample
    t = theta.astype(np.float64)
    ref, _ = mlp.forward(t, X.astype(np.float64))
    bound, _ = mlp.forward(np.abs(t), np.abs(X).astype(np.float64))
    assert np.all(np.abs(got[:n] - ref) <= 200 * 2.0 ** -24 * bound)
