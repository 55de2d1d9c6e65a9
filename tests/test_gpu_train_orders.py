"""Training on orders made by the library against the same orders passed in,
over more epochs and longer orders (copies above 64 KB) than test_gpu_train.py:
equal bit for bit, as the copies of each epoch's order are the only difference."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1011_4046_gb300 import inputs, sp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [512, 8192])  # the one-cluster kernel, launches per step
def test_library_orders_equal_passed_orders(batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, epochs = 40001, 4
    r = np.random.RandomState(2)
    x = r.rand(n, 16).astype(np.float32)
    y = (1.0 + x[:, 2] - x[:, 5] * x[:, 9]).astype(np.float32)
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    out = []
    for order in (None, inputs.epoch_orders(11, n, epochs)):
        m = sp.Model(seed=1)
        try:
            losses = m.train(xd.data_ptr(), yd.data_ptr(), n, epochs=epochs, batch=batch, lr=1e-3, order_seed=11, order=order)
            out.append((losses, *m.params()))
        finally:
            m.close()
    for a, b in zip(*out):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
