"""Minibatch training (csrc/sp_model.cu) where its shares and passes end: fewer
samples than CTAs, one and one more than a pass of sixteen per CTA, several
passes, a ragged last minibatch, and the largest minibatch of the one-cluster
kernel beside the first of the launch-by-launch path.  Compared with the FP64
oracle's run of the same minibatches by the bars of the training test of
test_gpu_model.py; two calls of one epoch equal one call of two."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp  # noqa: E402
from paper_1011_4046_gb300 import inputs, sp  # noqa: E402

pytestmark = pytest.mark.gpu


def _samples(n):
    r = np.random.RandomState(n)
    X = r.rand(n, 16).astype(np.float32)
    return X, (1.0 + X[:, 3] - X[:, 7] * X[:, 1] + 0.1 * r.randn(n)).astype(np.float32)


@pytest.mark.parametrize("n, batch", [(7, 3), (40, 16), (515, 256), (530, 257), (1400, 700), (4100, 4096), (4100, 4097)])
def test_training_steps_match_oracle(n, batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X, y = _samples(n)
    xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    theta = inputs.mlp_init(12)
    order = inputs.epoch_orders(5, n, 2)
    runs = []
    for calls in ([order], [order[:1], order[1:]], None):
        m = sp.Model()
        try:
            m.set_params(theta)
            if calls is None:
                losses = [m.train(xd.data_ptr(), yd.data_ptr(), n, epochs=2, batch=batch, lr=3e-3, order_seed=5)]
            else:
                losses = [m.train(xd.data_ptr(), yd.data_ptr(), n, epochs=len(o), batch=batch, lr=3e-3, order=o)
                          for o in calls]
            runs.append((np.concatenate(losses), m.params()[0]))
        finally:
            m.close()
    for losses, params in runs[1:]:
        assert np.array_equal(losses.view(np.uint32), runs[0][0].view(np.uint32))
        assert np.array_equal(params.view(np.uint32), runs[0][1].view(np.uint32))
    ref_theta, ref_losses = mlp.train(theta, X, y, order, batch=batch, lr=3e-3)
    assert np.allclose(runs[0][0], ref_losses, rtol=1e-3, atol=1e-6)
    scale = np.max(np.abs(ref_theta))
    assert np.all(np.abs(runs[0][1] - ref_theta) <= 1e-3 * np.abs(ref_theta) + 1e-4 * scale)
