"""Loss and gradients of the row-size network for batches around its 64-sample tiles, one CTA and
several, and more tiles than CTAs, against the FP64 oracle; and twice the same (fixed order)."""
import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 63, 64, 65, 127, 129, 4097, 304 * 64, 304 * 64 + 1])
def test_loss_and_gradients(n):
    from paper_1504_05022_gb300.predictor import Trainer
    rng = np.random.default_rng(n)
    X = rng.uniform(0, 12, size=(n, 8)).astype(np.float32)
    cls = rng.integers(0, 16, n).astype(np.int32)
    y = rng.uniform(0, 15, n).astype(np.float32)
    th = mlp.init_params(7, mu=X.mean(0), sigma=X.std(0) + 0.5).astype(np.float32)
    tr = Trainer(torch.from_numpy(th).cuda())
    args = [torch.from_numpy(a).cuda() for a in (X, cls, y)]
    loss, grad = (t.clone() for t in tr.loss_grad(*args))
    rl, rg = mlp.loss_and_grad(th.astype(np.float64), X.astype(np.float64), cls, y.astype(np.float64))
    # 32-bit arithmetic over at most 33 terms per neuron and n samples, as the other tests of it
    assert abs(loss.item() - rl) <= 1e-5 * abs(rl)
    g = grad.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - rg) <= 1e-4 * np.linalg.norm(rg)
    loss2, grad2 = tr.loss_grad(*args)
    assert torch.equal(loss, loss2) and torch.equal(grad, grad2)
