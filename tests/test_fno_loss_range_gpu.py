"""The training loss over FP32's whole range: squares beyond it, and infinities, as FP64 sums
give them from the same FP32 differences."""
import numpy as np
import pytest

from oracle import fno
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu


def _loss(target, mass_weight=0.0, neg_weight=0.0):
    """Loss of one step at learning rate 0 on a fixed network, and its FP64 value from the y buffer."""
    import torch
    cfg = dict(W=16, m=8, L=1, H=32)
    n, batch = 64, 2
    s = L.Surrogate(n=n, width=16, modes=8, layers=1, hidden=32, max_batch=batch)
    s.set_params(fno.flatten(fno.init_params(1, **cfg), **cfg).astype(np.float32))
    s.set_loss_weights(mass_weight, neg_weight)
    u = torch.from_numpy(np.random.default_rng(3).uniform(0, 1, (batch, 5, n, n)).astype(np.float32)).cuda()
    one = torch.ones(batch, device="cuda")
    x = s.make_input(u, one, -one)
    y = s.forward(x)
    t = target(y)
    loss = s.train_step(x, t, 0.0)
    y64 = s._y[:batch].cpu().numpy()
    scale = np.ones((batch, 5, 1, 1), dtype=np.float32)
    # the infection scale of E and I, from the input's scale channel
    scale[:, 1:3] = np.power(10.0, 4.0 * x[:, 7, 0, 0].cpu().numpy().astype(np.float64) - 4.0)[:, None, None, None]
    d = (y64 - t.cpu().numpy()).astype(np.float64) / scale.astype(np.float64)
    with np.errstate(over="ignore"):
        return loss, np.mean(d * d)


@pytest.mark.parametrize("weights", [(0.0, 0.0), (30.0, 30.0)])
def test_squares_beyond_float_range(weights):
    def target(y):
        t = y.clone()
        t[0, 0, 3, 5] = 1e25
        t[1, 4, 7, 1] = -3e30
        return t
    loss, want = _loss(target, *weights)
    assert loss == pytest.approx(want, rel=1e-6) and want > 1e50


def test_an_infinite_target_gives_an_infinite_loss():
    def target(y):
        t = y.clone()
        t[0, 2, 1, 1] = float("inf")
        return t
    loss, want = _loss(target)
    assert np.isinf(want) and np.isinf(loss) and loss > 0
