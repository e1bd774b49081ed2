"""The fault-injection hook of the surrogate's tensor-core products on the shapes of the fused kernels:
with stall set, a training step returns SSLBM_ERR_TIMEOUT and skips the update; afterwards the same
handle trains as one that never stalled."""
import numpy as np
import pytest

from oracle import fno
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,m,H,n", [(32, 12, 64, 64), (16, 8, 32, 64)])
def test_stalled_products_time_out_on_fused_shapes(W, m, H, n):
    import torch
    cfg = dict(W=W, m=m, L=2, H=H)
    theta = fno.flatten(fno.init_params(1, **cfg), **cfg).astype(np.float32)
    u = torch.from_numpy(np.random.default_rng(3).uniform(0, 1, (1, 5, n, n)).astype(np.float32)).cuda()
    one = torch.ones(1, device="cuda")
    s = L.Surrogate(n=n, width=W, modes=m, layers=2, hidden=H, max_batch=1)
    assert s.fused
    s.set_params(theta)
    x = s.make_input(u, one, -one)
    s.set_wait_limit(polls=2000, stall=True)
    with pytest.raises(L.SslbmError) as e:
        s.train_step(x, u, 1e-3)
    assert e.value.status == L.SSLBM_ERR_TIMEOUT
    assert np.array_equal(s.get_params().view(np.uint32), theta.view(np.uint32))
    s.set_wait_limit()
    fresh = L.Surrogate(n=n, width=W, modes=m, layers=2, hidden=H, max_batch=1)
    fresh.set_params(theta)
    a, b = s.train_step(x, u, 1e-3), fresh.train_step(x, u, 1e-3)
    assert a == pytest.approx(b, rel=1e-6)
    np.testing.assert_allclose(s.get_params(), fresh.get_params(), rtol=1e-3, atol=1e-3)
