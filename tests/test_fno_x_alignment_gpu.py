"""An x that starts off a 16-byte boundary is refused by the host, before anything is launched, by
every call that reads it, on the fused and the separate kernels; the same values aligned are taken
afterwards."""
import numpy as np
import pytest

from oracle import fno
from paper_2603_19789_gb300 import sslbm as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,m,layers,H,n", [(32, 12, 1, 64, 64), (16, 8, 1, 32, 128), (8, 4, 1, 16, 32)])
def test_unaligned_x_is_refused(W, m, layers, H, n):
    import torch
    cfg = dict(W=W, m=m, L=layers, H=H)
    s = L.Surrogate(n=n, width=W, modes=m, layers=layers, hidden=H, max_batch=1)
    s.set_params(fno.flatten(fno.init_params(1, **cfg), **cfg).astype(np.float32))
    u = torch.rand((1, 5, n, n), device="cuda")
    one = torch.ones(1, device="cuda")
    x = s.make_input(u, one, -one)
    shifted = torch.empty(x.numel() + 1, device="cuda")[1:].view(x.shape)
    shifted.copy_(x)
    assert shifted.data_ptr() % 16 == 4
    y, dy = torch.empty_like(u), torch.full_like(u, 1e-3)

    def refused(call):
        with pytest.raises(L.SslbmError) as e:
            call()
        assert e.value.status == L.SSLBM_ERR_BAD_ARG

    s.forward(x, y)
    refused(lambda: s.backward(shifted, dy))
    s.backward(x, dy)
    refused(lambda: s.forward(shifted, y))
    refused(lambda: s.infer(shifted, y))
    refused(lambda: s.train_step(shifted, u, 0.0))
    torch.cuda.synchronize()
    assert np.isfinite(s.get_grads()).all()
