"""sslbm_fno_backward on a copy of the forward pass's x that starts one float past a 16-byte
boundary, on the shapes of the fused kernels (which copy x in 16-byte groups): every gradient
element against the FP64 oracle within the bound of tests/fno_cases.py, as for an aligned x."""
import numpy as np
import pytest

from oracle import fno
from paper_2603_19789_gb300 import sslbm as L

from fno_cases import assert_within, bf16_round

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,m,layers,H,n,batch", [(32, 12, 2, 64, 64, 2), (16, 8, 1, 32, 128, 1)])
def test_backward_takes_an_unaligned_copy_of_x(W, m, layers, H, n, batch):
    import torch
    cfg = dict(W=W, m=m, L=layers, H=H)
    g = np.random.default_rng(n + layers)
    params = {k: v + 0.05 * g.standard_normal(v.shape) for k, v in fno.init_params(1, **cfg).items()}
    theta = fno.flatten(params, **cfg).astype(np.float32)
    p64 = fno.unflatten(theta.astype(np.float64), **cfg)
    for name in p64:
        if name[0] in "BQ" and p64[name].ndim == 2:
            p64[name] = bf16_round(p64[name]).astype(np.float64)
    u = g.uniform(0, 1, (batch, 5, n, n)).astype(np.float32)
    s = L.Surrogate(n=n, width=W, modes=m, layers=layers, hidden=H, max_batch=batch)
    assert s.fused
    s.set_params(theta)
    r0 = torch.from_numpy(g.uniform(1.2, 4.0, batch).astype(np.float32)).cuda()
    logd = torch.from_numpy(g.uniform(-3, -1, batch).astype(np.float32)).cuda()
    x = s.make_input(torch.from_numpy(u).cuda(), r0, logd)
    s.forward(x)
    buf = torch.empty(x.numel() + 1, device="cuda")
    shifted = buf[1:].view(x.shape)
    shifted.copy_(x)
    assert shifted.data_ptr() % 16 == 4
    dy = g.standard_normal((batch, 5, n, n)).astype(np.float32) * 1e-3
    s.backward(shifted, torch.from_numpy(dy).cuda())
    torch.cuda.synchronize()
    grads = fno.unflatten(s.get_grads().astype(np.float64), **cfg)
    xg = x.cpu().numpy().astype(np.float64)
    _, cache = fno.forward(p64, xg, **cfg)
    go = fno.backward(p64, cache, dy.astype(np.float64), **cfg)
    sd = fno.gradient_rounding_sd(p64, xg, cache, dy.astype(np.float64), **cfg)
    for name in go:
        assert_within(grads[name], go[name], sd[name], f"gradient {name}")
