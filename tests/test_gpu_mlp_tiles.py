"""Network kernels at the edges of their sample tiles (16 and 128 samples forward, 48 or 64 in the gradient) and with a
gradient buffer that starts off a 16-byte boundary, against the FP64 network oracle. FP32 sums of at most a few thousand
terms of either sign: 1e-4 of the largest output, 1e-3 of the gradient's norm."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(64, 64, 16), (48, 32, 12)])
@pytest.mark.parametrize("B,shift", [(1, 0), (15, 1), (17, 2), (47, 0), (49, 3), (65, 0), (129, 1), (14593, 0)])
def test_forward_and_gradient_at_tile_edges(sizes, B, shift):
    import torch
    from oracle import mlp as omlp
    from paper_1808_05066_gb300 import hdg
    nin, nh, nout = sizes
    P = hdg.hdg_mlp_param_count(nin, nh, nout)
    dev = torch.device("cuda", 0)
    params = torch.empty(((14 * P + 3) // 4,), dtype=torch.float32, device=dev)
    hdg.hdg_mlp_init(params, nin, nh, nout, 5)
    rng = np.random.default_rng(B)
    x = rng.normal(size=(B, nin)).astype(np.float32)
    t = rng.normal(scale=0.3, size=(B, nout)).astype(np.float32)
    xd, td = torch.from_numpy(x).to(dev), torch.from_numpy(t).to(dev)
    y = torch.empty((B, nout), dtype=torch.float32, device=dev)
    hdg.hdg_mlp_forward(params, nin, nh, nout, xd, B, y)
    buf = torch.full((P + 8,), 7.0, dtype=torch.float32, device=dev)
    grad = buf[shift:shift + P]
    loss = torch.empty(1, dtype=torch.float32, device=dev)
    hdg.hdg_mlp_gradient(params, grad, nin, nh, nout, xd, td, B, loss)
    torch.cuda.synchronize()
    w16 = params[3 * P:3 * P + (P + 1) // 2].view(torch.bfloat16)[:P].double().cpu().numpy()
    x64, t64 = x.astype(np.float64), t.astype(np.float64)
    y_o, _ = omlp.forward(w16, x64, nin, nh, nout)
    g_o = omlp.gradient(w16, x64, t64, nin, nh, nout)
    assert np.abs(y.cpu().numpy() - y_o).max() <= 1e-4 * np.abs(y_o).max()
    assert np.linalg.norm(grad.cpu().numpy() - g_o) <= 1e-3 * np.linalg.norm(g_o)
    assert abs(float(loss.item()) - omlp.loss(w16, x64, t64, nin, nh, nout)) <= 1e-4 * abs(float(loss.item()))
    assert bool((buf[:shift] == 7.0).all()) and bool((buf[shift + P:] == 7.0).all())
