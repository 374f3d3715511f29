"""What a training step allocates: activations of the batch, and K slices only for layers whose weight
gradient is cut into several (a layer of one slice goes straight to the gradient array)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_one_slice_layers_need_no_slices():
    from paper_1911_10274_gb300 import titan as T
    n_in, hidden, B = 128, 4096, 128            # 32 x 32 tiles of a hidden layer: one slice each
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(B, n_in, device="cuda", generator=g).bfloat16()
    t = torch.randn(B, device="cuda", generator=g)
    net = T.MLP(n_in, hidden, seed=3)
    p0 = net.get_params()
    loss, grad = torch.empty(1, device="cuda"), torch.full((net.n_params,), float("nan"), device="cuda")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net.gradient(x, t, loss, grad)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    activations = 3 * B * hidden * (4 + 2 + 2) + 4 * (B // 32) * hidden * 4
    assert taken <= activations + (32 << 20), taken         # the slices of one layer alone would be 64 MiB
    # Adam's first step moves a parameter by lr g / (|g| + eps): by lr, but for eps and the rounding of p
    net.train_step(x, t, 1e-3)
    net.sync()
    gr = grad.cpu().numpy()
    assert np.isfinite(gr).all()
    big = np.abs(gr) > 1e-3 * np.abs(gr).max()
    assert big.sum() > 1000
    d = (net.get_params() - p0)[big] + 1e-3 * np.sign(gr[big])
    assert np.abs(d).max() <= 1e-3 * (1e-8 / np.abs(gr[big]).min() + 1e-5) + 6e-8 * np.abs(p0).max()
