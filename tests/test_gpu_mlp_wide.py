"""The surrogate with hidden layers wide enough for 256-column tiles with a GELU in the epilogue (K from 4096
and at least 304 tiles), forward, gradient and bias gradients, against FP64 at sampled entries."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_forward_and_gradients_with_wide_tiles():
    torch = pytest.importorskip("torch")
    from paper_1911_10274_gb300 import titan as T
    n_in, hid, B = 128, 4096, 128 * 19
    rng = np.random.default_rng(3)
    net = T.MLP(n_in, hid, seed=0)
    p = np.concatenate([w.ravel() for w in (
        rng.standard_normal((hid, n_in)) * np.sqrt(1.6 / n_in), 0.1 * rng.standard_normal(hid),
        rng.standard_normal((hid, hid)) * np.sqrt(1.6 / hid), 0.1 * rng.standard_normal(hid),
        rng.standard_normal((hid, hid)) * np.sqrt(1.6 / hid), 0.1 * rng.standard_normal(hid),
        rng.standard_normal(hid) / np.sqrt(hid), 0.1 * rng.standard_normal(1))]).astype(np.float32)
    net.set_params(p)
    x = torch.randn(B, n_in, device="cuda", generator=torch.Generator(device="cuda").manual_seed(5)).bfloat16()
    t = torch.randn(B, device="cuda", generator=torch.Generator(device="cuda").manual_seed(6))
    y, loss, grad = torch.empty(B, device="cuda"), torch.empty(1, device="cuda"), torch.empty(net.n_params, device="cuda")
    net.forward(x, y)
    net.gradient(x, t, loss, grad)
    W = [torch.tensor(np.array(w), device="cuda") for w in net.unpack(p)]
    # the network in FP64 on the BF16 weights; every activation rounded to BF16 as the products read it
    h, Z = x.double(), []
    for l in range(3):
        z = h @ W[2 * l].bfloat16().double().T + W[2 * l + 1].double()
        Z.append(z)
        h = torch.nn.functional.gelu(z).bfloat16().double()
        W.append(h)                              # W[8 + l]: the activation behind layer l
    want = h @ W[6].double() + W[7].double()
    # the bounds of test_gpu_mlp: a BF16 rounding may fall either way where FP32 and FP64 sums straddle its boundary
    assert (y.double() - want).abs().max().item() <= 3e-2 * want.abs().max().item()
    d = 2 * (want - t.double()) / B
    assert abs(loss.item() - ((want - t.double()) ** 2).mean().item()) <= 3e-2 * loss.item()
    g = net.unpack(grad.cpu().numpy())
    phi = lambda z: 0.5 * (1 + torch.erf(z / 2 ** 0.5)) + z * torch.exp(-z * z / 2) / (2 * np.pi) ** 0.5  # noqa: E731
    dz = (d[:, None] * W[6].double()[None] * phi(Z[2])).bfloat16().double()
    for l in (2, 1, 0):
        a = x.double() if l == 0 else W[8 + l - 1]
        for got, ref in ((g[2 * l], dz.T @ a), (g[2 * l + 1], dz.sum(0))):
            ref = ref.cpu().numpy()
            assert np.linalg.norm(got - ref) <= 3e-2 * np.linalg.norm(ref), l
        if l:
            dz = ((dz @ W[2 * l].bfloat16().double()) * phi(Z[l - 1])).bfloat16().double()
