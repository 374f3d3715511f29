"""The surrogate's kernels at the edges of their forms (widths the one-kernel pass takes and does
not, one block of 128 rows and many, K slices of each count) against torch in FP64 on the same
BF16 weights.  Tolerances as in the MLP tests: activations are stored in BF16 (2^-9 a value)."""
import numpy as np
import pytest

from oracle import mlp as ref
from paper_1911_10274_gb300 import titan as T

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_in,hidden,B", [(128, 128, 128), (384, 256, 640), (256, 384, 1280), (640, 512, 2176),
                                           (1280, 1024, 256), (256, 512, 4096), (128, 640, 384)])
def test_forward_and_gradient(n_in, hidden, B):
    net = T.MLP(n_in, hidden, seed=hidden + B)
    rng = np.random.default_rng(B)
    p = net.get_params()
    idx = net.unpack(np.arange(net.n_params))
    for b in (1, 3, 5, 7):                                        # biases that are not zero
        p[idx[b].ravel()] = rng.normal(0, 0.1, idx[b].size)
    net.set_params(p)
    pr = p.astype(np.float64)
    for w in (0, 2, 4):
        pr[idx[w].ravel()] = torch.as_tensor(p[idx[w].ravel()]).bfloat16().double().numpy()
    x = torch.as_tensor(rng.normal(0, 1, (B, n_in)), dtype=torch.float32).bfloat16().cuda()
    t = torch.as_tensor(rng.normal(0, 0.3, B), dtype=torch.float32).cuda()
    xr = x.float().cpu().numpy().astype(np.float64)
    y, loss = torch.empty(B, device="cuda"), torch.empty(1, device="cuda")
    grad = torch.empty(net.n_params, device="cuda")
    net.forward(x, y)
    y_ref, _, _ = ref.forward(pr, xr, n_in, hidden)
    assert np.abs(y.cpu().numpy() - y_ref).max() <= 3e-2 * np.abs(y_ref).max()
    net.gradient(x, t, loss, grad)
    l_ref, g_ref = ref.loss_and_grad(pr, xr, t.cpu().numpy().astype(np.float64), n_in, hidden)
    assert float(loss) == pytest.approx(l_ref, rel=3e-2)
    g = grad.cpu().numpy().astype(np.float64)
    for sl in idx[:-1]:
        gs, rs = g[sl.ravel()], g_ref[sl.ravel()]
        assert np.linalg.norm(gs - rs) <= 3e-2 * np.linalg.norm(rs)


def test_training_step_on_a_view_off_the_16_byte_grid_and_a_growing_batch():
    rng = np.random.default_rng(3)
    nets = [T.MLP(256, 256, seed=1) for _ in range(2)]
    for B in (128, 512, 256):
        data = torch.as_tensor(rng.normal(0, 1, B * 256 + 1), dtype=torch.float32).bfloat16().cuda()
        off = data[1:].view(B, 256)
        t = torch.as_tensor(rng.normal(0, 1, B), dtype=torch.float32).cuda()
        assert off.data_ptr() % 16
        on, loss = off.clone(), torch.empty(2, device="cuda")
        torch.cuda.synchronize()
        for net, x, k in zip(nets, (on, off), (0, 1)):
            net.train_step(x, t, 1e-3, loss[k:k + 1])
            net.sync()
        assert loss[0] == loss[1]
        assert np.array_equal(nets[0].get_params(), nets[1].get_params())


@pytest.mark.parametrize("offset", [0, 1, 4, 8])
@pytest.mark.parametrize("M,N,K", [(128, 128, 64), (256, 1280, 128), (2048, 5120, 192)])
def test_product_into_a_view_at_any_offset(M, N, K, offset):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, device="cuda", generator=g).bfloat16()
    B = torch.randn(N, K, device="cuda", generator=g).bfloat16()
    flat = torch.full((M * N + 16,), 7.0, device="cuda")
    C = flat[offset:offset + M * N].view(M, N)
    T.titan_gemm_bf16_tn(A, B, C)
    torch.cuda.synchronize()
    T.titan_gemm_check()
    want = A.double() @ B.double().T
    assert (C.double() - want).abs().max().item() <= 1e-4 * want.abs().max().item()
    assert torch.all(flat[:offset] == 7.0) and torch.all(flat[offset + M * N:] == 7.0)
