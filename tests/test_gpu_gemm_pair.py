"""The CTA-pair product at the sizes where it can go wrong: one k-block, fewer
k-blocks than ring stages, a remainder of the ring, bands of fewer than eight tile
rows, a last wave of few tiles, several tiles per pair; equal bits to the one-CTA
kernel (the same products summed in the same order over K), which an output that
is not 32-byte aligned still takes."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M,N,K", [(2048, 2560, 64), (2304, 2304, 832), (4864, 4096, 448), (256, 19456, 384),
                                   (19456, 256, 320), (2560, 4096, 4096)])
def test_pair_product(M, N, K):
    from paper_1911_10274_gb300 import titan as T
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, device="cuda", generator=g).bfloat16()
    B = torch.randn(N, K, device="cuda", generator=g).bfloat16()
    C = torch.full((M, N), float("nan"), device="cuda")
    one = torch.full((M * N + 1,), float("nan"), device="cuda")[1:].view(M, N)
    T.titan_gemm_bf16_tn(A, B, C)
    T.titan_gemm_bf16_tn(A, B, one)
    torch.cuda.synchronize()
    T.titan_gemm_check()
    ref = A.double() @ B.double().T
    # BF16 products are exact in FP32; K sums of FP32 rounding each
    assert (C.double() - ref).abs().max().item() <= 1e-4 * ref.abs().max().item()
    assert torch.equal(C, one)
