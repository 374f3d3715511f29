"""The CTA-pair product at shapes that its rule leaves to it and where it can go wrong: one k-block, fewer
k-blocks than ring stages, a remainder of the ring, bands of fewer than eight tile rows, one tile a pair and
several, a last wave of few tiles; equal bits to the one-CTA kernel, which an output off the 32-byte grid
takes."""
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(5120, 4864, 64), (5120, 5120, 128), (5376, 4864, 320), (4864, 4096, 704), (256, 97280, 384), (97280, 256, 64),
          (2048, 4864, 512), (1280, 4864, 1088), (2560, 4096, 4096), (1024, 4864, 8192), (256, 19456, 8192)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_pairs_equal_one_cta_tiles(M, N, K):
    torch = pytest.importorskip("torch")
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
    assert torch.equal(C, one)
    rows = torch.arange(0, M, max(1, M // 512), device="cuda")               # FP64 on every 512th part of the rows
    ref = A[rows].double() @ B.double().T
    # BF16 products are exact in FP32; K sums of FP32 rounding each
    assert (C[rows].double() - ref).abs().max().item() <= 1e-4 * ref.abs().max().item()
