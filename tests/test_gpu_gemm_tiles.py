"""The staged tensor-core GEMM at the edges of its tiles, chunks and stages.
Operands are small whole numbers, so every product and partial sum is exact in
fp32 (|sum| <= 4 K < 2^24): the result must equal the integer product."""
import pytest

from paper_2007_07379_gb300 import build, pbits

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    pbits.load()


@pytest.mark.parametrize("M,N,K", [
    (1, 1, 8), (63, 17, 24), (64, 32, 128), (65, 33, 136), (127, 48, 120), (129, 16, 640),
    (256, 256, 4096), (256, 48, 1000), (4096, 256, 48), (4096, 256, 256), (20000, 256, 512),
    (130, 300, 513 * 8)])
def test_exact_products(M, N, K):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(M * 1000 + N * 10 + K)
    A = torch.randint(-2, 3, (M, K), generator=gen, device="cuda").to(torch.bfloat16)
    B = torch.randint(-2, 3, (N, K), generator=gen, device="cuda").to(torch.bfloat16)
    bias = torch.randint(-8, 9, (N,), generator=gen, device="cuda").float()
    D = torch.full((M, N), float("nan"), device="cuda")
    pbits.gemm_bf16(A, B, D, bias=bias)
    want = (A.double() @ B.double().T + bias.double()).float()
    assert torch.equal(D, want)
    # ReLU, bf16 output, mask: the rounding of the exact value
    mask = torch.randint(0, 2, (M, N), generator=gen, device="cuda").to(torch.bfloat16)
    E = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    pbits.gemm_bf16(A, B, E, mask=mask, flags=pbits.EPI_RELU | pbits.EPI_OUT_BF16 | pbits.EPI_MASK)
    want = torch.relu(A.double() @ B.double().T) * (mask > 0)
    assert torch.equal(E, want.to(torch.bfloat16))
    # accumulation into D
    pbits.gemm_bf16(A, B, D, flags=pbits.EPI_ACCUM)
    assert torch.equal(D, (2 * (A.double() @ B.double().T) + bias.double()).float())
