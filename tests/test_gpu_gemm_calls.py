"""What pb_gemm_bf16 accepts beyond the plain call.  Operands are small whole
numbers, so every product and sum is exact and results are compared exactly."""
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


def _operands(M, N, K, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    draw = lambda r, c: torch.randint(-2, 3, (r, c), generator=gen, device="cuda").to(torch.bfloat16)
    return draw(M, K), draw(N, K)


@pytest.mark.parametrize("extra", [16, 32, 16 | 1 << 20])
@pytest.mark.parametrize("flags", [0, pbits.EPI_RELU, pbits.EPI_OUT_BF16])
def test_other_flag_bits_are_ignored(flags, extra):
    import torch
    A, B = _operands(130, 24, 40, seed=flags + extra)
    dtype = torch.bfloat16 if flags & pbits.EPI_OUT_BF16 else torch.float32
    want, got = (torch.full((130, 24), 7.0, device="cuda", dtype=dtype) for _ in range(2))
    pbits.gemm_bf16(A, B, want, flags=flags)
    pbits.gemm_bf16(A, B, got, flags=flags | extra)
    assert torch.equal(got, want)


@pytest.mark.parametrize("M", [1, 100, 128, 300, 5000])
@pytest.mark.parametrize("N,K", [(64, 64), (33, 72), (17, 256)])
def test_result_over_an_operand(M, N, K):
    """D in A's place row by row, and (one row tile) in B's place: each CTA
    reads the rows that it writes before it writes them."""
    import torch
    A, B = _operands(M, N, K, seed=M + N + K)
    want = (A.double() @ B.double().T).to(torch.bfloat16)
    X = A.clone()
    pbits.gemm_bf16(X, B, X[:, :N], flags=pbits.EPI_OUT_BF16)
    assert torch.equal(X[:, :N], want) and torch.equal(X[:, N:], A[:, N:])
    if M <= 128:
        buf = torch.zeros((max(M, N), K), dtype=torch.bfloat16, device="cuda")
        buf[:N] = B
        pbits.gemm_bf16(A, buf[:N], buf[:M, :N], flags=pbits.EPI_OUT_BF16)
        assert torch.equal(buf[:M, :N], want)
