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
