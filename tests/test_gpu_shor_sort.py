"""The sort of the column samples at the edges of the block that is sorted in
shared memory: y of every sample and all probabilities against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2007_07379_gb300 import build, pbits

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    pbits.load()


@pytest.mark.parametrize("T", [1, 2, 3, 31, 65, 2049, 4096, 4097, 8192, 20000])
def test_sorted_samples(T):
    N, a, n = 961, 3, 10
    x = np.random.default_rng(T).integers(0, 2 ** n, T).astype(np.uint32)
    sc = pbits.ShorColumns(n, T)
    y = sc.run(N, a, x, want_y=True)
    ref = np.array([pow(a, int(v), N) for v in x])
    assert np.array_equal(y, ref)
    want, _ = oracle.shor_columns(N, a, n, x)
    # each FP32 phasor within 1e-6: a group's |sum|^2 moves by 1e-6 g^2 at most; tenfold
    _, g = np.unique(ref, return_counts=True)
    tol = 1e-5 * float(np.sum(g.astype(np.float64) ** 2)) / (2 ** n * T) + 1e-12
    assert np.all(np.abs(sc.prob.cpu().numpy() - want) <= tol)
