"""The one-pass peak search against the definition, in numpy: exact counts,
positions and maxima, for values and thresholds of either sign, zero,
infinities and NaN."""
import numpy as np
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


@pytest.mark.parametrize("n", [1, 2, 5, 13, 21, 23])
@pytest.mark.parametrize("special", [False, True])
def test_peaks_match_definition(n, special):
    import torch
    rng = np.random.default_rng(n)
    v = rng.standard_normal(1 << n).round(1)  # ties and zeros too
    if special:
        for k, x in enumerate([-0.0, 0.0, np.inf, -np.inf, np.nan, -np.nan, 5e-324, -5e-324]):
            v[rng.integers(0, 1 << n, 1 + (1 << n) // 64)] = x
    sc = pbits.ShorColumns(n, 1)
    sc.prob.copy_(torch.from_numpy(v))
    with np.errstate(invalid="ignore"):
        peak = (v >= np.roll(v, 1)) & (v > np.roll(v, -1))
        for thr in (2.5, 0.3, 5e-324, 0.0, -0.0, -1.1, -np.inf, np.inf, np.nan):
            want = np.flatnonzero(peak & ~(v < thr))
            count, pos, mx = sc.peaks(thr, 4096)
            assert count == len(want)
            assert len(pos) == min(count, 4096) and np.all(np.isin(pos, want))
            if count <= 4096:
                assert np.array_equal(pos, want)
            assert mx == np.fmax(v, 0.0).max()
