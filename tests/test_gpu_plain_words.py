"""Plain sweeps from comparison words: chains and histograms bit-identical to
the oracle's at the edges of the kernel's periods, tasks and thresholds
(integers: exact equality)."""
import numpy as np
import pytest

import oracle
from paper_2007_07379_gb300 import build, pbits
from paper_2007_07379_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    pbits.load()


@pytest.mark.parametrize("n,d,chains,sweeps,J,shape", [
    (1, 1, 33, (1, 37), 3.0, None),           # one p-bit a sweep
    (4, 8, 64, (15, 1, 17), 0.0, None),       # thresholds 2^31: decided by plane 0; 16-sweep periods
    (3, 11, 64, (1, 2, 31, 33), 0.4, None),   # one bits in every plane; 33 p-bits
    (8, 8, 64, (64,), 5.6, (32, 32)),         # thr1 below 2^24; classes beyond the consumers
    (8, 8, 64, (64,), 5.4, (224, 352)),       # just above
    (12, 20, 64, (1, 7, 9, 40), 9.0, None),   # thr3 < 2^8
    (29, 9, 32, (13,), 4.0, None),            # one transpose: 3 + 29 rows
    (30, 9, 32, (13,), 4.0, None),            # two transposes
    (32, 33, 40, (5,), 6.0, None),            # more than 1024 p-bits: odd tail of a 2-sweep period
    (32, 64, 32, (3,), 7.5, None),            # the largest model: 1-sweep periods
    (6, 8, 5000, (70,), 4.0, None),           # more groups than SMs: two CTAs an SM
])
def test_edges_bit_exact(n, d, chains, sweeps, J, shape):
    g = W.random_circuit(n, d, 100 * n + d)
    alphas = None if n <= 12 else np.arange(32, dtype=np.uint32)
    m = pbits.Model(n, d, g, J)
    r = pbits.Run([m], [pbits.RunCfg(seed=77, chains=chains, alphas=alphas, burn_in=2, record_every=3)])
    if shape:
        r.set_shape(*shape)
    for s in sweeps:
        r.sweeps(s)
    r.wait()
    ref = oracle.gibbs(n, d, g, J=J, seed=77, chains=chains, sweeps=sum(sweeps), burn_in=2,
                       record_every=3, alphas=alphas)
    assert np.array_equal(pbits.unslice_state(r.get_state(), chains), ref["state"])
    cnt, valid, samples = r.histogram()
    assert np.array_equal(cnt, ref["cnt"])
    assert valid == ref["valid"] and samples == ref["samples"]
