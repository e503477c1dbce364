"""General-gate sweeps from comparison and acceptance words at the edges of
their periods, classes and histogram placement: chain words and counts equal
the oracle's exactly, phase sums within the stated per-term bound (3e-7 a
term, 7.4e-10 a gate, plus the FP64 sum)."""
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


@pytest.mark.parametrize("n,d,chains,sweeps,J,frac,shape", [
    (2, 3, 33, (1, 2, 31), 3.0, 1.0, None),        # every one-qubit gate general; 16-sweep periods
    (6, 9, 64, (15, 1, 17), 0.5, 0.5, None),       # thresholds with one bits in every plane
    (8, 16, 64, (21,), 5.6, 0.3, (32, 32)),        # classes beyond the consumers
    (5, 8, 5000, (40,), 3.0, 0.35, None),          # two CTAs an SM
    (12, 10, 64, (11,), 4.0, 0.3, None),           # 4096 bins of phase sums beside the tables
    (13, 8, 64, (9,), 4.0, 0.3, None),             # bins in global memory
    (30, 35, 32, (3,), 5.0, 0.05, None),           # more than 1024 p-bits
])
def test_edges_bit_exact(n, d, chains, sweeps, J, frac, shape):
    g, mats = W.random_general_circuit(n, d, 10 * n + d, frac_u=frac)
    alphas = None if n <= 13 else np.arange(16, dtype=np.uint32)
    m = pbits.Model(n, d, g, J, mats=mats)
    r = pbits.Run([m], [pbits.RunCfg(seed=78, chains=chains, alphas=alphas)])
    if shape:
        r.set_shape(*shape)
    for s in sweeps:
        r.sweeps(s)
    r.wait()
    ref = oracle.u_gibbs(n, d, g, mats, J=J, seed=78, chains=chains, sweeps=sum(sweeps), alphas=alphas)
    assert np.array_equal(pbits.unslice_state(r.get_state(), chains), ref["state"])
    sums, cnt, valid, samples = r.phase_sums()
    assert np.array_equal(cnt, ref["cnt"])
    assert valid == ref["valid"] and samples == ref["samples"]
    tol = cnt * (3e-7 + m.info()["n_u"] * 7.4e-10) + 1e-9
    assert np.all(np.abs(sums - ref["sum"]) <= tol)


def test_plain_model_beside_a_general_one():
    """A plain circuit in a general-gate run keeps its exact phase classes."""
    g1, mats1 = W.random_general_circuit(5, 8, 3, frac_u=0.4)
    g2 = W.random_circuit(6, 7, 9)
    ms = [pbits.Model(5, 8, g1, 3.0, mats=mats1), pbits.Model(6, 7, g2, 3.0)]
    r = pbits.Run(ms, [pbits.RunCfg(seed=5, chains=70), pbits.RunCfg(seed=6, chains=100)])
    r.sweeps(19)
    ref = oracle.gibbs(6, 7, g2, J=3.0, seed=6, chains=100, sweeps=19)
    assert np.array_equal(pbits.unslice_state(r.get_state(1), 100), ref["state"])
    assert np.array_equal(r.histogram(1)[0], ref["cnt"])
    ref = oracle.u_gibbs(5, 8, g1, mats1, J=3.0, seed=5, chains=70, sweeps=19)
    assert np.array_equal(pbits.unslice_state(r.get_state(0), 70), ref["state"])
