"""The persistent launch of several plain models against the oracle, model by
model: one CTA taking several uneven models in turn, classes larger than the
consumers, the form without a persistent grid, short and long launches."""
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


# qubits, layers, chains, J (thresholds below and above 2^24), bins (0: all)
MODELS = [(2, 3, 40, 0.0, 0), (6, 8, 256, 4.0, 0), (11, 20, 64, 6.0, 0), (20, 40, 33, 7.0, 16), (1, 9, 32, 3.0, 0),
          (32, 24, 40, 5.6, 8)]


@pytest.mark.parametrize("persistent", ["0", "1"])
@pytest.mark.parametrize("shape", [None, (32, 32, 1), (32, 352, 0), (224, 96, 1)])
@pytest.mark.parametrize("lengths", [(3,), (2, 70)])
def test_models_bit_exact(persistent, shape, lengths, monkeypatch):
    monkeypatch.setenv("PB_PERSISTENT", persistent)
    # more groups than a grid of one CTA an SM holds: CTAs take several models
    what = [(n, d, W.hadamard_chain(d) if n == 1 else W.random_circuit(n, d, 10 * n + d), chains, J,
             np.arange(bins, dtype=np.uint32) if bins else None)
            for n, d, chains, J, bins in MODELS] * 2
    what.append((5, 7, W.random_circuit(5, 7, 3), 6400, 4.0, None))
    r = pbits.Run([pbits.Model(n, d, g, J) for n, d, g, _, J, _ in what],
                  [pbits.RunCfg(seed=90 + i, chains=c, alphas=a) for i, (_, _, _, c, _, a) in enumerate(what)])
    if shape:
        r.set_shape(*shape)
    assert (r.shape()["grid"] > 0) == (persistent == "1")
    for k in lengths:
        r.sweeps(k)
    r.wait()
    for i, (n, d, g, chains, J, alphas) in enumerate(what):
        ref = oracle.gibbs(n, d, g, J=J, seed=90 + i, chains=chains, sweeps=sum(lengths), alphas=alphas)
        cnt, valid, samples = r.histogram(i)
        assert np.array_equal(pbits.unslice_state(r.get_state(i), chains), ref["state"]), i
        assert valid == ref["valid"] and samples == ref["samples"] and np.array_equal(cnt, ref["cnt"]), i
