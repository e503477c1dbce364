"""Exact-sampler launches of plain models (PB_ELIM) against the oracle: both
places where the counts are kept (shared memory, and global memory where the
bins are too many or the samples too few to pay for it), warp counts that
follow the launch's length, and several models in one launch."""
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


def _run(what, lengths, **kw):
    """what: (n, d, chains) of every model; lengths: samples of every launch."""
    gates = [W.random_circuit(n, d, 50 + n) for n, d, _ in what]
    models = [pbits.Model(n, d, g, W.default_J(n, d, g)) for (n, d, _), g in zip(what, gates)]
    r = pbits.Run(models, [pbits.RunCfg(seed=30 + i, chains=c, sampler=pbits.PB_ELIM, **kw)
                           for i, (_, _, c) in enumerate(what)])
    for k in lengths:
        r.sweeps(k)
    r.wait()
    for i, ((n, d, chains), g) in enumerate(zip(what, gates)):
        ref = oracle.elim(n, d, g, seed=30 + i, chains=chains, sweeps=sum(lengths), **kw)
        cnt, valid, samples = r.histogram(i)
        assert valid == ref["valid"] and samples == ref["samples"], i
        assert np.array_equal(cnt, ref["cnt"]), i
        assert np.array_equal(pbits.unslice_state(r.get_state(i), chains), ref["state"]), i


@pytest.mark.parametrize("lengths", [[1], [4, 5], [31], [32], [33, 1, 64], [130]])
@pytest.mark.parametrize("chains", [40, 9760])
def test_both_sides_of_the_shared_histogram(lengths, chains):
    _run([(6, 8, chains)], lengths)  # 64 bins: from 32 samples on


@pytest.mark.parametrize("lengths", [[95], [96], [97, 3]])
def test_recorded_samples_decide(lengths):
    _run([(6, 8, 100)], lengths, burn_in=2, record_every=3)


@pytest.mark.parametrize("n,d,chains,lengths", [(13, 6, 200, [9, 3]), (12, 20, 64, [2, 2050]), (14, 5, 9760, [5])])
def test_many_bins(n, d, chains, lengths):
    _run([(n, d, chains)], lengths)


@pytest.mark.parametrize("lengths", [[3, 2], [16, 40], [520, 7]])
def test_several_models(lengths):
    _run([(4, 9, 100), (11, 12, 64), (7, 30, 33), (2, 3, 5000)], lengths)
