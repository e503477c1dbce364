"""Launches of few sweeps, whose period, producers and shared memory shrink
with them: chains and counts equal the oracle's at the lengths where the
period changes, from one p-bit a layer to models of one sweep a period, with
few and with many chain groups, and over launches of different lengths."""
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


def _check(runs, sweeps):
    for (n, d, g, J, seed, chains, alphas), r, i in runs:
        ref = oracle.gibbs(n, d, g, J=J, seed=seed, chains=chains, sweeps=sweeps, alphas=alphas)
        cnt, valid, samples = r.histogram(i)
        assert np.array_equal(pbits.unslice_state(r.get_state(i), chains), ref["state"])
        assert valid == ref["valid"] and samples == ref["samples"] and np.array_equal(cnt, ref["cnt"])


@pytest.mark.parametrize("n,d,chains", [(1, 4, 64), (3, 4, 200), (3, 4, 9760), (6, 8, 9760), (8, 16, 100),
                                        (12, 20, 64), (24, 32, 40), (32, 64, 40)])
def test_lengths(n, d, chains):
    g = W.hadamard_chain(d) if n == 1 else W.random_circuit(n, d, 17)
    alphas = None if n <= 12 else np.arange(8, dtype=np.uint32)
    m = pbits.Model(n, d, g, 3.0)
    for lengths in ([1], [2], [3], [4, 1], [5], [7, 2], [8], [9], [12], [15, 16], [17], [33], [64]):
        if n * d * chains * sum(lengths) > 3e7:
            continue
        r = pbits.Run([m], [pbits.RunCfg(seed=9, chains=chains, alphas=alphas)])
        for k in lengths:
            r.sweeps(k)
        _check([((n, d, g, 3.0, 9, chains, alphas), r, 0)], sum(lengths))


@pytest.mark.parametrize("sweeps", [1, 2, 5, 13, 40])
def test_uneven_models_in_one_launch(sweeps, monkeypatch):
    """One CTA a group (no persistent grid): the largest model's period sets
    the launch's shared memory, the smaller ones take longer periods in it."""
    monkeypatch.setenv("PB_PERSISTENT", "0")
    what = [(n, d, W.random_circuit(n, d, n), 3.0, 40 + n, chains, None)
            for n, d, chains in ((2, 3, 96), (5, 7, 33), (11, 20, 64))]
    r = pbits.Run([pbits.Model(n, d, g, J) for n, d, g, J, *_ in what],
                  [pbits.RunCfg(seed=s, chains=c) for *_, s, c, _ in what])
    r.sweeps(sweeps)
    _check([(w, r, i) for i, w in enumerate(what)], sweeps)


@pytest.mark.parametrize("n,d,chains", [(3, 4, 100), (3, 4, 9760), (8, 16, 100), (12, 20, 64)])
@pytest.mark.parametrize("lengths", [[1], [2, 3], [5], [8], [13], [24], [33]])
def test_general_gates(n, d, chains, lengths):
    g, mats = W.random_general_circuit(n, d, 6, frac_u=0.5)
    r = pbits.Run([pbits.Model(n, d, g, 3.0, mats=mats)], [pbits.RunCfg(seed=5, chains=chains)])
    for k in lengths:
        r.sweeps(k)
    ref = oracle.u_gibbs(n, d, g, mats, J=3.0, seed=5, chains=chains, sweeps=sum(lengths))
    sums, cnt, valid, samples = r.phase_sums()
    assert np.array_equal(pbits.unslice_state(r.get_state(), chains), ref["state"])
    assert valid == ref["valid"] and samples == ref["samples"] and np.array_equal(cnt, ref["cnt"])
    # the bound of a term, times the count
    n_u = int(np.sum(g[:, 0] == W.U))
    assert np.all(np.abs(sums - ref["sum"]) <= cnt * (3e-7 + n_u * 7.4e-10) + 1e-9)
