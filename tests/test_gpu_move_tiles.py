"""The learned move over chain counts whose 64-row tiles take each split of
log q over the GPU: chains are independent given the run's seed, so the
chains of a small run equal the first ones of a large run bit for bit."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n,d,hidden", [(5, 7, 64), (16, 24, 256)])
def test_chains_do_not_depend_on_the_split(n, d, hidden):
    g = W.random_circuit(n, d, 40 + n)
    m = pbits.Model(n, d, g, 0.1)  # most moves are accepted or refused by log q
    net = pbits.Mlp(n, d, hidden=hidden, batch=1024, seed=3)
    alphas = np.arange(4, dtype=np.uint32)
    ref = None
    for chains in (32, 64, 70, 64 * 76, 64 * 77, 64 * 151 + 1, 64 * 153):
        r = pbits.Run([m], [pbits.RunCfg(seed=9, chains=chains, alphas=alphas, sampler=pbits.PB_LEARNED,
                                         proposal=net, mh_every=1)])
        r.sweeps(12)
        r.wait()
        s = pbits.unslice_state(r.get_state(), chains)
        if ref is None:
            ref = s
            assert not np.array_equal(s, pbits.unslice_state(_plain(m, alphas), 32))
        assert np.array_equal(s[:min(len(ref), chains)], ref[:chains])
        if chains > len(ref):
            ref = s


def _plain(m, alphas):
    r = pbits.Run([m], [pbits.RunCfg(seed=9, chains=32, alphas=alphas)])
    r.sweeps(12)
    r.wait()
    return r.get_state()
