"""The autotuner's choice and its cache file."""
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


def _ms(r, sweeps):
    best = float("inf")
    for _ in range(4):
        r.sweeps(sweeps)
        best = min(best, r.stats()["last_ms"])
    return best


def test_tuned_shape_is_not_slower_than_the_default():
    """The tiny circuit runs best with one consumer warp, its default shape:
    two cost 14 %, so 5 % tells them apart."""
    wl = W.tiny()
    m = pbits.Model(wl.n, wl.d, wl.gates, wl.J)
    plain, tuned = (pbits.Run([m], [pbits.RunCfg(seed=wl.seed, chains=wl.chains)]) for _ in range(2))
    tuned.tune(trial_sweeps=5000)
    assert _ms(tuned, 5000) <= 1.05 * _ms(plain, 5000), (plain.shape(), tuned.shape())


def test_cached_shape_of_another_kind_of_run(tmp_path):
    """A cache file is used again by the same run, but a plain run's entry is
    no answer for a general-gate run of equal n, d and chains (its 608 threads
    are more than that run takes), and an entry whose shape the run refuses
    leads to trials, not to an error."""
    cache = str(tmp_path / "tune.txt")
    n, d, chains = 12, 20, 256
    m = pbits.Model(n, d, W.random_circuit(n, d, 4), 6.0)
    plain = pbits.Run([m], [pbits.RunCfg(seed=1, chains=chains)])
    plain.tune(trial_sweeps=5, cache_path=cache)
    lines = open(cache).read().splitlines()
    assert len(lines) == 1
    key = lines[0].split()[0]
    with open(cache, "w") as f:
        f.write(f"{key} 224 352 0 1.0\n")
    g, mats = W.random_general_circuit(n, d, 4, frac_u=0.3)
    general = pbits.Run([pbits.Model(n, d, g, 6.0, mats=mats)], [pbits.RunCfg(seed=1, chains=chains)])
    general.tune(trial_sweeps=5, cache_path=cache)
    assert len(open(cache).read().splitlines()) == 2
    # fewer bins: trials of its own
    few = pbits.Run([m], [pbits.RunCfg(seed=1, chains=chains, alphas=[0, 1])])
    few.tune(trial_sweeps=5, cache_path=cache)
    assert len(open(cache).read().splitlines()) == 3
    # the same run: a hit
    again = pbits.Run([m], [pbits.RunCfg(seed=1, chains=chains)])
    assert again.tune(trial_sweeps=5, cache_path=cache) == 1.0
    assert (again.shape()["consumers"], again.shape()["producers"]) == (224, 352)
    # a refused entry: trials
    with open(cache, "w") as f:
        f.write(f"{key} 225 352 0 1.0\n")
    again.tune(trial_sweeps=5, cache_path=cache)
    assert again.shape()["consumers"] % 32 == 0 and len(open(cache).read().splitlines()) == 2
