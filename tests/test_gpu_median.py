"""The median rule: sigma^2 is exactly the lower median of the squared distances
(inputs on the 2^-16 grid: the distances are exact), by one pass over the
distances between two sampled keys and by radix passes, whichever the data's
ties and the order call for."""
from types import SimpleNamespace

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from gpu_util import Ctx, lib
    g = Ctx(lib())
    yield g
    g.close()


def _series(kind, n, rng):
    if kind == "iid":
        return rng.integers(-2 ** 18, 2 ** 18, (n, 8)).astype(np.float64) * 2.0 ** -16
    if kind == "ties":                      # a few dozen distinct distances
        return rng.integers(0, 3, (n, 4)).astype(np.float64)
    if kind == "half_equal":                # the median inside a large group of equal distances
        X = rng.integers(-2 ** 18, 2 ** 18, (n, 4)).astype(np.float64) * 2.0 ** -16
        X[: (3 * n) // 4] = X[0]
        return X
    X = rng.integers(-2 ** 10, 2 ** 10, (n, 4)).astype(np.float64) * 2.0 ** -16   # two clusters: about half
    X[n // 2:] += 100.0                                                            # of the distances to each side
    return X


def _lower_median(X):
    n = X.shape[0]
    v = []
    for i in range(n - 1):
        v.append(((X[i + 1:] - X[i]) ** 2).sum(1))      # exact in float64 for these inputs
    v = np.concatenate(v)
    r = (len(v) - 1) // 2
    return np.partition(v, r)[r]


@pytest.mark.parametrize("kind", ["iid", "ties", "half_equal", "clusters"])
@pytest.mark.parametrize("n", [2, 3, 64, 65, 257, 1024, 4097, 4899, 4900, 7001])
def test_sigma_is_the_exact_median(G, n, kind):
    X = _series(kind, n, np.random.default_rng(n))
    m = _lower_median(X)
    if m == 0.0:
        X = X + np.arange(n)[:, None] * 2.0 ** -16       # sigma = 0 leaves no graph
        m = _lower_median(X)
    _, _, _, s = G.graph(X)
    assert float(s) == np.sqrt(m)


def test_batched_medians_with_ties(G):
    from test_gpu_batched import _check, _run
    rng = np.random.default_rng(8)
    pairs = [SimpleNamespace(X=(rng.integers(0, 4, (n, 6)).astype(np.float64), rng.integers(0, 4, (n, 6)).astype(np.float64)))
             for n in (90, 150, 333)]
    F, tops, stats = _run(G, pairs, 10, 0, G.cdl.CDL_F64)
    _check(pairs, F, tops, stats, 0)
