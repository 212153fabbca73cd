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


@pytest.mark.parametrize("top", [64, 65, 127])
@pytest.mark.parametrize("T", [63, 64, 256, 257, 511, 512, 513, 1100])
def test_distance_exact_at_the_digit_extremes(G, T, top):
    """Two series whose base-256 digits are as large as they get, so that the exact
    float32 sums of a chunk of samples reach their bound: sigma^2 is their distance."""
    for d0, d1, s in ((-128, -128, 1), (127, 127, 1), (-128, -128, -1), (127, -128, -1)):
        a = (top << 16) + (d1 << 8) + d0
        b = s * ((top << 16) + (d1 << 8) - 127)
        A = np.full(T, a, dtype=object)
        B = np.full(T, b, dtype=object)
        A[::7] = -A[::7]
        X = np.array([A, B], dtype=np.float64) * 2.0 ** -16
        d2 = int(((A - B) ** 2).sum())                    # Python integers
        _, _, _, sg = G.graph(X)
        assert float(sg) == np.sqrt(np.float64(d2) * 2.0 ** -32)


@pytest.mark.parametrize("T", [64, 257, 300])
def test_batched_distances_on_every_route(G, T):
    """One batch with graphs on the grid (through the tensor cores; long series on small
    orders, whose digit planes have no room, through int64) and off it (float64)."""
    from test_gpu_batched import _check, _run
    from workloads import iid_pair
    pairs = []
    for p, n in enumerate((90, 127, 129, 200, 333)):
        X1, X2 = (np.array(x) for x in iid_pair(n, T, 3, 40 + p).X)
        if p % 2:
            X1 = X1 + 1e-7                                # X2 stays on the grid
        pairs.append(SimpleNamespace(X=(X1, X2)))
    F, tops, stats = _run(G, pairs, 10, 3, G.cdl.CDL_F64)
    _check(pairs, F, tops, stats, 3)
