"""Graphs of float64 series on no grid: the residue distances (16 samples and
more) and the entries they leave to the float64 kernel, against extended
precision. A float64 sum of T rounded squares is within (T + 2) 2^-53 of its
value, relative; the residue form promises less, so that bound holds for both."""
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


def _series(kind, n, T, rng):
    X = rng.standard_normal((n, T))
    if kind == "offset":            # a large common level (temperatures in kelvin, pressures)
        X = 1013.25 + 4.0 * X
    elif kind == "duplicates":      # equal and nearly equal series, and one equal to node 0
        X[n // 2] = X[1]
        X[n // 3] = X[2 % n] * (1 + 1e-9)
        X[n - 1] = X[0]
    elif kind == "outlier":         # fill values in a few stations
        X[n // 2] = -9999.0
        X[n // 3, ::3] = 1e15
    elif kind == "scales":          # nodes of very different magnitudes
        X *= 10.0 ** rng.uniform(-8, 8, (n, 1))
    elif kind == "tiny":
        X *= 1e-140
    return X


def _d2(X, rows):
    W = X.astype(np.longdouble)
    return np.stack([((W[i] - W) ** 2).sum(1) for i in rows])


@pytest.mark.parametrize("n,T", [(2, 16), (64, 17), (129, 64), (300, 1024), (257, 1025), (640, 100)])
@pytest.mark.parametrize("kind", ["plain", "offset", "duplicates", "outlier", "scales"])
def test_graph_of_series_on_no_grid(G, kind, n, T):
    X = _series(kind, n, T, np.random.default_rng(n * T))
    rows = np.unique(np.r_[0, 1, n // 3, n // 2, n - 1])
    d2 = _d2(X, rows)
    sigma = float(np.sqrt(np.median(d2[-1].astype(np.float64)))) or 1.0
    A, D, vol, sg = G.graph(X, sigma)
    A = A.cpu().numpy()
    assert np.array_equal(A, A.T)
    t = d2 / (2 * np.longdouble(sigma) ** 2)
    ref = np.exp(-t)
    ref[np.arange(len(rows)), rows] = 0
    eps = 2e-14 + (T + 6) * 2.0 ** -53 * t.astype(np.float64)      # the exponential's bar and the argument's
    ok = t < 650
    assert np.all(np.abs(A[rows] - ref)[ok] <= (eps * ref.astype(np.float64))[ok])
    assert np.all(A[rows][~ok] <= 1e-280)


@pytest.mark.parametrize("kind", ["plain", "offset", "duplicates", "tiny"])
def test_median_distance_on_no_grid(G, kind):
    n, T = 200, 33
    X = _series(kind, n, T, np.random.default_rng(5))
    iu = np.triu_indices(n, 1)
    d = np.sort(np.sqrt(_d2(X, range(n))[iu]))
    exact = float(d[(len(d) - 1) // 2])
    sg = float(G.graph(X)[3].item())
    assert abs(sg - exact) <= (T + 6) * 2.0 ** -53 * exact


def test_non_finite_series_leaves_the_others_alone(G):
    X = np.random.default_rng(6).standard_normal((150, 40))
    other = np.delete(np.arange(150), 70)
    ref = G.graph(X[other], 4.0)[0].cpu().numpy()
    X[70, 3] = np.nan
    A = G.graph(X, 4.0)[0].cpu().numpy()
    np.testing.assert_allclose(A[np.ix_(other, other)], ref, rtol=5e-14)
