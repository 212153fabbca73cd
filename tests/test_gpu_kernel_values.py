"""Kernel values A_ij = exp(-d2_ij / (2 sigma^2)) and their degrees against
extended precision, over the exponent range and the edges of the 64-node tiles.
One-sample series on the 2^-16 grid make d2 an exact integer multiple of 2^-32.
The bound on A is that of the exponential (2.1e-15) plus the rounding of the
float64 factor 1 / (2 sigma^2) (three roundings) times the argument."""
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


@pytest.mark.parametrize("n", [2, 63, 64, 65, 129, 700])
@pytest.mark.parametrize("tmax", [1e-12, 1.0, 40.0, 700.0, 1e5])
def test_kernel_values(G, n, tmax):
    rng = np.random.default_rng(n)
    x = rng.integers(-2 ** 20, 2 ** 20, (n, 1)).astype(np.float64) * 2.0 ** -16
    x[n - 1] = x[0]                                       # a distance of zero
    d2 = ((x.astype(np.longdouble) - x.T) ** 2)
    sigma = float(np.sqrt(max(d2.max(), 1) / (2 * np.longdouble(tmax))))
    A, D, vol, _ = G.graph(x, sigma)
    A, D = A.cpu().numpy(), D.cpu().numpy()
    assert np.array_equal(A, A.T) and np.all(np.diag(A) == 0)
    assert A[0, n - 1] == 1.0
    t = d2 / (2 * np.longdouble(sigma) ** 2)
    ref = np.exp(-t)
    ref[np.arange(n), np.arange(n)] = 0
    err = np.abs(A - ref).astype(np.float64)
    tol = (2.1e-15 + 2.0 ** -53 + 3 * 2.0 ** -53 * t) * ref + np.longdouble(2.0) ** -1074
    assert np.all(err <= tol)
    # float-float sums: 2^-46 for each of the at most log-depth or 16-term partial sums
    assert np.all(np.abs(D - A.astype(np.longdouble).sum(1)) <= 64 * 2.0 ** -46 * A.sum(1) + n * 2.0 ** -100)
    assert abs(float(vol) - float(D.astype(np.longdouble).sum())) <= n * 2.0 ** -53 * float(D.sum())


def test_kernel_values_at_the_median(G):
    rng = np.random.default_rng(3)
    for n in (64, 65, 130):
        X = rng.integers(-2 ** 18, 2 ** 18, (n, 5)).astype(np.float64) * 2.0 ** -16
        A, D, _, s = G.graph(X)
        A = A.cpu().numpy().astype(np.longdouble)
        W = X.astype(np.longdouble)
        d2 = ((W[:, None] - W[None]) ** 2).sum(-1)
        iu = np.triu_indices(n, 1)
        m = np.sort(d2[iu])[(len(iu[0]) - 1) // 2]
        assert float(s) == float(np.sqrt(np.float64(m)))
        ref = np.exp(-d2 / (2 * np.longdouble(float(s)) ** 2))
        np.fill_diagonal(ref, 0)
        assert np.max(np.abs(A - ref)) <= 6e-15
