"""Off-grid distances where the first node is an outlier or not finite: the other
nodes' distances still come from the residue form. Its squared distances are
correctly rounded but for 2^-5 of a unit (about 2^-59 relative), so the median
distance is within 2^-54 (1 + 2^-5) + 2^-53 of the exact one, relative; a float64
sum of 2000 squares is off by several units."""
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
    X[1:64] *= 5.0                     # the first 64 x 64 blocks hold no median distance
    if kind == "fill":
        X[0] = -9999.0
    elif kind == "fill_in_two":        # of the five nodes that the common series comes from
        X[0] = X[(n - 1) // 2] = 1e15
    elif kind == "nan":
        X[0, T // 2] = np.nan
    elif kind == "inf":
        X[0] = np.inf
    return X


@pytest.mark.parametrize("kind", ["plain", "fill", "fill_in_two", "nan", "inf"])
@pytest.mark.parametrize("seed", range(4))
def test_median_distance_is_correctly_rounded(G, kind, seed):
    n, T = 640, 2000
    X = _series(kind, n, T, np.random.default_rng(seed))
    iu, ju = np.triu_indices(n, 1)
    sq = (X * X).sum(1)
    with np.errstate(invalid="ignore"):
        d2 = sq[:, None] + sq[None, :] - 2 * X @ X.T
    far = ~np.isfinite(d2[iu, ju])     # non-finite distances sort last
    order = np.argsort(np.where(far, np.inf, d2[iu, ju]), kind="stable")
    rank = (iu.size - 1) // 2
    near = order[rank - 100:rank + 101]
    W = X.astype(np.longdouble)
    exact = np.sort(((W[iu[near]] - W[ju[near]]) ** 2).sum(1))[100]
    sigma = float(G.graph(X)[3].item())
    err = abs(np.longdouble(sigma) / np.sqrt(exact) - 1)
    assert err <= (0.5 * (1 + 2.0 ** -5) + 1) * 2.0 ** -53
