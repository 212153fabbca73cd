"""Float64 and float32 chains on graphs whose degrees lie many orders of
magnitude apart: a node far from all others (a Gaussian kernel gives it weights
of 1e-10 to 1e-25), or weights that follow node strengths. The embedding of such
a node is about D^{-1/2}, up to 1e12 times the others', and the residual still
has to reach the tolerance."""
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


def _graph(kind, n, rng):
    w = np.triu(rng.uniform(0.5, 1.0, (n, n)), 1)
    if kind.startswith("far"):                     # node n // 2 hangs on weights of 10^-x
        w[n // 2] *= 10.0 ** -float(kind[3:])
        w[:, n // 2] *= 10.0 ** -float(kind[3:])
    else:                                          # strengths over x orders of magnitude
        s = 10.0 ** rng.uniform(-float(kind[8:]) / 2, 0, n)
        w *= np.outer(s, s)
    return w + w.T


@pytest.mark.parametrize("name", ["f64", "f32"])
@pytest.mark.parametrize("kind", ["far10", "far18", "far25", "strength10", "strength20"])
@pytest.mark.parametrize("n,k", [(65, 1), (300, 33), (1100, 16)])
def test_residual_reaches_the_tolerance(G, name, kind, n, k):
    cdl = G.cdl
    A = torch.from_numpy(_graph(kind, n, np.random.default_rng(n))).cuda()
    D, vol = A.sum(1), A.sum().reshape(1)
    Y = G.project(A, k, 3)
    ch = G.chain(A, D, vol, 8, {"f64": cdl.CDL_F64, "f32": cdl.CDL_F32}[name])
    try:
        Z, stats = G.solve(ch, A, Y, max_iter=8, rel_tol=1e-12)
    finally:
        cdl.cdl_chain_free(ch)
    a, z, y = (t.cpu().numpy().astype(np.longdouble) for t in (A, Z, Y))
    r = y - (a.sum(1)[:, None] * z - a @ z)
    # the float64 degrees of the caller are within n 2^-53 of the sums here: D Z carries that into the check
    slack = n * 2.0 ** -53 * np.linalg.norm((a.sum(1)[:, None] * np.abs(z)).astype(np.float64))
    assert stats.rel_res <= 1e-12
    assert np.linalg.norm(r.astype(np.float64)) <= 2e-12 * np.linalg.norm(Y.cpu().numpy()) + slack
