"""Scores and edge scores of embeddings whose rows lie far apart in size: nodes of
tiny degree have embeddings up to 1e12 times the others', and a change that is
small beside them must not cost the other nodes' scores their bits."""
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


def _case(kind, n, k, rng):
    """Z1, Z2 and |A1 - A2|; the odd nodes' own edges do not change."""
    Z1 = rng.standard_normal((n, k))
    P = 0.1 * rng.standard_normal((n, k))
    odd = np.zeros(n, dtype=bool)
    if kind != "plain":
        odd[[n // 3, n - 1]] = True
    if kind == "far":             # huge embeddings, equal to 12 digits
        Z1[odd] *= 1e9
        P[odd] *= 1e-2
    elif kind == "far_flipped":   # huge, of opposite sign in the two graphs
        Z1[odd] *= 1e9
        P[odd] = -2 * Z1[odd] + 1e-3 * rng.standard_normal((odd.sum(), k))
    elif kind == "tiny":          # tiny embeddings that change by their own size, the others by 1e-6
        P[~odd] *= 1e-5
        Z1[odd] *= 1e-9
        P[odd] = Z1[odd]
    dA = np.triu(rng.uniform(0.1, 1.0, (n, n)), 1)
    dA[odd] = 0
    dA[:, odd] = 0
    return Z1, Z1 + P, dA + dA.T, odd


def _exact(Z1, Z2, v1, v2, dA):
    L = np.longdouble
    s1, s2 = np.sqrt(L(v1)), np.sqrt(L(v2))
    a, b = s2 * Z2.astype(L) - s1 * Z1.astype(L), s2 * Z2.astype(L) + s1 * Z1.astype(L)
    F, mag = np.zeros(len(a), L), np.zeros(len(a), L)
    for i in range(len(a)):
        p = (a[i] - a) * (b[i] - b)
        F[i] = (dA[i] * np.abs(p.sum(1))).sum()
        # the size of what the caller's float64 Z, scaled and combined, leaves undecided
        mag[i] = (dA[i] * ((np.abs(b[i]) + np.abs(b)) * np.abs(b[i] - b) + (np.abs(b[i]) + np.abs(b)) *
                           np.abs(a[i] - a)).sum(1)).sum()
    return F, mag


@pytest.mark.parametrize("kind", ["plain", "far", "far_flipped", "tiny"])
@pytest.mark.parametrize("vols", [(3.0, 3.0), (1.0, 4.0), (3.0, 3.0003)])
@pytest.mark.parametrize("n,k", [(70, 8), (200, 64), (130, 300)])
def test_float64_scores(G, kind, vols, n, k):
    """a and b come from three roundings of entries of their row's size (2^-52 of it at most together), the
    residue form adds less, and the sums over k and n are of rounded terms: 4 units of 2^-53 on `mag`."""
    cdl = G.cdl
    Z1, Z2, dA, odd = _case(kind, n, k, np.random.default_rng(n + k))
    F, mag = _exact(Z1, Z2, *vols, dA)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (dA, np.zeros_like(dA), Z1, Z2)]
    v = [torch.full((1,), x, dtype=torch.float64, device="cuda") for x in vols]
    got, _ = G.score(t[0], t[1], t[2], t[3], v[0], v[1], 0, cdl.CDL_F64)
    err = np.abs(got.cpu().numpy() - F).astype(np.float64)
    assert np.all(err <= 4 * 2.0 ** -53 * mag.astype(np.float64) + n * 2.0 ** -53 * F.astype(np.float64))
