"""The cut search of the anomalous edge set at the bottom of the float64 range,
where its windows of 16 binades meet key 0: scores of 2^-1003 and below,
subnormal ones among them, with the cut under a window that overlaps the one
before it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import caddelag as O   # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from gpu_util import Ctx, lib
    g = Ctx(lib())
    yield g
    g.close()


# exponents of the one largest score, of fifty in the overlap and of all others
@pytest.mark.parametrize("top,mid,low", [(-1003, -1013, -1021), (-990, -1012, -1030), (-1003, -1018, -1024),
                                         (-1010, -1015, -1022)])
@pytest.mark.parametrize("frac", [0.999, 0.5, 1e-3])
def test_cut_below_the_overlap(G, top, mid, low, frac):
    cdl = G.cdl
    n = 200
    iu, ju = np.triu_indices(n, 1)
    e = np.full(iu.size, 2.0 ** low)
    e[77] = 2.0 ** top
    e[100:150] = 2.0 ** mid
    A1 = np.zeros((n, n))
    A1[iu, ju] = 0.5 * e
    A1 += A1.T
    Z2 = np.eye(n)                     # every commute-time change is 2, Delta E is 2 |A1 - A2|
    E = np.zeros((n, n))
    E[iu, ju] = e
    delta = frac * (iu.size - 51) * 2.0 ** low
    out = O.anomalous_edges(E, delta)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A1, 0 * A1, 0 * Z2, Z2)]
    v = torch.ones(1, dtype=torch.float64, device="cuda")
    ij = torch.full((iu.size, 2), -7, dtype=torch.int64, device="cuda")
    val = torch.zeros(iu.size, dtype=torch.float64, device="cuda")
    st, res = cdl.cdl_cad_edges(G.h, t[0], t[1], cdl.CDL_F64, t[2], t[3], v, v, n, n, cdl.CDL_F64, delta, iu.size, ij,
                                val, None, 0, 0, None, None, None)
    G.check(st)
    assert res.n_edges == len(out["edges"]) and res.remaining < delta
    assert np.array_equal(ij[:res.n_edges].cpu().numpy(), out["edges"])
    assert res.threshold == 2.0 ** low
