"""The forms that run where a workspace cap leaves no room for the residue planes
against those that run with them: under the smallest cap that the call is accepted
with, the other form is taken (the launch counts say so) and meets the same bounds.
Shapes at the edges of the CUDA-core kernels' tiles: one, two and more than two
64-column tiles, more columns than rows, odd orders."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from workloads import iid_pair   # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from gpu_util import Ctx, lib
    g = Ctx(lib())
    yield g
    g.close()


def _with_cap(cdl, cap, call):
    st, h = cdl.cdl_ctx_create(0, torch.cuda.current_stream().cuda_stream, cap)
    assert st == 0
    try:
        return call(h)
    finally:
        assert cdl.cdl_ctx_destroy(h) == 0


def _smallest_cap(cdl, call):
    lo, hi = 0, 1 << 31
    while hi - lo > 256:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if _with_cap(cdl, mid, call) == 0 else (mid, hi)
    return hi


def _dtype(cdl, name):
    return {"f64": cdl.CDL_F64, "f32": cdl.CDL_F32}[name]


@pytest.mark.parametrize("name", ["f64", "f32"])
@pytest.mark.parametrize("n,k", [(65, 1), (257, 65), (600, 16), (300, 300), (130, 1024)])
def test_solve(G, name, n, k):
    cdl = G.cdl
    d = 3
    A, D, vol, _ = G.graph(iid_pair(n, 16, 1, seed=n).X[0])
    Y = G.project(A, k, 3)
    out = {}

    def call(h, keep=None):
        st, ch = cdl.cdl_chain_build(h, A, cdl.CDL_F64, D, vol, n, d, _dtype(cdl, name))
        if st != 0:
            return st
        Z, stats = torch.empty((n, k), dtype=torch.float64, device="cuda"), cdl.cdl_solve_stats()
        assert cdl.cdl_ctx_reset_counters(h) == 0
        o = cdl.cdl_solve_opts(60, 1e-12, cdl.CDL_SOLVE_FULL_RESIDUAL)
        st = cdl.cdl_chain_solve(h, ch, A, cdl.CDL_F64, Y, k, o, Z, stats)
        assert cdl.cdl_sync(h) == 0
        if keep:
            out[keep] = (Z.cpu().numpy(), stats.iters, cdl.cdl_ctx_timing(h, cdl.CDL_KC_RESIDUAL)[2],
                         cdl.cdl_ctx_timing(h, cdl.CDL_KC_APPLY)[2])
        assert cdl.cdl_chain_free(ch) == 0
        return st

    cap = _smallest_cap(cdl, call)
    assert _with_cap(cdl, 0, lambda h: call(h, "residues")) == 0
    assert _with_cap(cdl, cap, lambda h: call(h, "capped")) == 0
    Z, it, res, app = out["residues"]
    assert (res, app) == ((3 * it, 2 * d * it) if name == "f64" else (1 + 2 * it, d * it))
    Zc, itc, resc, appc = out["capped"]
    assert (resc, appc) == (1 + itc, d * itc)          # one split of A, one launch a step; one product a level
    L = np.diag(D.cpu().numpy()) - A.cpu().numpy()
    y = Y.cpu().numpy()
    for z in (Z, Zc):
        assert np.linalg.norm(y - L @ z) <= 3e-12 * np.linalg.norm(y)
    assert np.linalg.norm(Z - Zc) <= 1e-10 * np.linalg.norm(Z)


@pytest.mark.parametrize("name,tol", [("f64", 1e-12), ("f32", 1e-10)])
@pytest.mark.parametrize("n,k", [(2, 1), (65, 33), (300, 200), (130, 1024)])
def test_scores(G, name, tol, n, k):
    cdl = G.cdl
    rng = np.random.default_rng(n + k)
    A = [np.triu(rng.uniform(0, 1, (n, n)), 1) for _ in range(2)]
    A = [torch.from_numpy(a + a.T).cuda() for a in A]
    Z1 = rng.standard_normal((n, k))
    Z = [torch.from_numpy(z).cuda() for z in (Z1, Z1 + 0.05 * rng.standard_normal((n, k)))]
    vol = [torch.full((1,), v, dtype=torch.float64, device="cuda") for v in (3.0, 4.0)]
    out = []

    def call(h, keep=False):
        F = torch.empty(n, dtype=torch.float64, device="cuda")
        st = cdl.cdl_cad_score(h, A[0], A[1], cdl.CDL_F64, *Z, *vol, n, k, _dtype(cdl, name), 0, F, None)
        assert cdl.cdl_sync(h) == 0
        if keep:
            out.append((F.cpu().numpy(), cdl.cdl_ctx_timing(h, cdl.CDL_KC_MISC)[2]))
        return st

    cap = _smallest_cap(cdl, call)
    for c in (0, cap):
        assert _with_cap(cdl, c, lambda h: call(h, True)) == 0
    # maxima, residues and the sums of the partials; operands (float32: after the columns' maxima) and the sums
    assert (out[0][1], out[1][1]) == (3, 2 if name == "f64" else 3)
    if name == "f32":
        assert not np.array_equal(out[0][0], out[1][0]) or n == 2
    np.testing.assert_allclose(out[0][0], out[1][0], rtol=tol, atol=tol * out[1][0].max())
