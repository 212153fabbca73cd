"""Float64 and float32 chain squarings through residues on the tensor cores:
level i + 1 against the exact square of the stored level i, at the edges of
the 256-blocks and of the 1024-wide exact chunks, for magnitudes down to
underflow, for non-finite levels, and against the CUDA-core form that runs
when the workspace is not to be had."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from workloads import iid_pair   # noqa: E402

pytestmark = pytest.mark.gpu

# unit roundoff; a bound on the rows' rounding, half a unit of 2^-59.9 (16 moduli) or 2^-29.5 (8) of the row
# norm at most per entry (errors of one sign in every entry do not occur)
TYPES = {"f64": (np.float64, 2.0 ** -53, 2.0 ** -60), "f32": (np.float32, 2.0 ** -24, 2.0 ** -29)}


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from gpu_util import Ctx, lib
    g = Ctx(lib())
    yield g
    g.close()


def _dtype(cdl, name):
    return {"f64": cdl.CDL_F64, "f32": cdl.CDL_F32}[name]


def _levels(G, n, d, name, seed=0):
    A, D, vol, _ = G.graph(iid_pair(n, 8, 1, seed=seed).X[0])
    ch = G.chain(A, D, vol, d, _dtype(G.cdl, name))
    try:
        return [G.level(ch, i, TYPES[name][0]).cpu().numpy().copy() for i in range(d)]
    finally:
        G.cdl.cdl_chain_free(ch)


def _check_square(S, C, name, rows):
    """Rows `rows` of C against S S in extended precision (63 bits or more)."""
    _, u, unit = TYPES[name]
    n = S.shape[0]
    scale = np.abs(S).max() or 1.0
    W = (S.astype(np.longdouble)) / np.longdouble(scale)
    R = W[rows] @ W
    norm = np.sqrt((W * W).sum(1)).astype(np.float64)
    got = C[rows].astype(np.longdouble) / np.longdouble(scale) / np.longdouble(scale)
    bound = u * np.abs(R).astype(np.float64) + np.sqrt(n) * unit * norm[rows][:, None] * norm[None, :] + 1e-300
    assert np.all(np.abs(got - R).astype(np.float64) <= bound)


@pytest.mark.parametrize("name", ["f64", "f32"])
@pytest.mark.parametrize("n", [2, 63, 256, 257, 1023, 1025, 2100])
def test_square_is_exact_to_one_rounding(G, name, n):
    L = _levels(G, n, 3, name, seed=n)
    rows = np.unique(np.r_[0, 1, n // 2, n - 1, np.random.default_rng(n).integers(0, n, 8)])
    for i in range(2):
        _check_square(L[i], L[i + 1], name, rows)
        assert np.array_equal(L[i + 1], L[i + 1].T)
        assert not L[i + 1][n:].any()


@pytest.mark.parametrize("name", ["f64", "f32"])
def test_levels_underflow_to_zero(G, name):
    """Well-connected graphs' levels decay like lambda^(2^i): every level stays finite, and the last are zero."""
    L = _levels(G, 300, 12, name)
    big = [float(np.abs(x).max()) for x in L]
    assert all(np.isfinite(x).all() for x in L) and big[-1] == 0.0
    for a, b in zip(big, big[1:]):
        assert b <= a


@pytest.mark.parametrize("name", ["f64", "f32"])
def test_non_finite_level_stays_non_finite(G, name):
    cdl = G.cdl
    A, D, vol, _ = G.graph(iid_pair(300, 8, 1, seed=1).X[0])
    A[7] = 0
    A[:, 7] = 0
    D[7] = 0                                          # a node without neighbours: D^(-1/2) is infinite
    ch = G.chain(A, D, vol, 2, _dtype(cdl, name))
    try:
        S, C = (G.level(ch, i, TYPES[name][0]).cpu().numpy() for i in range(2))
    finally:
        cdl.cdl_chain_free(ch)
    assert np.isnan(S).any() and np.array_equal(np.isnan(C), np.isnan(S @ S))   # 0 NaN is NaN: the padding too


@pytest.mark.parametrize("name", ["f64", "f32"])
def test_without_workspace_the_cuda_core_form_runs(G, name):
    cdl = G.cdl
    n, npad = 600, 768
    A, D, vol, _ = G.graph(iid_pair(n, 8, 1, seed=2).X[0])
    elem = np.dtype(TYPES[name][0]).itemsize
    cap = 2 * npad * npad * elem + 12 * npad * npad + (1 << 20)   # the chain and the small buffers only
    st, h = cdl.cdl_ctx_create(0, torch.cuda.current_stream().cuda_stream, cap)
    assert st == 0
    out = []
    for ctx in (G.h, h):
        st, ch = cdl.cdl_chain_build(ctx, A, cdl.CDL_F64, D, vol.data_ptr(), n, 2, _dtype(cdl, name))
        assert st == 0 and cdl.cdl_sync(ctx) == 0
        out.append(G.level(ch, 1, TYPES[name][0]).cpu().numpy().copy())
        cdl.cdl_chain_free(ch)
    assert cdl.cdl_ctx_destroy(h) == 0
    S = _levels(G, n, 1, name, seed=2)[0].astype(np.float64)
    bound = n * TYPES[name][1] * 2 * (np.abs(S) @ np.abs(S)) + 1e-300
    assert np.all(np.abs(out[0].astype(np.float64) - out[1]) <= bound)
    assert not np.array_equal(out[0], out[1])          # two forms did run


@pytest.mark.parametrize("name", ["f64", "f32"])
@pytest.mark.parametrize("n,k", [(3, 1), (257, 65), (600, 16), (300, 300)])
def test_solve_with_and_without_workspace(G, name, n, k):
    """The exact-product applies and residuals against the forms that run under a workspace cap too small
    for them: both solutions meet the tolerance, so they agree to it (times the graph's condition)."""
    cdl = G.cdl
    npad = (n + 255) // 256 * 256
    A, D, vol, _ = G.graph(iid_pair(n, 16, 1, seed=n).X[0])
    Y = G.project(A, k, 3)
    elem = np.dtype(TYPES[name][0]).itemsize
    cap = 4 * npad * npad * elem + 8 * n * n + 300 * npad * k + (1 << 18)
    st, h = cdl.cdl_ctx_create(0, torch.cuda.current_stream().cuda_stream, cap)
    assert st == 0
    Zs = []
    for ctx in (G.h, h):
        st, ch = cdl.cdl_chain_build(ctx, A, cdl.CDL_F64, D, vol.data_ptr(), n, 4, _dtype(cdl, name))
        assert st == 0
        Z = torch.empty((n, k), dtype=torch.float64, device="cuda")
        stats = cdl.cdl_solve_stats()
        assert cdl.cdl_chain_solve(ctx, ch, A, cdl.CDL_F64, Y, k, cdl.cdl_solve_opts(60, 1e-12, 0), Z, stats) == 0
        assert cdl.cdl_sync(ctx) == 0 and stats.rel_res <= 1e-12
        Zs.append(Z.cpu().numpy())
        cdl.cdl_chain_free(ch)
    assert cdl.cdl_ctx_destroy(h) == 0
    L = np.diag(D.cpu().numpy()) - A.cpu().numpy()
    for Z in Zs:
        assert np.linalg.norm(Y.cpu().numpy() - L @ Z) <= 3e-12 * np.linalg.norm(Y.cpu().numpy())
    assert np.linalg.norm(Zs[0] - Zs[1]) <= 1e-10 * np.linalg.norm(Zs[0])


@pytest.mark.parametrize("name,tol", [("f64", 1e-12), ("f32", 1e-10)])
@pytest.mark.parametrize("n,k", [(2, 1), (65, 33), (129, 16), (300, 200), (130, 1024)])
def test_scores_with_and_without_workspace(G, name, tol, n, k):
    """Residue scores against the CUDA-core ones that run under a workspace cap too small for the planes,
    with rows of very different scales, a node without an embedding, and equal embeddings."""
    cdl = G.cdl
    rng = np.random.default_rng(n + k)
    A = [rng.uniform(0, 1, (n, n)) for _ in range(2)]
    A = [torch.from_numpy(np.triu(a, 1) + np.triu(a, 1).T).cuda() for a in A]
    Z1 = rng.standard_normal((n, k)) * 10.0 ** rng.uniform(-3, 0, (n, 1))
    Z2 = Z1 + 0.05 * rng.standard_normal((n, k)) * np.abs(Z1)
    Z1[n // 2] = Z2[n // 2] = 0
    Z2[n - 1] = Z1[n - 1]
    Zt = [torch.from_numpy(z).cuda() for z in (Z1, Z2)]
    vol = [torch.full((1,), v, dtype=torch.float64, device="cuda") for v in (3.0, 4.0)]
    nb = (n + 63) // 64
    cap = 32 * n * k + 8 * nb * n + 4 * n + 16 * k + 8192       # the float planes and the partial sums only
    st, h = cdl.cdl_ctx_create(0, torch.cuda.current_stream().cuda_stream, cap)
    assert st == 0
    Fs = []
    for ctx in (G.h, h):
        F = torch.empty(n, dtype=torch.float64, device="cuda")
        top = torch.empty(2, dtype=torch.int64, device="cuda")
        st = cdl.cdl_cad_score(ctx, A[0], A[1], cdl.CDL_F64, Zt[0], Zt[1], vol[0], vol[1], n, k, _dtype(cdl, name), 2,
                               F, top)
        assert st == 0 and cdl.cdl_sync(ctx) == 0
        Fs.append(F.cpu().numpy())
    assert cdl.cdl_ctx_destroy(h) == 0
    np.testing.assert_allclose(Fs[0], Fs[1], rtol=tol, atol=tol * Fs[1].max())
