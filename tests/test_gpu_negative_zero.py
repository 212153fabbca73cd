"""Absent edges written as -0.0: a program that has the Laplacian forms A = -L
with a zeroed diagonal, and every pair without an edge (and the diagonal) is
then -0.0, a finite, non-negative weight like 0.0."""
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


def _graphs(n, seed):
    """The same sparse weights with absent edges as 0.0 and as -0.0."""
    rng = np.random.default_rng(seed)
    a = rng.uniform(0.1, 1.0, (n, n)) * (rng.random((n, n)) < 0.3)
    a[np.arange(n - 1), np.arange(1, n)] = 0.5          # connected
    a = np.triu(a, 1)
    a = torch.from_numpy(a + a.T).cuda()
    b = torch.where(a == 0, torch.full_like(a, -0.0), a)
    assert torch.equal(torch.signbit(b), a == 0)
    return a, b


# one chunk of edges per warp, several, a chunk of 4096 and a part of the next; one word of signs, and all four
@pytest.mark.parametrize("n,k", [(2, 1), (200, 7), (700, 33), (700, 130), (5000, 16)])
def test_projection(G, n, k):
    a, b = _graphs(n, n)
    ya, yb = G.project(a, k, 5), G.project(b, k, 5)
    assert torch.equal(ya, yb) and torch.isfinite(ya).all() and bool(ya.any())


def test_projection_ignores_the_diagonal(G):
    a, _ = _graphs(300, 1)
    d = a.clone()
    d.fill_diagonal_(2.0 ** 60)
    assert torch.equal(G.project(a, 16, 5), G.project(d, 16, 5))


@pytest.mark.parametrize("name", ["f64", "f32"])
def test_solve_without_workspace(G, name):
    """The float-float residual, which runs where the cap leaves no room for the residue planes (32 npad^2 bytes)."""
    cdl = G.cdl
    n, npad, k, d = 300, 512, 8, 2
    dtype, elem = {"f64": (cdl.CDL_F64, 8), "f32": (cdl.CDL_F32, 4)}[name]
    cap = d * elem * npad * npad + 8 * n * n + (1 << 18)
    assert cap < 32 * npad * npad
    Zs = []
    for A in _graphs(n, 3):
        D, vol = A.sum(1), A.sum().reshape(1)
        Y = G.project(_graphs(n, 3)[0], k, 5)
        st, h = cdl.cdl_ctx_create(0, torch.cuda.current_stream().cuda_stream, cap)
        assert st == 0
        st, ch = cdl.cdl_chain_build(h, A, cdl.CDL_F64, D, vol, n, d, dtype)
        assert st == 0
        Z = torch.empty((n, k), dtype=torch.float64, device="cuda")
        assert cdl.cdl_chain_solve(h, ch, A, cdl.CDL_F64, Y, k, cdl.cdl_solve_opts(60, 1e-10, 0), Z, None) == 0
        assert cdl.cdl_sync(h) == 0
        Zs.append(Z)
        cdl.cdl_chain_free(ch)
        assert cdl.cdl_ctx_destroy(h) == 0
    assert torch.equal(*Zs)
