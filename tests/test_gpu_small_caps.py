"""Calls under workspace caps that leave room only for what the call cannot do
without: they run, with the same results up to the order of sums."""
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


class Capped:
    """A context with a cap of its own."""

    def __init__(self, G, cap):
        self.cdl = G.cdl
        st, self.h = G.cdl.cdl_ctx_create(0, torch.cuda.current_stream().cuda_stream, cap)
        assert st == 0

    def __enter__(self):
        return self.h

    def __exit__(self, *exc):
        assert self.cdl.cdl_ctx_destroy(self.h) == 0


# n above one split by the number of warps, above 4096 edges, and k of one and of two Philox blocks
@pytest.mark.parametrize("n,k", [(600, 32), (1000, 200), (5000, 16)])
@pytest.mark.parametrize("splits,more", [(0, 0), (2, 0), (2, -1)])
def test_projection(G, n, k, splits, more):
    """Only the column sums of the centring (one 256-row block per column), then room for `splits` partial sums, or
    for these alone, less a byte."""
    cdl = G.cdl
    A = G.graph(iid_pair(n, 8, 1, seed=n).X[0])[0]
    ref = G.project(A, k, 3)
    Y = torch.empty_like(ref)
    cap = (1 + more) * ((n + 255) // 256 + 1) * k * 8 + splits * n * k * 8 + more
    with Capped(G, cap) as h:
        assert cdl.cdl_project(h, A, cdl.CDL_F64, n, k, 3, Y) == 0
        assert cdl.cdl_sync(h) == 0
    # exact digit sums, one float64 rounding per split or chunk of 4096 edges
    np.testing.assert_allclose(Y.cpu().numpy(), ref.cpu().numpy(), rtol=0, atol=64 * 2.0 ** -53 * float(ref.abs().max()))


@pytest.mark.parametrize("name", ["f64", "f32"])
@pytest.mark.parametrize("n,k", [(20, 3), (130, 8), (700, 8)])
def test_edges(G, name, n, k):
    """The edge scores (8 n^2), the partial sums and the operand copies of the CUDA-core scores, counts and offsets
    per row, and 512 bytes; the cut search has no room of its own. Sums over as few as one block, and entries left
    over that take further passes, give the same set."""
    cdl = G.cdl
    g = [G.graph(iid_pair(n, 8, 2, seed=n).X[i]) for i in range(2)]
    rng = np.random.default_rng(n)
    Z = [torch.from_numpy(rng.standard_normal((n, k))).cuda() for _ in range(2)]
    nb = (n + 63) // 64
    cap = max(8 * nb * n, 17 * 24) + 8 * n * n + 8 * n + 8 * n + 16 * n + 16 + 16 * n * k + 16 * k + 512
    out = []
    for frac in (0.9, 0.2):
        for c in (0, cap):
            with Capped(G, c) as h:
                m = n * (n - 1) // 2
                F = torch.empty(n, dtype=torch.float64, device="cuda")
                v = (torch.ones(1, dtype=torch.float64, device="cuda"), torch.full((1,), 2.0, dtype=torch.float64,
                                                                                   device="cuda"))
                sd = cdl.CDL_F64 if name == "f64" else cdl.CDL_F32
                assert cdl.cdl_cad_score(G.h, g[0][0], g[1][0], cdl.CDL_F64, *Z, *v, n, k, sd, 0, F, None) == 0
                delta = frac * 0.5 * float(F.sum())
                ij = torch.full((m, 2), -1, dtype=torch.int64, device="cuda")
                de = torch.zeros(m, dtype=torch.float64, device="cuda")
                st, r = cdl.cdl_cad_edges(h, g[0][0], g[1][0], cdl.CDL_F64, *Z, *v, n, k, sd, delta, m, ij, de, None, 0,
                                          0, None, None, None)
                assert st == 0 and cdl.cdl_sync(h) == 0
                out.append((r.n_edges, ij.cpu().numpy()))
    for a, b in (out[:2], out[2:]):
        assert a[0] == b[0] > 0 and np.array_equal(a[1], b[1])


def _smallest_cap(cdl, call):
    """The smallest cap, to 256 bytes, under which call(ctx) returns CDL_OK."""
    lo, hi = 0, 1 << 30
    while hi - lo > 256:
        mid = (lo + hi) // 2
        st, h = cdl.cdl_ctx_create(0, torch.cuda.current_stream().cuda_stream, mid)
        assert st == 0
        lo, hi = (lo, mid) if call(h) == 0 else (mid, hi)
        assert cdl.cdl_ctx_destroy(h) == 0
    return hi


@pytest.mark.parametrize("n,T", [([20] * 6, 300), ([100, 130, 90], 600)])
def test_batch_of_series_too_long_for_digit_planes(G, n, T):
    """A plan without the tensor-core distances holds nothing for them: no tensor maps, and 64 bytes of selection
    state per graph, as the 32 KB histogram beside it, so every graph's share is a whole number of 64 bytes. The
    bound is the plan's size with none of it, counted for these two (measured before those distances came)."""
    cdl = G.cdl
    k, d = (4, 2) if len(n) == 6 else (16, 4)
    N = sum(n)
    rng = np.random.default_rng(N)
    X = [torch.from_numpy(np.round(rng.standard_normal((N, T)) * 65536) / 65536).cuda() for _ in range(2)]
    F = torch.empty(N, dtype=torch.float64, device="cuda")
    top = torch.empty((len(n), 2), dtype=torch.int64, device="cuda")
    o = cdl.cdl_batch_opts(k, d, cdl.CDL_BF16, cdl.CDL_F32, 3, 0.0, cdl.cdl_solve_opts(20, 1e-10, 0), 2, 0, 0)
    nn = np.array(n, dtype=np.int64)
    cap = _smallest_cap(cdl, lambda h: cdl.cdl_caddelag_batched(h, len(n), nn, T, X[0], X[1], o, F, top, None))
    assert cap <= {6: 15028224, 3: 16943104}[len(n)]


@pytest.mark.parametrize("name", ["f64", "f32"])
def test_the_same_call_gives_the_same_bits_whatever_ran_before(G, name):
    """Residue planes of an earlier solve stand in the room that the scores' planes need under this cap: they are
    given up for them at once, so the first call and the second take the same form and give the same bits, those
    of a context of their own."""
    cdl = G.cdl
    n, npad, k, ks = 300, 512, 8, 1024
    dtype = cdl.CDL_F64 if name == "f64" else cdl.CDL_F32
    A, D, vol, _ = G.graph(iid_pair(n, 8, 1, seed=4).X[0])
    A2 = G.graph(iid_pair(n, 8, 1, seed=5).X[0])[0]
    Y = G.project(A, k, 3)
    rng = np.random.default_rng(1)
    Z = [torch.from_numpy(rng.standard_normal((n, ks))).cuda() for _ in range(2)]
    planes = 16 if name == "f64" else 13
    # the scores' planes (rows padded to 128, 2 ks columns), their small buffers, and half of the solve's planes
    cap = 2 * planes * 384 * 2 * ks * 2 + 2 * 8 * 5 * n + (1 << 20) + 16 * npad * npad

    def score(h):
        F = torch.empty(n, dtype=torch.float64, device="cuda")
        assert cdl.cdl_cad_score(h, A, A2, cdl.CDL_F64, Z[0], Z[1], vol, vol, n, ks, dtype, 0, F, None) == 0
        assert cdl.cdl_sync(h) == 0
        return F

    with Capped(G, cap) as h:
        alone = score(h)
    with Capped(G, cap) as h:
        st, ch = cdl.cdl_chain_build(h, A, cdl.CDL_F64, D, vol, n, 2, cdl.CDL_F64)
        assert st == 0
        Zs = torch.empty((n, k), dtype=torch.float64, device="cuda")
        assert cdl.cdl_chain_solve(h, ch, A, cdl.CDL_F64, Y, k, cdl.cdl_solve_opts(40, 1e-10, 0), Zs, None) == 0
        first, second = score(h), score(h)
        cdl.cdl_chain_free(ch)
    assert torch.equal(first, second) and torch.equal(first, alone)


@pytest.mark.parametrize("name,elem", [("f64", 8), ("f32", 4)])
def test_solve_of_many_columns(G, name, elem):
    """One level and k far above n: the solve's buffers are what the cap has to hold. Residual, iterate and its
    partial products, Z as float pairs and dZ, and 64 KB for the rest; no room of its own for the centring (17 rows
    of 1024 column sums, 139 KB)."""
    cdl = G.cdl
    n, npad, k = 300, 512, 1024
    A, D, vol, _ = G.graph(iid_pair(n, 8, 1, seed=6).X[0])
    Y = G.project(A, k, 3)
    dtype = cdl.CDL_F64 if name == "f64" else cdl.CDL_F32

    def call(h):
        st, ch = cdl.cdl_chain_build(h, A, cdl.CDL_F64, D, vol, n, 1, dtype)
        if st == 0:
            Z = torch.empty((n, k), dtype=torch.float64, device="cuda")
            st = cdl.cdl_chain_solve(h, ch, A, cdl.CDL_F64, Y, k, cdl.cdl_solve_opts(60, 1e-9, 0), Z, None)
            cdl.cdl_sync(h)
            cdl.cdl_chain_free(ch)
        return st

    # the partial products: with 152 SMs (npad / 64 or / 128) x 16 tiles leave room for 9 or 16 splits, 8 or 16 of
    # the 64 blocks of K each
    splits = {"f64": 8, "f32": 16}[name]
    bound = n * k * 8 + npad * k * elem * (1 + splits) + 2 * n * k * 4 + npad * k * 4 + (1 << 16)
    assert _smallest_cap(cdl, call) <= bound
