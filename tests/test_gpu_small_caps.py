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
@pytest.mark.parametrize("splits", [0, 2])
@pytest.mark.parametrize("more", [0, -1])
def test_projection(G, n, k, splits, more):
    """Only the column sums of the centring (one 256-row block per column), then room for `splits` partial sums, or
    for these alone, less a byte."""
    if splits == 0 and more:
        pytest.skip("nothing to leave out")
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
