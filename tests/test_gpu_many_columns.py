"""Solves with many more right-hand sides than nodes, one column, and edges of the
32-column tiles in which the iterate is updated and centred."""
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


@pytest.mark.parametrize("name", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("n,k", [(65, 1), (64, 31), (64, 33), (65, 1024), (300, 640)])
def test_every_column_is_solved_and_centred(G, name, n, k):
    cdl = G.cdl
    A, D, vol, _ = G.graph(iid_pair(n, 16, 1, seed=n).X[0])
    Y = G.project(A, k, 3)
    ch = G.chain(A, D, vol, 6, {"f64": cdl.CDL_F64, "f32": cdl.CDL_F32, "bf16": cdl.CDL_BF16}[name])
    try:
        Z, _ = G.solve(ch, A, Y, max_iter=60, rel_tol=1e-11)
    finally:
        cdl.cdl_chain_free(ch)
    d, y, z = D.cpu().numpy(), Y.cpu().numpy(), Z.cpu().numpy()
    L = np.diag(d) - A.cpu().numpy()
    # the whole of Y to the tolerance (blocks of 128 columns each to theirs), so each column to that times ||Y||
    assert np.linalg.norm(y - L @ z) <= 2e-11 * np.linalg.norm(y)
    # D-weighted column means: a float64 sum of n products, subtracted once
    assert np.all(np.abs(d @ z) <= 4 * n * 2.0 ** -53 * (d @ np.abs(z)) + 1e-300)
