"""Embeddings that are equal, or opposite, under equal volumes score exactly 0: a (or b)
is 0 whatever the rounding of sqrt(vol) Z."""
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


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("name", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("n,k", [(2, 1), (140, 9), (257, 65)])
def test_score_is_zero(G, n, k, name, sign):
    cdl = G.cdl
    rng = np.random.default_rng(n + k)
    Z = rng.standard_normal((n, k))
    Z[0, 0] = 0.0
    A = np.triu(rng.uniform(0.1, 1.0, (n, n)), 1)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A + A.T, 0 * A, Z, sign * Z)]
    v = [torch.full((1,), 3.0, dtype=torch.float64, device="cuda") for _ in range(2)]
    F, _ = G.score(*t, *v, 0, {"f64": cdl.CDL_F64, "f32": cdl.CDL_F32, "bf16": cdl.CDL_BF16}[name])
    assert not F.cpu().numpy().any()
