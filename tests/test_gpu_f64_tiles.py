"""The float64 form's tiled kernel at the edges of its tiles (8, 16, 32, 64, by
problem size), its K blocks (16) and offset chunks (256), with and without K
ranges: float64 sums in another order, within 2 (K + 2) eps of |u| |v|."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [(9, 9, 1), (16, 17, 15), (31, 9, 255), (48, 48, 257), (65, 130, 513), (200, 90, 31), (9, 600, 2000),
         (129, 1000, 300), (300, 300, 1000), (700, 900, 700)]


@pytest.fixture(scope="module")
def sc():
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a visible GPU")
    import paper_2007_08056_gb300 as mod
    mod.load()
    return mod


@pytest.mark.parametrize("flip", [False, True], ids=["columns", "rows"])
@pytest.mark.parametrize("G", [1, 3])
@pytest.mark.parametrize("M,N,K", SIZES)
def test_tiles(sc, M, N, K, G, flip):
    """`flip`: operands stored with their rows as the unit-stride side."""
    rng = np.random.default_rng(M + N + K)
    es, du, dv = ("ji,kj->ik", (K, M), (N, K)) if flip else ("ij,jk->ik", (M, K), (K, N))
    p = sc.Plan(es, (G,), ((1, -1), (0,), du), ((1, -1), (0,), dv), "fp64")
    u, v = rng.standard_normal(p.shape_u), rng.standard_normal(p.shape_v)
    w = p.contract(torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()).cpu().numpy()
    p.check_device_error()
    for q in range(G):
        a, b = (u[q].T, v[q].T) if flip else (u[q], v[q])
        want = a @ b
        assert np.all(np.abs(w[q] - want) <= 2 * (K + 2) * 2.0 ** -53 * (np.abs(a) @ np.abs(b)))
