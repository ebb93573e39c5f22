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


@pytest.mark.parametrize("M,N,K,G", [(24, 24, 1500, 2), (48, 48, 1024, 3), (300, 300, 1800, 3), (200, 200, 800, 1),
                                     (128, 128, 2048, 8), (640, 640, 2000, 2), (9, 130, 5000, 1),
                                     (32, 32, 4096, 1)])
def test_products_repeat_bit_for_bit(sc, M, N, K, G):
    """Every tile size with K ranges (2 to 16 of them): the partial sums are added
    in one order, so that a product gives the same bits each time, also where it adds
    to W (the second products of a complex contraction)."""
    rng = np.random.default_rng(M + K)
    p = sc.Plan("ij,jk->ik", (G,), ((1, -1), (0,), (M, K)), ((1, -1), (0,), (K, N)), "fp64")
    draw = lambda s: torch.from_numpy(rng.standard_normal(s)).cuda()
    u, v = draw(p.shape_u), draw(p.shape_v)
    uc, vc = torch.complex(u, draw(p.shape_u)), torch.complex(v, draw(p.shape_v))
    first, firstc = p.contract(u, v), p.contract_complex(uc, vc)
    for _ in range(20):
        assert torch.equal(p.contract(u, v), first)
        assert torch.equal(p.contract_complex(uc, vc), firstc)
    bound = 2 * (K + 2) * 2.0 ** -53 * (u.abs() @ v.abs()).reshape(first.shape)
    assert bool(((first - (u @ v).reshape(first.shape)).abs() <= bound).all())
    want = uc @ vc
    bound = 4 * (K + 2) * 2.0 ** -53 * (uc.abs() @ vc.abs()).reshape(firstc.shape)
    assert bool(((firstc - want.reshape(firstc.shape)).abs() <= bound).all())
