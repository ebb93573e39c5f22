"""The default split form (four FP16 digits of 10 bits) at the sizes and values
where its GEMM can go wrong: half tiles and remainders of M and N, one column of
K up to several folds of the diagonals, split K ranges, and entries whose digits
are at their limits so that every partial sum is.

An entry is rounded to 39 bits below its row's 2^(E+1) and the digit pairs with
i + j >= 4 are dropped (three of 2^-40 each), so an output is within
K 2^(Eu+1) 2^(Ev+1) (2 x 2^-40 + 3 x 2^-40) of the exact sum, plus the rounding
of the diagonals d >= 2 (2^-20 of the products, FP32 sums of at most 544 columns
between folds, rounded by 2^5 of 16 x 2^38 a step: below 2^-37 K of the same
scale) and of R (2^-39); 2^-36 K covers them all.  A row whose largest entry is
within about 2^-10 below 2^(E+1) is scaled by 2^(E+2) instead, so that no leading
digit is 512 and the sums of diagonals 0 and 1 stay below 2^24."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [(8, 8, 1), (127, 63, 31), (128, 64, 33), (129, 65, 64), (257, 127, 96), (40, 129, 577),
         (8, 200, 1100), (9, 8, 8200), (130, 140, 32768)]


@pytest.fixture(scope="module")
def sc():
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a visible GPU")
    import paper_2007_08056_gb300 as mod
    mod.load()
    return mod


def draw(kind, shape, rng):
    if kind == "normal":
        return rng.standard_normal(shape) * 2.0 ** rng.integers(-30, 30, shape[:-1] + (1,))
    if kind == "largest":      # rounds up to the next power of two at 39 bits: E raised
        return np.full(shape, 2.0 - 2.0 ** -45)
    if kind == "top":          # the largest that is not raised: leading digits of 511, then 511, 509
        return np.full(shape, 2.0 - 2.0 ** -9 - 3 * 2.0 ** -20) * (1 - 2.0 ** -36 * rng.integers(0, 2, shape))
    if kind == "aligned":      # every digit 410 in size: all partial sums grow with K
        return np.full(shape, 0.1) * np.where(rng.random(shape[:-1] + (1,)) < 0.5, 1.0, -1.0)
    # lower digits of -512: X = 300 2^30 - 512 (2^20 + 2^10 + 1)
    return np.full(shape, (300 * 2.0 ** 30 - 512 * (2.0 ** 20 + 2.0 ** 10 + 1)) / 2.0 ** 38)


@pytest.mark.parametrize("kind", ["normal", "largest", "top", "aligned", "lowest"])
@pytest.mark.parametrize("M,N,K", SIZES)
def test_digits_and_tiles(sc, M, N, K, kind):
    rng = np.random.default_rng(M + 7 * N + 13 * K)
    p = sc.Plan("ij,jk->ik", (1,), ((1, -1), (0,), (M, K)), ((1, -1), (0,), (K, N)), "split_bf16")
    assert p.info.tensor_core == 1
    u, v = draw(kind, (M, K), rng), np.ascontiguousarray(draw(kind, (N, K), rng).T)
    w = p.contract(torch.from_numpy(u).cuda().reshape(p.shape_u), torch.from_numpy(v).cuda().reshape(p.shape_v))
    torch.cuda.synchronize()
    p.check_device_error()
    got = w.cpu().numpy().reshape(M, N)
    # 2^(E+1), of the raised rows too
    scale = lambda x, axis: 2.0 ** np.ceil(np.log2(np.abs(x).max(axis) * (1 + 2.0 ** -9)))
    bound = K * 2.0 ** -36 * np.outer(scale(u, 1), scale(v, 0))
    assert np.all(np.abs(got - u @ v) <= bound + 1e-15 * (np.abs(u) @ np.abs(v)))


@pytest.mark.parametrize("G,M,N,K", [(1, 130, 70, 128), (1, 130, 70, 2048), (1, 70, 130, 40000),
                                     (3, 1300, 1172, 96), (3, 1300, 1172, 128), (3, 1300, 1172, 2048),
                                     (5, 2000, 190, 192), (5, 2000, 190, 2048)])
@pytest.mark.parametrize("top", [1023.0, 1021.0])
def test_one_sign_just_below_a_power_of_two(sc, G, M, N, K, top):
    """Integers 1021 and 1023: leading digits of 511 and 512 below their row's own
    power of two, the second ones -512.  64 products of 512^2 are 2^24, which leaves
    FP32 no room for the rest of a drain, so rows with 1023 are raised; 1019 and 1021
    are not: 64 x 511^2 and 64 x 511 x 512 are the most that diagonals 0 and 1 hold.
    The sums must be exact (K ranges, wide and narrow tiles)."""
    rng = np.random.default_rng(K)
    u = np.full((G, M, K), top)
    v = np.full((G, K, N), top)
    u[:, :, 0], v[:, 0, :] = top - 2.0, top - 2.0
    u[:, ::3, :] -= 2.0 * rng.integers(0, 2, (G, (M + 2) // 3, K))
    p = sc.Plan("ij,jk->ik", (G,), ((1, -1), (0,), (M, K)), ((1, -1), (0,), (K, N)), "split_bf16")
    w = p.contract(torch.from_numpy(u).cuda().reshape(p.shape_u), torch.from_numpy(v).cuda().reshape(p.shape_v))
    p.check_device_error()
    assert np.array_equal(w.cpu().numpy().reshape(G, M, N), u @ v)      # |sums| < 2^53


@pytest.mark.parametrize("M,N,K", [(96, 80, 1024), (300, 260, 1024), (64, 72, 9000)])
def test_entries_near_one_from_below(sc, M, N, K):
    """cos of small angles: nine leading digits in ten would be 512 at the row's own
    power of two.  Within the split form's 1e-10 in the 2-norm, 1e-9 at most."""
    rng = np.random.default_rng(M)
    u, v = np.cos(0.02 * rng.standard_normal((M, K))), np.cos(0.02 * rng.standard_normal((K, N)))
    p = sc.Plan("ij,jk->ik", (1,), ((1, -1), (0,), (M, K)), ((1, -1), (0,), (K, N)), "split_bf16")
    w = p.contract(torch.from_numpy(u).cuda().reshape(p.shape_u), torch.from_numpy(v).cuda().reshape(p.shape_v))
    e = w.cpu().numpy().reshape(M, N) - u @ v
    assert np.linalg.norm(e) <= 1e-10 * np.linalg.norm(u @ v)
    assert np.all(np.abs(e) <= 1e-9 * (u @ v))


def test_exact_products_of_either_sign(sc):
    """Entries +-1 (leading digit 256) and small multiples of 2^-9: two digits each, so
    every product is in diagonals 0 to 2, whose sums here are integers that FP32 holds,
    and the result is the exact sum."""
    rng = np.random.default_rng(3)
    M, N, K = 130, 70, 20000
    u, v = (rng.choice([1.0, -1.0, 2.0 ** -9, 3.0 * 2.0 ** -9], (r, K)) for r in (M, N))
    u[:, 0] = v[:, 0] = 1.0
    p = sc.Plan("ij,jk->ik", (1,), ((1, -1), (0,), (M, K)), ((1, -1), (0,), (K, N)), "split_bf16")
    w = p.contract(torch.from_numpy(u).cuda().reshape(p.shape_u),
                   torch.from_numpy(np.ascontiguousarray(v.T)).cuda().reshape(p.shape_v))
    ui, vi = (np.rint(x * 2.0 ** 9).astype(np.int64) for x in (u, v))
    exact = (ui @ vi.T).astype(np.float64) * 2.0 ** -18    # |sum| < 2^53
    assert np.array_equal(w.cpu().numpy().reshape(M, N), exact)


@pytest.mark.parametrize("M,N,K", [(2000, 190, 100), (1990, 129, 700), (2040, 192, 33)])
def test_narrow_tiles(sc, M, N, K):
    """Five irreps whose 128-column tiles need two rounds of the SMs and whose
    64-column tiles need one: the narrow kernel."""
    G = 5
    p = sc.Plan("ij,jk->ik", (G,), ((1, -1), (0,), (M, K)), ((1, -1), (0,), (K, N)), "split_bf16")
    rng = np.random.default_rng(M)
    u, v = rng.standard_normal(p.shape_u), rng.standard_normal(p.shape_v)
    w = p.contract(torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()).cpu().numpy()
    p.check_device_error()
    for q in range(G):
        bound = K * 2.0 ** -36 * 64.0    # |entries| < 8 = 2^(E+1)
        assert np.all(np.abs(w[q] - u[q] @ v[q]) <= bound)


@pytest.mark.parametrize("K", [20, 64, 90, 545, 1056])
@pytest.mark.parametrize("M,N", [(1300, 1172), (19300, 40)])
def test_several_tiles_per_cta(sc, M, N, K):
    """Three irreps in more tiles than stay resident, so that a CTA walks several:
    full ones and ones with half their columns or a few rows, of 1, 2, 3, 18 and 33
    stages (K ranges of odd and even length start the next tile's waits); the second
    shape takes the narrow kernel.  The same bound as above."""
    G = 3
    p = sc.Plan("ij,jk->ik", (G,), ((1, -1), (0,), (M, K)), ((1, -1), (0,), (K, N)), "split_bf16")
    rng = np.random.default_rng(K)
    u, v = rng.standard_normal(p.shape_u), rng.standard_normal(p.shape_v)
    ud, vd = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    w = p.contract(ud, vd)
    again = p.contract(ud, vd)
    p.check_device_error()
    assert torch.equal(w, again)
    w = w.cpu().numpy()
    for q in range(G):
        assert np.all(np.abs(w[q] - u[q] @ v[q]) <= K * 2.0 ** -36 * 64.0)


@pytest.mark.parametrize("N", [70, 40])
def test_row_and_column_scales_to_the_ends_of_the_range(sc, N):
    """Small integers times powers of two, with zero rows and columns: the sums are
    exact, so every result is the sum rounded once, normal, subnormal or 0."""
    M, K = 130, 64
    rng = np.random.default_rng(N)
    u, v = (rng.integers(-31, 32, (r, K)).astype(np.float64) for r in (M, N))
    a = np.resize([-600, -511, -480, 0, 490, 505, -540], M)
    b = np.resize([0, -560, -511, -470, 480, 495], N)
    u[5], u[64], v[3], v[N - 1] = 0, 0, 0, 0
    p = sc.Plan("ij,jk->ik", (1,), ((1, -1), (0,), (M, K)), ((1, -1), (0,), (K, N)), "split_bf16")
    us, vs = np.ldexp(u, a[:, None]), np.ldexp(v, b[:, None])
    w = p.contract(torch.from_numpy(us).cuda().reshape(p.shape_u),
                   torch.from_numpy(np.ascontiguousarray(vs.T)).cuda().reshape(p.shape_v))
    p.check_device_error()
    assert np.array_equal(w.cpu().numpy().reshape(M, N), np.ldexp(u @ v.T, a[:, None] + b[None, :]))
