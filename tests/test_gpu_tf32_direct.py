"""The TF32 form that reads its long operand's float64 entries itself: both
roles, one and two MMAs per tile, ragged row tiles, K not a multiple of a stage
or an offset chunk, zeros, entries beyond FP32's normal range, and the shapes
next to its rule, which take the two-step path.  Products of TF32-rounded operands (relative 2^-11 each) summed in
FP32: within K-independent 2^-10 of |u| |v|, plus 2^-20 K^(1/2) of it for the
sums."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sc():
    if not torch.cuda.is_available():
        pytest.fail("a GPU test ran without a visible GPU")
    import paper_2007_08056_gb300 as mod
    mod.load()
    return mod


# (G, long rows, short rows, K): direct where 128-row tiles by G are at least 128,
# the short side is at most 512 and a quarter of the long one
CASES = [(1, 16500, 512, 100), (1, 16400, 300, 514), (2, 8200, 257, 64), (4, 4100, 256, 1040), (1, 17000, 8, 70),
         (1, 16384, 31, 258), (1, 16000, 40, 80), (1, 16500, 520, 96), (128, 100, 24, 66)]


@pytest.mark.parametrize("long_is_u", [True, False], ids=["U", "V"])
@pytest.mark.parametrize("G,R,S,K", CASES)
def test_long_operand(sc, G, R, S, K, long_is_u):
    rng = np.random.default_rng(R + S + K)
    es, du, dv = ("ik,jk->ij", (R, K), (S, K)) if long_is_u else ("ik,jk->ij", (S, K), (R, K))
    p = sc.Plan(es, (G,), ((1, -1), (0,), du), ((1, -1), (0,), dv), "tf32")
    u, v = rng.standard_normal(p.shape_u), rng.standard_normal(p.shape_v)
    a = u if long_is_u else v
    a[..., 5, :] = 0.0
    a[..., 7, ::3] = 0.0
    a[..., 9, :] *= 1e-41        # subnormal in FP32
    a[..., 11, :] *= 2.0 ** 100
    a[..., 12, 1] = 1.0 + 2.0 ** -11 + 2.0 ** -40   # just above a tie
    w = p.contract(torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()).cpu().numpy()
    p.check_device_error()
    for q in range(G):
        want, mag = u[q] @ v[q].T, np.abs(u[q]) @ np.abs(v[q]).T
        # (entries below 2^-126 keep fewer bits, or none)
        low = K * 2.0 ** -126 * max(np.abs(u[q]).max(), np.abs(v[q]).max())
        assert np.all(np.abs(w[q] - want) <= (2.0 ** -10 + 2.0 ** -20 * np.sqrt(K)) * mag + low)
