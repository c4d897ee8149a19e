"""MW_PLAIN at the edges of its 4 x 8 tiles and of its k chunks (8 to 64 columns,
by the number of pieces), and a plan with too many pieces for them (the general
kernel).  The diagonal sums are exact in any order and the accumulation of s_t
takes t in order, so every product is bit for bit that of its own 16 x 16 blocks
computed alone; each is also within the bound."""
import numpy as np
import pytest

from conftest import to_dev
from oracle import exact
from synthetic import SplitMix64, loguniform_mdouble

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,M,N,K,w", [
    (2, 1, 1, 1, 0), (2, 4, 8, 63, 0), (2, 5, 9, 65, 0), (4, 3, 7, 9, 0), (4, 33, 41, 130, 0),
    (8, 9, 17, 33, 0), (8, 6, 10, 71, 0), (2, 70, 20, 300, 12),
    (4, 18, 20, 40, 4),                  # 55 or more pieces: the general kernel
])
def test_tiles_and_chunks(mw, cuda, m, M, N, K, w):
    rng = SplitMix64(1700 + m + M + K)
    A, B = loguniform_mdouble(rng, m, M, K, -4, 4), loguniform_mdouble(rng, m, K, N, -4, 4)
    tA, tB = to_dev(A, cuda), to_dev(B, cuda)
    plan = mw.plan_for(tA, tB, "plain", w=w)
    C = mw.mw_gemm(tA, tB, plan).cpu().numpy()
    assert exact.exact_product_full(A, B).error_ratio(C).max() <= 1.0
    for i in range(0, M, 16):
        for j in range(0, N, 16):
            sub = mw.mw_gemm(tA[:, i:i + 16], tB[:, :, j:j + 16], plan).cpu().numpy()
            assert np.array_equal(sub, C[:, i:i + 16, j:j + 16]), (i, j)
