"""Inner products for every compiled number of 24-bit digits, on entries whose
words lie at any distance: later words within a few binary orders of the first
(the range check on the digits), zero and subnormal words, zero entries, with and
without the diagonals past S.  Every product is the oracle's error-free summation
with the same digits bit for bit (a function of the plan and the operands alone)."""
import numpy as np
import pytest

from conftest import to_dev
from oracle import slicing
from synthetic import SplitMix64, loguniform_mdouble

pytestmark = pytest.mark.gpu


def entries(m, rows, cols, seed):
    rng = np.random.RandomState(seed)
    X = loguniform_mdouble(SplitMix64(seed), m, rows, cols, -9, 9)
    for j in range(1, m):
        X[j] = X[j - 1] * 2.0 ** -rng.randint(1, 64, (rows, cols)) * rng.choice([1, -1], (rows, cols))
    X[1:][rng.rand(m - 1, rows, cols) < 0.2] = 0.0
    X[:, rng.rand(rows, cols) < 0.05] = 0.0
    X[:, 1, :] = 0.0                              # a zero vector
    X[m - 1, 2, :5] = 5e-324                      # subnormal words
    X[1, 0, :9] = X[0, 0, :9] * np.array([1, -1, .5, -.5, .75, .25, -.25, .3, 0.])
    return X


@pytest.mark.parametrize("m,S", [(2, 4), (2, 5), (2, 6), (2, 7), (2, 8), (4, 8), (4, 9), (4, 10),
                                 (4, 11), (4, 12), (8, 17), (8, 19), (8, 21), (16, 35), (16, 36)])
@pytest.mark.parametrize("extra", [0, 3])
def test_every_digit_count(mw, cuda, m, S, extra):
    count, K = 3, 301
    A, B = entries(m, count, K, 50 * m + S), entries(m, count, K, 50 * m + S + 1000)
    plan = mw.mw_plan_gemm(m, "dot", 1, 1, K, 0, 0)
    plan.S_A = plan.S_B = S
    plan.D = S + extra
    plan.range_A = plan.range_B = 3000
    C = mw.mw_dot_batched(to_dev(A, cuda), to_dev(B, cuda), plan).cpu().numpy()
    for i in range(count):
        a = np.ascontiguousarray(A[:, i:i + 1])
        b = np.ascontiguousarray(B[:, i][:, :, None])
        want = slicing.SlicedProduct(a, b, 24, S, S, plan.D).result()[:, 0, 0]
        assert np.array_equal(C[:, i], want), i
