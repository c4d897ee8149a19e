"""mw_convolve_batched where the coefficients' shared exponents change along the
series (segments cut again), at the edges of the rows of 32 coefficients, with
few and with many series, and past the length whose digits fit in shared memory.
Every checked coefficient equals the oracle's error-free summation of its inner
product (a_0..a_i against b_i..b_0) with the same plan bit for bit: the oracle's
words are a function of the plan and the operands alone, so there is no
tolerance."""
import numpy as np
import pytest

from conftest import to_dev
from oracle.slicing import SlicedProduct
from synthetic import SplitMix64, loguniform_mdouble, uniform_mdouble

pytestmark = pytest.mark.gpu


def coefficient(a, b, i, plan):
    """Coefficient i of a b (m, n): the inner product of a_0..a_i with b_i..b_0."""
    row = np.ascontiguousarray(a[:, None, :i + 1])
    col = np.ascontiguousarray(b[:, i::-1][:, :, None])
    return SlicedProduct(row, col, plan.w, plan.S_A, plan.S_B, plan.D).result()[:, 0, 0]


def check(mw, cuda, A, B, series=None, where=None):
    tA, tB = to_dev(A, cuda), to_dev(B, cuda)
    plan = mw.plan_convolve(tA, tB)
    C = mw.mw_convolve_batched(tA, tB, plan).cpu().numpy()
    for s in range(A.shape[1]) if series is None else series:
        for i in range(A.shape[2]) if where is None else where:
            assert np.array_equal(C[:, s, i], coefficient(A[:, s], B[:, s], i, plan)), (s, i)


@pytest.mark.parametrize("m,count,n", [
    (2, 3, 31), (4, 2, 32), (8, 2, 33), (16, 1, 34), (2, 2, 64), (4, 1, 65), (8, 1, 97),
    (4, 1300, 2), (2, 700, 96),
])
def test_rows_and_series_counts(mw, cuda, m, count, n):
    rng = SplitMix64(1600 + m + n)
    A, B = loguniform_mdouble(rng, m, count, n, -6, 6), uniform_mdouble(rng, m, count, n)
    check(mw, cuda, A, B, series=sorted({0, count // 2, count - 1}))


@pytest.mark.parametrize("m", [2, 4, 8, 16])
def test_exponent_grows_along_the_series(mw, cuda, m):
    """A new largest entry at most coefficients of one operand or both, leading zeros,
    an all-zero operand and words that are not normalised."""
    rng = SplitMix64(1640 + m)
    n = 70
    A, B = uniform_mdouble(rng, m, 6, n), uniform_mdouble(rng, m, 6, n)
    grow = 2.0 ** (np.arange(n) // (4 if m < 16 else 12))   # m = 16 plans spreads up to 23 bits
    A[:, 0] *= grow
    A[:, 1] *= grow
    B[:, 1] *= 2.0 ** (np.arange(n) // 9)
    A[:, 2] *= grow[::-1]                              # falls: one segment
    A[:, 3, :40] = 0.0
    B[:, 3, :5] = 0.0
    A[:, 4] = 0.0
    A[0, 5, 33] = 0.0
    A[1, 5, 33] = 4.0                                  # leading word zero, the second 4
    B[m - 1, 5, 64] = 8.0                              # the last word far above the first
    check(mw, cuda, A, B)


def test_longer_than_shared_memory(mw, cuda):
    rng = SplitMix64(1660)
    m, n = 8, 1700
    A, B = uniform_mdouble(rng, m, 1, n), uniform_mdouble(rng, m, 1, n)
    check(mw, cuda, A, B, where=[0, 31, 255, 256, 1024, n - 1])


def test_status_of_the_whole_series(mw, cuda):
    """A spread wider than the plan's, only at the last coefficient, raises MW_WRANGE."""
    rng = SplitMix64(1670)
    A, B = uniform_mdouble(rng, 2, 2, 80), uniform_mdouble(rng, 2, 2, 80)
    tA, tB = to_dev(A, cuda), to_dev(B, cuda)
    plan = mw.plan_convolve(tA, tB)
    mw.mw_convolve_batched(tA, tB, plan)
    tA[:, 1, 79] *= 2.0 ** -60
    with pytest.raises(mw.MWRangeError):
        mw.mw_convolve_batched(tA, tB, plan)
