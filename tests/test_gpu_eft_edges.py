"""mw_elementwise where the ordering of two_sum's operands and the dropped zero
products of a division could show: equal exponents, cancellation, zeros of both
signs, subnormals, infinities, NaN and sums that overflow.  Additions are
compared bit for bit (NaN with NaN) with the same sweeps of Knuth's two_sum in
numpy: the C oracle drops terms that are exactly zero on the way, which leaves
finite words alone but not which words of a sum that is not finite are NaN.
Products and quotients with zero words are the C oracle's."""
import numpy as np
import pytest

from conftest import to_dev
from oracle import textbook

pytestmark = pytest.mark.gpu

TINY = 5e-324
FINITE = [0.0, -0.0, 1.0, -1.0, 1.0 + 2.0 ** -52, -1.0 + 2.0 ** -53, 2.0 ** 53, -2.0 ** 53 - 2.0,
          2.0 ** -53, 3.0 * 2.0 ** -54, -2.0 ** -54, 1.5, -1.9999999999999998, TINY, -TINY,
          2.0 ** -1022, -2.0 ** -1022 + TINY, 2.0 ** -970]
LARGE = [1.7976931348623157e308, -1.7976931348623157e308, 2.0 ** 1023, np.inf, -np.inf, np.nan]


def same(got, want):
    ok = (got.view(np.uint64) == want.view(np.uint64)) | (np.isnan(got) & np.isnan(want))
    assert ok.all(), np.argwhere(~ok)[:5]


def pool(values, m, n, seed):
    """(m, n) words drawn from `values`: not normalised, every order of magnitude."""
    rng = np.random.RandomState(seed)
    return np.array(values)[rng.randint(0, len(values), (m, n))]


def two_sum(a, b):
    s = a + b
    bv = s - a
    return s, (a - (s - bv)) + (b - bv)


def fast_two_sum(a, b):
    s = a + b
    return s, b - (s - a)


def knuth_add(A, B):
    """The m-double addition, every zero term kept."""
    m = len(A)
    if m == 2:
        s, e = two_sum(A[0], B[0])
        t, f = two_sum(A[1], B[1])
        s, e = fast_two_sum(s, e + t)
        return np.stack(fast_two_sum(s, e + f))
    x = [w for pair in zip(A, B) for w in pair]
    out = []
    for _ in range(m):
        s, errors = x[-1], []
        for v in reversed(x[:-1]):
            s, e = two_sum(v, s)
            errors.insert(0, e)
        out.append(s)
        x = errors
    return np.stack(out)


@pytest.mark.parametrize("m", [2, 4, 8])
@pytest.mark.parametrize("values", [FINITE, FINITE + LARGE], ids=["finite", "special"])
def test_add(mw, cuda, m, values):
    n = 20011
    A, B = pool(values, m, n, 10 + m), pool(values, m, n, 20 + m)
    with np.errstate(all="ignore"):
        want = knuth_add(A, B)
    same(mw.mw_elementwise("add", to_dev(A, cuda), to_dev(B, cuda)).cpu().numpy(), want)


@pytest.mark.parametrize("m", [2, 4, 8])
@pytest.mark.parametrize("op", ["mul", "div"])
def test_zero_words(mw, cuda, m, op):
    """Words that are zero (short m-doubles, integers, zero numerators)."""
    n = 5003
    rng = np.random.RandomState(40 + m)
    A, B = (rng.randint(-50, 51, (m, n)) * 2.0 ** (-60.0 * np.arange(m))[:, None] for _ in range(2))
    for X in (A, B):
        X[1:, : n // 2][rng.rand(m - 1, n // 2) < 0.7] = 0.0
    A[:, ::7] = 0.0
    B[0][B[0] == 0.0] = 3.0
    want = textbook.TextbookC().elementwise(op, A, B)
    got = mw.mw_elementwise(op, to_dev(A, cuda), to_dev(B, cuda)).cpu().numpy()
    assert np.array_equal(got, want)
