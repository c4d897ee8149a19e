"""MW_PLAIN with more pieces than the 4 x 8 tiles' shared memory takes, which the general
kernel multiplies (and, beside it, a plan that does fit), and products large enough for
that kernel to be the faster one.  The diagonal sums are exact
integers (the oracle's); both kernels add them, scaled, into an accumulator of m + 1
words in order of t with two-sums, and renormalise that into m words: the same steps in
numpy give the same words bit for bit."""
import numpy as np
import pytest

from conftest import to_dev
from oracle import exact, slicing
from synthetic import SplitMix64, loguniform_mdouble

pytestmark = pytest.mark.gpu


def two_sum(a, b):
    s = a + b
    bv = s - a
    return s, (a - (s - bv)) + (b - bv)


def words(sp, m):
    """(m, M, N) words from the diagonal sums of the sliced product sp."""
    D, M, N = sp.D, len(sp.A.rows), len(sp.B.rows)
    e = sp.A.E[:, None] + sp.B.E[None, :] + 4
    acc = [np.zeros((M, N)) for _ in range(m + 1)]
    for t in range(D):
        x = np.ldexp(sp.s[t].astype(np.float64), e - sp.w * (t + 2))
        for j in range(m + 1):
            acc[j], x = two_sum(acc[j], x)
        for j in range(m, 0, -1):
            acc[j - 1], acc[j] = two_sum(acc[j - 1], acc[j])
    out = []
    for _ in range(m):
        s = acc[-1]
        errs = [None] * len(acc)
        for i in range(len(acc) - 2, -1, -1):
            s, errs[i + 1] = two_sum(acc[i], s)
        out.append(s)
        acc = errs[1:] + [np.zeros((M, N))]
    return np.stack(out)


@pytest.mark.parametrize("m,M,N,K,w,lo,general", [
    (8, 18, 20, 40, 4, -4, True), (8, 33, 17, 19, 4, -4, True), (8, 1, 1, 1, 5, -4, True),
    (4, 35, 30, 17, 4, -40, True), (2, 70, 65, 33, 4, -80, True), (4, 10, 12, 40, 4, -4, False),
])
def test_words(mw, cuda, m, M, N, K, w, lo, general):
    rng = SplitMix64(1800 + m + M + K)
    A, B = loguniform_mdouble(rng, m, M, K, lo, -lo), loguniform_mdouble(rng, m, K, N, lo, -lo)
    if K > 1:
        A[0, 0, :2] = 2.0 ** lo, 2.0 ** -lo              # the whole spread
        B[0, :2, 0] = 2.0 ** -lo, 2.0 ** lo
    tA, tB = to_dev(A, cuda), to_dev(B, cuda)
    plan = mw.plan_for(tA, tB, "plain", w=w)
    # pieces of 8 columns of k and the sums of 8 warps, in the 227 KB a block can have
    tiles = 8 * ((4 * plan.S_A + 8 * plan.S_B) * 10 + 8 * plan.D * 32)
    assert (tiles > 232448) == general, (plan, tiles)
    C = mw.mw_gemm(tA, tB, plan).cpu().numpy()
    sp = slicing.SlicedProduct(A, B, plan.w, plan.S_A, plan.S_B, plan.D)
    assert np.array_equal(C, words(sp, m))
    assert exact.exact_product_full(A, B).error_ratio(C).max() <= 1.0


@pytest.mark.parametrize("m,M,N,K,w", [(4, 512, 512, 64, 0), (4, 500, 517, 50, 0), (4, 450, 460, 17, 8)])
def test_large_products(mw, cuda, m, M, N, K, w):
    """Equal to the products of their corners, which the small tiles multiply."""
    rng = SplitMix64(1850 + M)
    A, B = loguniform_mdouble(rng, m, M, K, -4, 4), loguniform_mdouble(rng, m, K, N, -4, 4)
    tA, tB = to_dev(A, cuda), to_dev(B, cuda)
    plan = mw.plan_for(tA, tB, "plain", w=w)
    C = mw.mw_gemm(tA, tB, plan).cpu().numpy()
    for i in (slice(0, 33), slice(240, 272), slice(M - 20, M)):
        for j in (slice(0, 40), slice(250, 270), slice(N - 11, N)):
            sub = mw.mw_gemm(tA[:, i].contiguous(), tB[:, :, j].contiguous(), plan).cpu().numpy()
            assert np.array_equal(sub, C[:, i, j]), (i, j)
