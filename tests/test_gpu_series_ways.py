"""mw_convolve_batched where coefficients are taken one by one beside whole rows of them:
few series of any length (several CTAs a series), series whose exponents grow all along
(nearly every coefficient cut on a grid of its own), and lengths between 300 and 1,200
with several pairs of rows and several parts.  Every checked coefficient equals the inner
product of a_0..a_i with b_i..b_0 by mw_dot_batched with the same plan bit for bit (the
words are a function of the plan and the operands), a few of them the oracle's."""
import numpy as np
import pytest
import torch

from oracle.slicing import SlicedProduct

pytestmark = pytest.mark.gpu


def series(m, count, n, growth, seed, cuda):
    """Random series; `growth`: binades that the entries of (a, b) grow over their length."""
    gen = torch.Generator(device=cuda).manual_seed(seed)
    out = []
    for g in growth:
        X = torch.empty((m, count, n), dtype=torch.float64, device=cuda)
        for j in range(m):
            u = torch.rand((count, n), dtype=torch.float64, device=cuda, generator=gen) * 2 - 1
            X[j] = u if j == 0 else X[j - 1] * u * 2.0 ** -53
        out.append(X * torch.exp2(torch.floor(torch.arange(n, device=cuda).double() * g / n)))
    return out


def inner(mw, A, B, i, plan):
    """Coefficient i of every series, (m, count)."""
    return mw.mw_dot_batched(A[:, :, :i + 1].contiguous(), B[:, :, :i + 1].flip(2).contiguous(), plan)


def check(mw, A, B, where, oracle=()):
    plan = mw.plan_convolve(A, B)
    C = mw.mw_convolve_batched(A, B, plan)
    for i in where:
        assert torch.equal(C[:, :, i], inner(mw, A, B, i, plan)), i
    for s, i in oracle:
        row = np.ascontiguousarray(A[:, s, None, :i + 1].cpu().numpy())
        col = np.ascontiguousarray(B[:, s, :i + 1].flip(1)[:, :, None].cpu().numpy())
        ref = SlicedProduct(row, col, plan.w, plan.S_A, plan.S_B, plan.D).result()[:, 0, 0]
        assert np.array_equal(C[:, s, i].cpu().numpy(), ref), (s, i)


@pytest.mark.parametrize("m", [2, 4, 8, 16])
@pytest.mark.parametrize("count,n", [(1, 1), (1, 31), (1, 33), (2, 64), (3, 65), (1, 130), (20, 97),
                                     (40, 16), (160, 40), (1300, 33), (400, 100)])
@pytest.mark.parametrize("growth", [(0, 0), (45, 0), (40, 45)])
def test_few_and_many_series(mw, cuda, m, count, n, growth):
    if m == 16:
        growth = tuple(min(g, 4) for g in growth)    # m = 16 plans spreads up to 23 bits
    A, B = series(m, count, n, growth, 100 * m + n, cuda)
    check(mw, A, B, range(n), oracle=[(count - 1, n - 1), (0, n // 2)])


@pytest.mark.parametrize("m,count,n,growth", [
    (2, 300, 600, (0, 0)), (2, 300, 600, (45, 40)), (4, 160, 1000, (0, 0)), (4, 20, 700, (45, 0)),
    (8, 200, 520, (0, 0)), (8, 160, 513, (45, 45)), (8, 1, 1200, (0, 0)), (8, 2, 1100, (45, 45)),
    (16, 2, 700, (4, 0)), (16, 100, 300, (0, 0)), (2, 1, 2500, (20, 20)), (4, 5, 1300, (0, 45)),
])
def test_long_series(mw, cuda, m, count, n, growth):
    A, B = series(m, count, n, growth, n + m, cuda)
    step = max(1, n // 40)
    check(mw, A, B, sorted({*range(0, n, step), *range(0, n, 32), n - 1}), oracle=[(0, 40), (0, n - 1)])


def microseconds(f, n=10):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    f()
    out = []
    for _ in range(7):
        torch.cuda.synchronize()
        a.record()
        for _ in range(n):
            f()
        b.record()
        b.synchronize()
        out.append(a.elapsed_time(b) / n * 1e3)
    return sorted(out)[3]


@pytest.mark.parametrize("m,count,n", [(8, 1, 128), (4, 1, 64), (2, 40, 128), (8, 100, 512)])
def test_growing_series_against_inner_products(mw, cuda, m, count, n):
    """No slower than three times as many inner products of full length cost (the work of
    twice the series' products): one warp walking a row once for every coefficient took
    up to 27 times that of the triangle."""
    A, B = series(m, count, n, (45, 45), 7, cuda)
    plan = mw.plan_convolve(A, B)
    C = torch.empty_like(A)
    D = torch.empty((m, count * n), dtype=torch.float64, device=cuda)
    X = A.repeat(1, 1, n).reshape(m, count * n, n)
    Y = B.repeat(1, 1, n).reshape(m, count * n, n)
    t = microseconds(lambda: mw.mw_convolve_batched(A, B, plan, C=C, check=False))
    assert t <= 3 * microseconds(lambda: mw.mw_dot_batched(X, Y, plan, C=D, check=False))
