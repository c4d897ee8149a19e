"""The exact fusion for every number of diagonals: each output of a single product
is the greedy rounding of the integer its stored diagonal sums make (Python
integers), and the same problem in a batch gives the same words.  Every limb
count the kernels are compiled for, whole and ragged last limbs, ragged sizes."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from conftest import to_dev
from oracle.exact import greedy_words
from synthetic import SplitMix64, uniform_mdouble

pytestmark = pytest.mark.gpu


def check(mw, cuda, m, M, N, K, plan):
    rng = SplitMix64(1900 + m)
    A, B = to_dev(uniform_mdouble(rng, m, M, K), cuda), to_dev(uniform_mdouble(rng, m, K, N), cuda)
    off, total = mw.workspace_layout(plan, M, N, K)
    ws = torch.zeros(total, dtype=torch.uint8, device=cuda)
    C = mw.mw_gemm(A, B, plan, ws=ws, check=False)
    D = plan.D
    s = ws[off[3]:off[3] + 4 * D * M * N].view(torch.int32).cpu().numpy().reshape(D, N, M)
    E = ws[:8 * (M + N)].view(torch.int32).cpu().numpy()
    got = C.cpu().numpy()
    for i in sorted({0, min(1, M - 1), M // 2, M - 1}):
        for j in sorted({0, min(1, N - 1), N // 2, N - 1}):
            X = sum(int(s[t, j, i]) << (plan.w * (D - 1 - t)) for t in range(D))
            ex = int(E[i]) + int(E[2 * M + j]) + 4 - plan.w * (D + 1)
            assert list(got[:, i, j]) == list(greedy_words(Fraction(X) * Fraction(2) ** ex, m)), (D, i, j)
    assert torch.equal(mw.Batch([A], [B], plan=plan).run()[0], C), D
    mw.get_status()


@pytest.mark.parametrize("m,lo,hi", [(2, 13, 34), (4, 26, 50), (8, 52, 73), (16, 104, 128)])
def test_every_diagonal_count(mw, cuda, m, lo, hi):
    for D in range(lo, hi):
        plan = mw.mw_plan_gemm(m, "ozaki", 33, 9, 20, 20, 20)
        plan.S_A = plan.S_B = min(max(D - 3, 1), {2: 78, 4: 78, 8: 78, 16: 126}[m])
        plan.D = D
        plan.range_A = plan.range_B = 4000
        check(mw, cuda, m, 33, 9, 20, plan)


@pytest.mark.parametrize("M,N", [(1, 1), (32, 8), (31, 7), (64, 17), (3, 130), (257, 4)])
def test_ragged_sizes(mw, cuda, M, N):
    check(mw, cuda, 4, M, N, 12, mw.mw_plan_gemm(4, "ozaki", M, N, 12, 20, 20))


def test_other_widths(mw, cuda):
    for w in (6, 7):
        check(mw, cuda, 8, 34, 10, 20, mw.mw_plan_gemm(8, "ozaki", 34, 10, 20, 20, 20, w=w))
