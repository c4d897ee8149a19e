"""Both operands' exponents in one launch (reductions up to 2,048, operands up to 1.5 M
words) and apart: exponents and spreads in the workspace, measured spreads and words of
products on either side of the limit, all four transposes, with zero rows,
subnormal and single nonzero words, non-finite input reported."""
import numpy as np
import pytest
import torch

from conftest import to_dev
from oracle import slicing
from synthetic import SplitMix64, loguniform_mdouble

pytestmark = pytest.mark.gpu


def rows_of(X):
    """(E, spread) of every row of X (m, R, K): ilogb + 1 of the largest word of each entry."""
    E, S = [], []
    for r in range(X.shape[1]):
        es = [e for k in range(X.shape[2])
              if (e := slicing.entry_exponent(X[:, r, k])) is not None]
        E.append(max(es) if es else 0)
        S.append(max(es) - min(es) if es else 0)
    return E, S


@pytest.mark.parametrize("transA,transB", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("m,M,N,K", [(2, 9, 17, 33), (4, 8, 1, 31), (8, 1, 8, 70), (16, 3, 5, 40),
                                     (2, 5, 6, 2048), (2, 5, 6, 2049), (4, 60, 130, 2048), (4, 62, 131, 2048)])
def test_exponents_and_words(mw, cuda, m, M, N, K, transA, transB):
    rng = SplitMix64(2000 + m + K)
    LA, LB = loguniform_mdouble(rng, m, M, K, -4, 4), loguniform_mdouble(rng, m, K, N, -4, 4)
    LA[:, M - 1, : K // 2] = 0.0
    LA[1, 0, K - 1], LA[0, 0, K - 1] = 8.0, 0.0          # a word larger than the first
    if M > 2:
        LA[:, 1] = 0.0                                   # a zero row
    LB[:, 3, 0] = 0.0
    A = np.ascontiguousarray(LA.transpose(0, 2, 1)) if transA else LA
    B = np.ascontiguousarray(LB.transpose(0, 2, 1)) if transB else LB
    tA, tB = to_dev(A, cuda), to_dev(B, cuda)
    (eA, sA), (eB, sB) = rows_of(LA), rows_of(np.ascontiguousarray(LB.transpose(0, 2, 1)))
    assert mw.mw_measure_spread(tA, tB, transA, transB) == (max(sA), max(sB))
    plan = mw.plan_for(tA, tB, "ozaki", transA, transB)
    off, total = mw.workspace_layout(plan, M, N, K)
    ws = torch.zeros(total, dtype=torch.uint8, device=cuda)
    C = mw.mw_gemm(tA, tB, plan, transA=transA, transB=transB, ws=ws).cpu().numpy()
    got = ws[:4 * (2 * M + 2 * N + 2)].view(torch.int32).cpu().tolist()
    assert got == eA + sA + eB + sB + [max(sA), max(sB)]
    assert np.array_equal(C, slicing.SlicedProduct(LA, LB, plan.w, plan.S_A, plan.S_B, plan.D).result())


def test_reports(mw, cuda):
    rng = SplitMix64(2100)
    A, B = loguniform_mdouble(rng, 2, 6, 40, -4, 4), loguniform_mdouble(rng, 2, 40, 7, -4, 4)
    plan = mw.plan_for(to_dev(A, cuda), to_dev(B, cuda), "ozaki")
    B[0, 11, 3] *= 2.0 ** -90
    with pytest.raises(mw.MWRangeError):
        mw.mw_gemm(to_dev(A, cuda), to_dev(B, cuda), plan)
    A[1, 2, 5] = np.inf
    with pytest.raises(mw.MWError, match="ENONFINITE"):
        mw.mw_gemm(to_dev(A, cuda), to_dev(B, cuda), plan)
