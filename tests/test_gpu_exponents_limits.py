"""Exponents and spreads at the reductions where they stop being taken for both operands
in one launch (by number of words, in a product and in the spread measurement), and for
very many short rows.  They are integers: equal to those of the words' exponents by
torch.frexp."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def exponents(X):
    """(E, spread) of the rows of X (m, R, K), every word nonzero."""
    e = torch.frexp(X)[1].amax(0)
    return e.amax(1), e.amax(1) - e.amin(1)


def entries(gen, shape, cuda):
    X = torch.rand(shape, dtype=torch.float64, device=cuda, generator=gen) + 2.0 ** -9
    X[0] *= torch.exp2(torch.randint(-3, 4, shape[1:], device=cuda, generator=gen).double())
    return X


@pytest.mark.parametrize("transA,transB", [(False, False), (True, True)])
@pytest.mark.parametrize("m,K", [(2, 1536), (2, 1537), (4, 1024), (4, 1025), (8, 512), (8, 513),
                                 (16, 512), (16, 513)])
def test_products(mw, cuda, m, K, transA, transB):
    gen = torch.Generator(device=cuda).manual_seed(K)
    M, N = 9, 20
    LA, LB = entries(gen, (m, M, K), cuda), entries(gen, (m, N, K), cuda)
    A = LA.transpose(1, 2).contiguous() if transA else LA
    B = LB if transB else LB.transpose(1, 2).contiguous()
    plan = mw.plan_for(A, B, "ozaki", transA, transB)
    ws = torch.zeros(mw.workspace_size(plan, M, N, K), dtype=torch.uint8, device=cuda)
    mw.mw_gemm(A, B, plan, transA=transA, transB=transB, ws=ws, check=False)
    mw.get_status()     # sixteen words of one magnitude add up past the digits' range (reported)
    (eA, sA), (eB, sB) = exponents(LA), exponents(LB)
    got = ws[:4 * (2 * M + 2 * N + 2)].view(torch.int32).long().cpu()
    assert torch.equal(got[:M], eA.long().cpu()) and torch.equal(got[M:2 * M], sA.long().cpu())
    assert torch.equal(got[2 * M:2 * M + N], eB.long().cpu())
    assert got[-2:].tolist() == [int(sA.max()), int(sB.max())]


@pytest.mark.parametrize("m,R,K,trans", [
    (2, 10, 2048, False), (2, 10, 2049, True), (4, 10, 1024, True), (4, 10, 1025, False),
    (8, 10, 1024, False), (8, 10, 1025, True), (16, 10, 1024, True), (16, 10, 1025, False),
    (2, 131072, 5, True), (2, 131073, 5, True), (2, 131073, 64, True), (2, 131073, 2, False),
    (2, 131073, 129, False),
])
def test_spread(mw, cuda, m, R, K, trans):
    gen = torch.Generator(device=cuda).manual_seed(R + K)
    LA, LB = entries(gen, (m, R, K), cuda), entries(gen, (m, 3, K), cuda)
    A = LA.transpose(1, 2).contiguous() if trans else LA
    assert mw.mw_measure_spread(A, LB, trans, True) == (int(exponents(LA)[1].max()),
                                                        int(exponents(LB)[1].max()))
