"""The residue split at the edges of its fixed-point lengths (4 to 12 limbs of 32
bits, 16 to 64 columns of digits) on entries of every shape: words at any distance, zero and
subnormal words, later words within two binary orders of the first, zero rows.
Exponents, residue planes, sums and words equal the residue oracle's bit for bit
(the planes are a function of the plan and the operands alone: no tolerance)."""
import numpy as np
import pytest
import torch

from oracle import crt
from test_gpu_crt import bf16_to_int, run_crt
from synthetic import SplitMix64, loguniform_mdouble

pytestmark = pytest.mark.gpu


def entries(m, rows, cols, seed):
    """m-doubles whose words lie anywhere below the first one."""
    rng = np.random.RandomState(seed)
    X = loguniform_mdouble(SplitMix64(seed), m, rows, cols, -10, 10)
    for j in range(1, m):
        X[j] = X[j - 1] * 2.0 ** -rng.randint(1, 70, (rows, cols)) * rng.choice([1, -1], (rows, cols))
    X[1:][rng.rand(m - 1, rows, cols) < 0.2] = 0.0
    X[:, rng.rand(rows, cols) < 0.05] = 0.0
    X[:, 2, :] = 0.0                              # a zero row
    X[m - 1, 3, :5] = 5e-324                      # subnormal words
    X[1, 4, :9] = X[0, 4, :9] * np.array([1, -1, .5, -.5, .75, .25, -.25, .3, 0.])   # near the first
    return X


@pytest.mark.parametrize("m,LA,LB", [
    (2, 110, 125), (2, 126, 157), (2, 158, 189), (2, 190, 253), (2, 254, 120), (2, 317, 318),
    (2, 381, 112), (2, 119, 127), (2, 128, 129), (4, 212, 221), (4, 222, 253), (4, 254, 255),
    (4, 317, 230), (4, 318, 216), (4, 381, 240), (4, 240, 248),
])
@pytest.mark.parametrize("trans", [False, True])
def test_fixed_point_lengths(mw, cuda, m, LA, LB, trans):
    M, N, K = 7, 9, 70
    A, B = entries(m, M, K, LA), np.ascontiguousarray(entries(m, N, K, LB).transpose(0, 2, 1))
    if trans:
        A, B = (np.ascontiguousarray(X.transpose(0, 2, 1)) for X in (A, B))
    plan = mw.mw_plan_gemm(m, "crt", M, N, K, 0, 0)
    plan.range_A = plan.range_B = 3000
    plan.S_A, plan.S_B = LA, LB
    need, total = LA + LB + 1 + np.log2(K), len(mw.crt_moduli())
    plan.D = next(n for n in range(1, total + 1) if mw.mw_crt_moduli_product_bits(n) > need)
    C, ws, off, _ = run_crt(mw, cuda, A, B, plan, trans, trans)
    rp = crt.ResidueProduct(A, B, LA, LB, mw.crt_moduli(plan.D), transA=trans, transB=trans)
    assert rp.A.in_range and rp.B.in_range
    Kp = -(-K // 64) * 64
    for X, R, at in ((rp.A, M, off[1]), (rp.B, N, off[2])):
        planes = ws[at:at + 2 * plan.D * R * Kp].view(torch.bfloat16)
        got = bf16_to_int(planes.reshape(plan.D, R, Kp))
        assert np.array_equal(got[:, :, :K], X.residues) and not got[:, :, K:].any()
    assert np.array_equal(C, rp.result())
