"""Where both operands' exponents are taken in one launch: not for reductions so long that
a warp a row takes longer than the passes over chunks, nor for very many short rows (the
measured limits stand beside the rule in mw_split.cu).  The library's host code on a
stand-in runtime; no GPU."""
import pytest

import host_runtime


@pytest.fixture(scope="module")
def host(mw, tmp_path_factory):
    lib = host_runtime.link(mw, str(tmp_path_factory.mktemp("host")))
    if lib is None:
        pytest.skip("no C++ compiler")
    return lib


def together(ls):
    pair = sum("exps_pair" in l[0] for l in ls)
    apart = sum("exps_rows" in l[0] or "exps_cols" in l[0] for l in ls)
    assert (pair, apart) in ((1, 0), (0, 2))
    return pair == 1


@pytest.mark.parametrize("m,mode,M,N,K,want", [
    (2, "ozaki", 64, 64, 64, True), (2, "ozaki", 32, 32, 1024, True),
    (2, "ozaki", 128, 128, 2048, False), (4, "ozaki", 32, 32, 1024, True),
    (4, "ozaki", 32, 32, 2048, False), (4, "crt", 32, 32, 2048, False),
    (4, "crt", 32, 32, 1024, True), (8, "ozaki", 32, 32, 512, True),
    (8, "ozaki", 32, 32, 2048, False), (8, "ozaki", 1, 1, 2048, False),
    (16, "ozaki", 32, 32, 512, True), (16, "ozaki", 1, 1, 2048, False),
    (2, "ozaki", 1024, 1024, 1024, False),
])
def test_products(host, m, mode, M, N, K, want):
    p = host.plan(m, mode, M, N, K, 4, 4)
    assert together(host.launches(lambda: host.gemm(p, M, N, K))) == want


@pytest.mark.parametrize("m,M,N,K,ta,tb,want", [
    (2, 2048, 2048, 1024, 0, 0, True), (2, 64, 64, 2048, 1, 1, True),
    (4, 128, 128, 1024, 0, 0, True), (4, 128, 128, 2048, 0, 0, False),
    (8, 512, 512, 1024, 0, 0, True), (8, 512, 512, 2048, 0, 0, False),
    (16, 1000, 1000, 1000, 0, 0, True), (16, 32, 32, 2048, 0, 0, False),
    (2, 1 << 19, 8, 16, 1, 0, False), (2, 1 << 19, 8, 64, 1, 0, True),
    (2, 1 << 19, 8, 2, 0, 0, True), (2, 1 << 19, 8, 256, 0, 0, False),
    (2, 8, 1 << 20, 4, 0, 0, False), (2, 65536, 8, 4, 1, 0, True),
])
def test_spread(host, m, M, N, K, ta, tb, want):
    assert together(host.launches(lambda: host.measure(m, M, N, K, ta, tb))) == want
