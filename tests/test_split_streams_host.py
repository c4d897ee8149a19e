"""Where the pieces of a small product's two operands are cut: in one launch for entries
of up to 256 bits, beside each other on two streams for wider ones (one after the other
where the operands as stored fill the GPU each).  The library's host code on a stand-in
runtime; no GPU."""
import pytest

import host_runtime


@pytest.fixture(scope="module")
def host(mw, tmp_path_factory):
    lib = host_runtime.link(mw, str(tmp_path_factory.mktemp("host")))
    if lib is None:
        pytest.skip("no C++ compiler")
    return lib


@pytest.mark.parametrize("m,range_,M,N,K,ta,tb,together", [
    (2, 4, 64, 64, 64, 0, 0, True), (4, 4, 64, 64, 64, 1, 0, True), (4, 4, 1, 1, 1, 0, 0, True),
    (4, 60, 64, 64, 64, 0, 0, False), (8, 4, 64, 64, 64, 0, 0, False),
    (8, 4, 8, 8, 8, 1, 1, False), (16, 4, 32, 32, 512, 1, 0, False), (16, 4, 64, 64, 64, 0, 1, False),
])
def test_wide_entries_on_two_streams(host, m, range_, M, N, K, ta, tb, together):
    p = host.plan(m, "ozaki", M, N, K, range_, range_)
    ls = host.launches(lambda: host.gemm(p, M, N, K, ta, tb))
    cuts = [l for l in ls if "pieces_" in l[0]]
    if together:
        assert len(cuts) == 1 and "pieces_pair" in cuts[0][0] and cuts[0][4] == 0
    else:
        assert len(cuts) == 2 and cuts[0][4] == 0 and cuts[1][4] != 0


@pytest.mark.parametrize("m,range_,n,ta,tb,two", [
    (4, 60, 256, 0, 0, True), (4, 60, 290, 0, 0, False), (4, 60, 362, 0, 0, False),
    (4, 60, 363, 0, 0, True), (4, 60, 290, 1, 0, True), (4, 60, 290, 0, 1, True),
    (8, 4, 300, 0, 0, False), (8, 4, 300, 1, 1, True),
])
def test_wide_entries_that_fill_the_gpu(host, m, range_, n, ta, tb, two):
    p = host.plan(m, "ozaki", n, n, n, range_, range_)
    cuts = [l for l in host.launches(lambda: host.gemm(p, n, n, n, ta, tb)) if "pieces_" in l[0]]
    assert len(cuts) == 2 and (cuts[1][4] != 0) == two


@pytest.mark.parametrize("m", [2, 4, 8, 16])
@pytest.mark.parametrize("S", [1, 9, 20, 31, 32, 47])
def test_plans_of_any_width(host, m, S):
    # pieces a caller chose: m = 16 has no kernel for entries of up to 256 bits
    p = host.plan(m, "ozaki", 16, 16, 16, 4, 4)
    p.S_A, p.S_B, p.D = S, 1, S
    for ta, tb in ((0, 0), (1, 0), (0, 1), (1, 1)):
        cuts = [l for l in host.launches(lambda: host.gemm(p, 16, 16, 16, ta, tb)) if "pieces_" in l[0]]
        assert len(cuts) == (1 if m < 16 and 8 * S + 3 <= 256 else 2)
