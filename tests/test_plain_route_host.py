"""Which kernel multiplies the pieces of MW_PLAIN: 4 x 8 outputs a CTA, or whole tiles where
that is the faster one (the measured times stand beside the rule in mw_plain.cu) or the
only one.  The library's host code on a stand-in runtime; no GPU."""
import pytest

import host_runtime


@pytest.fixture(scope="module")
def host(mw, tmp_path_factory):
    lib = host_runtime.link(mw, str(tmp_path_factory.mktemp("host")))
    if lib is None:
        pytest.skip("no C++ compiler")
    return lib


@pytest.mark.parametrize("m,M,N,K,w,split", [
    (2, 64, 64, 64, 0, True), (2, 512, 512, 300, 0, True), (2, 1024, 1024, 40, 0, True),
    (4, 400, 400, 300, 0, True), (4, 512, 512, 64, 0, False), (4, 512, 512, 300, 0, False),
    (4, 512, 512, 64, 8, False), (4, 512, 512, 64, 5, False), (4, 100, 2000, 100, 7, True),
    (4, 100, 2000, 100, 5, False), (8, 256, 256, 256, 0, True), (8, 1024, 1024, 40, 16, False),
    (8, 18, 20, 40, 4, False), (4, 3 << 20, 8, 8, 5, True),
])
def test_kernel(host, m, M, N, K, w, split):
    p = host.plan(m, "plain", M, N, K, 8, 8, w)
    names = [l[0] for l in host.launches(lambda: host.gemm(p, M, N, K))]
    assert any("plain_split_kernel" in n for n in names) == split
    assert any("plain_kernel" in n for n in names) == (not split)
