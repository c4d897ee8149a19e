"""Which kernel multiplies power series, and with how many CTAs and warps: series
whose digits leave room for the columns of fewer than four warps go to the inner-product
kernel; growing exponents get
a CTA a coefficient without two of them sharing one.  The library's host code on a stand-in
runtime of 152 SMs; no GPU."""
import pytest

import host_runtime


@pytest.fixture(scope="module")
def host(mw, tmp_path_factory):
    lib = host_runtime.link(mw, str(tmp_path_factory.mktemp("host")))
    if lib is None:
        pytest.skip("no C++ compiler")
    return lib


def launch(host, m, count, n, S):
    p = host.plan(m, "dot", 1, 1, n, 0, 0)
    p.S_A = p.S_B = S
    p.D = S + 1
    (l,) = host.launches(lambda: host.convolve(p, count, n))
    return ("series" if "series_kernel" in l[0] else "dot"), l[1], l[2] // 32


@pytest.mark.parametrize("m,count,n,S,kernel", [
    # digits beside four warps' columns, and beside three's
    (2, 600, 2944, 8, "series"), (2, 600, 3000, 8, "dot"), (4, 200, 2016, 12, "series"),
    (4, 200, 2050, 12, "dot"), (8, 76, 1120, 21, "series"), (8, 76, 1150, 21, "dot"),
])
def test_kernel(host, m, count, n, S, kernel):
    got, _, warps = launch(host, m, count, n, S)
    assert got == kernel
    assert kernel == "dot" or n < 512 or warps >= 4


def test_places_for_every_coefficient(host):
    # chunk of segment g on CTA (g + i0 / warps) mod ctas: 16 segments of one coefficient
    for m, S, n in ((8, 20, 16), (16, 36, 24), (8, 20, 44)):
        kernel, ctas, warps = launch(host, m, 1, n, S)
        assert kernel == "series"
        places = [(g + g // warps) % ctas for g in range(n)]
        assert len(set(places)) == n
