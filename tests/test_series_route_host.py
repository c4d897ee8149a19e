"""Which kernel multiplies power series, and with how many CTAs and warps: so few
coefficients that inner products fill the SMs once, and series whose digits leave room for
the columns of fewer than four warps, go to the inner-product kernel; growing exponents get
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
    (2, 1, 456, 7, "dot"), (2, 1, 457, 7, "series"), (2, 57, 8, 5, "dot"), (2, 58, 8, 5, "series"),
    (4, 1, 304, 11, "dot"), (4, 1, 305, 11, "series"), (4, 12, 24, 10, "dot"), (4, 13, 24, 10, "series"),
    (8, 1, 64, 20, "series"), (8, 1, 65, 20, "dot"), (8, 1, 304, 20, "dot"), (8, 1, 305, 20, "series"),
    (8, 4, 64, 20, "series"), (16, 1, 64, 36, "series"), (16, 1, 200, 36, "series"),
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
