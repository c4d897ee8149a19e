"""Which kernel multiplies power series, and with how many CTAs and warps: growing
exponents get a CTA a coefficient without two of them sharing one.  The library's host code on a stand-in
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


def test_places_for_every_coefficient(host):
    # chunk of segment g on CTA (g + i0 / warps) mod ctas: 16 segments of one coefficient
    for m, S, n in ((8, 20, 16), (16, 36, 24), (8, 20, 44)):
        kernel, ctas, warps = launch(host, m, 1, n, S)
        assert kernel == "series"
        places = [(g + g // warps) % ctas for g in range(n)]
        assert len(set(places)) == n
