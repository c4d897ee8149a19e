"""Every form runs on a second device of the same process: a kernel's limit of dynamic
shared memory is granted for one device at a time, so each device asks for it.  The
library's host code on a stand-in runtime with two devices; no GPU."""
import pytest

import host_runtime


@pytest.fixture(scope="module")
def host(mw, tmp_path_factory):
    lib = host_runtime.link(mw, str(tmp_path_factory.mktemp("host")))
    if lib is None:
        pytest.skip("no C++ compiler")
    return lib


def calls(h):
    """Calls of every form, some of each with more than 48 KB."""
    for m, mode, M, N, K, ta, tb, ra in [
            (2, "plain", 64, 64, 64, 0, 0, 4), (4, "plain", 64, 64, 256, 0, 0, 4),
            (8, "plain", 40, 40, 64, 0, 0, 4),
            (2, "ozaki", 64, 64, 64, 0, 0, 4), (2, "ozaki", 1024, 1024, 1024, 0, 0, 4),
            (4, "ozaki", 64, 64, 8192, 0, 0, 4), (8, "ozaki", 64, 64, 64, 1, 0, 4),
            (16, "ozaki", 64, 64, 64, 1, 0, 4),
            (2, "crt", 64, 64, 64, 0, 0, 4), (4, "crt", 300, 300, 300, 1, 0, 8)]:
        p = h.plan(m, mode, M, N, K, ra, ra)
        yield (mode, m, K), lambda p=p, a=(M, N, K, ta, tb): h.gemm(p, *a)
    for m, count, n in [(2, 300, 600), (4, 300, 600), (8, 2000, 128), (16, 100, 128), (8, 1, 1700)]:
        p = h.plan(m, "dot", 1, 1, n, 4, 4)
        yield ("series", m, n), lambda p=p, a=(count, n): h.convolve(p, *a)
    for m in (8, 16):
        p = h.plan(m, "dot", 1, 1, 1000, 4, 4)
        yield ("dot", m, 1000), lambda p=p: h.dot(p, 100, 1000)
        p = h.plan(m, "ozaki", 40, 40, 40, 4, 4)
        yield ("batch", m, 40), lambda p=p: h.batch(p, [(40, 30, 40), (20, 40, 10)])


def test_second_device(host):
    host.device(0)
    first = {key: host.launches(call) for key, call in calls(host)}
    assert all(first.values())
    assert {key[0] for key, ls in first.items() if any(l[3] > 49152 for l in ls)} == {
        "plain", "ozaki", "crt", "series", "dot", "batch"}
    host.device(1)
    for key, call in calls(host):
        ls = host.launches(call)
        assert [l[:4] for l in ls] == [l[:4] for l in first[key]], key
    host.device(0)
