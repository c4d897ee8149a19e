"""When an entry's fixed-point value T = sum_j trunc(x_j 2^F) is taken for certainly in
[-2^(wS-1), 2^(wS-1)) without a check of its digits (surely_in_range in csrc/mw_column.cuh,
compiled for the host): never for a T outside, and always for zeros and for normalised
entries whose exponent the grid covers."""
import math
import os
import random
import shutil
import struct
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2606_20863_gb300", "csrc")
PROGRAM = """
#include <cstdio>
#include "mw_column.cuh"
int main() {
  unsigned m, h0, h1;
  int top;
  while (scanf("%u %x %x %d", &m, &h0, &h1, &top) == 4) {
    bool r = m == 2 ? mw::surely_in_range<2>(h0, h1, top) : m == 4 ? mw::surely_in_range<4>(h0, h1, top)
           : m == 8 ? mw::surely_in_range<8>(h0, h1, top) : mw::surely_in_range<16>(h0, h1, top);
    printf("%d\\n", r);
  }
}
"""


@pytest.fixture(scope="module")
def sure(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("range")
    (d / "range.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-o", str(d / "range"), str(d / "range.cpp")],
                   check=True)

    def run(entries, tops):
        def high(x):
            return struct.unpack("<Q", struct.pack("<d", abs(x)))[0] >> 32 << 1
        lines = ["%d %x %x %d" % (len(x), high(x[0]), max(high(v) for v in x[1:]), t)
                 for x, t in zip(entries, tops)]
        out = subprocess.run([str(d / "range")], input="\n".join(lines), capture_output=True, text=True,
                             check=True).stdout.split()
        return [o == "1" for o in out]
    return run


@pytest.mark.parametrize("m", [2, 4, 8, 16])
def test_never_outside(sure, m):
    """|T| <= 2^F sum_j |x_j| < 2^(wS-1) is sum_j |x_j| < 2^(top + 1) for top = wS - 2 - F:
    exact sums of the magnitudes, words at every offset from the edge."""
    r = random.Random(m)
    entries, tops = [], []
    for _ in range(4000):
        top, most = r.choice([-1030, -1000, -3, 0, 40, 1000]), r.choice([2, 0, -1, -2, -3, -4])
        entries.append([math.ldexp(r.choice([1.0, 1.5, 2 - 2.0 ** -52, 0.0]),
                                   max(top + r.randint(-7, most), -1074)) for _ in range(m)])
        tops.append(top)
    got = sure(entries, tops)
    assert any(got) and not all(got)
    for x, top, ok in zip(entries, tops, got):
        total = sum(int(math.frexp(v)[0] * 2 ** 53) << (1200 + math.frexp(v)[1] - 53) for v in x)
        assert not ok or total < 1 << (1200 + top + 1)      # in units of 2^-1200


@pytest.mark.parametrize("m", [2, 4, 8, 16])
def test_zeros_and_normalised_entries(sure, m):
    for top in (-1000, -20, 0, 3, 900):
        normal = [math.ldexp(1 - 2.0 ** -53, top)] + [math.ldexp(1.0, top - 53 * j) if top - 53 * j > -1022
                                                     else 0.0 for j in range(1, m)]
        small = [math.ldexp(v, -5) for v in normal]
        later = [0.0] * (m - 1) + [math.ldexp(1.0, top - 6)]
        assert sure([[0.0] * m, normal, small, later], [top] * 4) == [True] * 4
