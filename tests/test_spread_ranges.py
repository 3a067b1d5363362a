"""Pair-batch ranges of the mixed adjoint on small systems (csrc/sched.h, spread_ranges), compiled with
the host C++ compiler: the items follow the SM count that they are given, never fall below the plain
cut and never outnumber the batches."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_03273_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "sched.h"
int main()
{
    int gx, ntile, nbatch, nsm;
    while (std::scanf("%d %d %d %d", &gx, &ntile, &nbatch, &nsm) == 4)
        std::printf("%d\n", qmmm::spread_ranges(gx, ntile, nbatch, nsm));
    return 0;
}
"""


@pytest.fixture(scope="module")
def ranges(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("spread")
    (d / "drv.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "drv.cpp"), "-o", str(d / "drv")], check=True)

    def run(cases):
        text = "".join("%d %d %d %d\n" % c for c in cases)
        out = subprocess.run([str(d / "drv")], input=text, capture_output=True, text=True, check=True).stdout
        return [int(x) for x in out.split()]

    return run


def test_spread_follows_the_sm_count(ranges):
    # one range, three charge tiles, 400 batches: as many ranges as fill the SMs
    assert ranges([(1, 3, 400, n) for n in (1, 2, 3, 76, 152)]) == [1, 1, 1, 25, 50]
    # fewer batches than that; the plain cut already at the line; no charges
    assert ranges([(1, 3, 7, 152), (51, 3, 408, 152), (50, 3, 400, 152), (2, 0, 16, 152)]) == [7, 51, 50, 2]
    cases = [(g, t, 8 * g - 5, n) for g in (1, 2, 17, 160) for t in (1, 2, 9, 200) for n in (76, 132, 152)]
    for (g, t, b, n), r in zip(cases, ranges(cases)):
        assert g <= r <= max(g, b) and (r == g or r * t <= n), (g, t, b, n)
        if r < b and g * t < n:  # no finer cut would fit
            assert (r + 1) * t > n
