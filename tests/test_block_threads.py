"""Block sizes of the class sweeps (csrc/sched.h, block_threads), compiled with the host C++ compiler:
a size chosen for a class is kept on every system; the 128-thread default is for sweeps of at most
four warps per SM."""
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
    int n, nsm, tiles[64], ns[64], asked[64], threads[64];
    if (std::scanf("%d %d", &n, &nsm) != 2) return 1;
    for (int c = 0; c < n; ++c)
        if (std::scanf("%d %d %d", &tiles[c], &ns[c], &asked[c]) != 3) return 1;
    qmmm::block_threads(n, tiles, ns, nsm, asked, threads);
    for (int c = 0; c < n; ++c) std::printf("%d ", threads[c]);
    return 0;
}
"""


@pytest.fixture(scope="module")
def threads(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("blocks")
    (d / "drv.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "drv.cpp"), "-o", str(d / "drv")], check=True)

    def run(tiles, ns, asked, nsm=152):
        text = f"{len(tiles)} {nsm}\n" + "".join(f"{t} {s} {a}\n" for t, s, a in zip(tiles, ns, asked))
        out = subprocess.run([str(d / "drv")], input=text, capture_output=True, text=True, check=True).stdout
        return [int(x) for x in out.split()]

    return run


# (tiles, slices): 37 warps, exactly 4 x 152 = 608, 609, many; classes without pairs among them
@pytest.mark.parametrize("tiles,ns,default", [([30, 7, 0], [1, 1, 1], 128), ([100, 1, 0], [6, 8, 1], 128),
                                              ([100, 1, 0], [6, 9, 1], 256), ([9000, 40, 3], [1, 4, 16], 256)])
def test_chosen_sizes_are_kept(threads, tiles, ns, default):
    assert threads(tiles, ns, [0, 0, 0]) == [default] * 3
    assert threads(tiles, ns, [1024, 256, 384]) == [1024, 256, 384]
    assert threads(tiles, ns, [0, 640, 0]) == [default, 640, default]
