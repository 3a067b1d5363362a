"""Charge slices of the fine-grained class sweeps (csrc/sched.h): fine_slices and slice_order,
compiled with the host C++ compiler and checked against their rule -- within the bounds, blocks no
longer than a quarter of the ideal sweep unless a bound stops the slicing, and launched longest
first."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_03273_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "sched.h"
int main()
{
    int n, nch, nsm, maxsl;
    while (std::scanf("%d %d %d %d", &n, &nch, &nsm, &maxsl) == 4) {
        int tiles[64], ns[64], order[64];
        double w[64], setup[64];
        for (int c = 0; c < n; ++c)
            if (std::scanf("%d %lf %lf", &tiles[c], &w[c], &setup[c]) != 3) return 1;
        qmmm::fine_slices(n, tiles, w, setup, nch, nsm, maxsl, ns);
        qmmm::slice_order(n, tiles, w, ns, order);
        for (int c = 0; c < n; ++c) std::printf("%d ", ns[c]);
        for (int c = 0; c < n; ++c) std::printf("%d ", order[c]);
        std::printf("\n");
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def fine(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("fine")
    (d / "drv.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "drv.cpp"), "-o", str(d / "drv")], check=True)

    def run(tiles, w, setup, nch, nsm, maxsl):
        n = len(tiles)
        text = f"{n} {nch} {nsm} {maxsl}\n" + "".join(f"{t} {a!r} {b!r}\n" for t, a, b in zip(tiles, w, setup))
        out = subprocess.run([str(d / "drv")], input=text, capture_output=True, text=True, check=True).stdout.split()
        return np.array(out[:n], int), np.array(out[n:], int)

    return run


@pytest.mark.parametrize("nch", [1, 31, 64, 1000, 20000])
@pytest.mark.parametrize("tiles", [[0] * 4, [1, 0, 0, 0], [1, 1, 1, 1], [4000, 900, 60, 1], [100000, 0, 3, 20]])
def test_slices_follow_the_rule(fine, tiles, nch):
    w, setup, nsm = [1.0, 3.5, 9.0, 40.0], [4.0, 20.0, 40.0, 90.0], 152
    for maxsl in (1, 8, 64):
        ns, order = fine(tiles, w, setup, nch, nsm, maxsl)
        assert sorted(order) == list(range(4))
        ideal = sum(t * a for t, a in zip(tiles, w)) / (8 * nsm)
        for c in range(4):
            most = max(1, min(maxsl, int(nch / max(32.0, setup[c]))))
            assert 1 <= ns[c] <= most
            if tiles[c] == 0:
                assert ns[c] == 1
            elif ns[c] < most:  # no bound stopped it: short enough, and no finer than asked for
                assert 4 * w[c] / ns[c] <= ideal * 1.001
                assert ns[c] == 1 or 4 * w[c] / (ns[c] - 1) >= ideal * 0.999
        t = [w[c] / ns[c] if tiles[c] else -1.0 for c in order]
        assert all(a >= b for a, b in zip(t, t[1:]))
