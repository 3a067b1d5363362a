"""Tilings of the two tensor-core reciprocal sums (tc_sf_shape, tc_mmr_shape of the built library, host
code): the limits of the hardware over every kmax, and the tiling that each system of
test_gpu_recip_tc.py and test_gpu_recip_tilings.py takes, so that a new tiling cannot leave a branch
of the kernels without a test unnoticed."""
import os
import shutil
import subprocess

import pytest

import paper_2408_03273_gb300 as q
from test_gpu_recip_tilings import CASES

CSRC = os.path.join(os.path.dirname(os.path.abspath(q.__file__)), "csrc")

DRIVER = r"""
#include <cstdio>
#include "qmmm_internal.h"
using namespace qmmm;
int main()
{
    int kx, ky, kz, n;
    while (std::scanf("%d %d %d %d", &kx, &ky, &kz, &n) == 4) {
        EwaldDev e{};
        e.kmax[0] = kx;
        e.kmax[1] = ky;
        e.kmax[2] = kz;
        e.nmm = n;
        TcShape s;
        MmrShape m[2];
        tc_sf_shape(e, s);
        tc_mmr_shape(e, 5, MMR_NP_FP64, m[0]);
        tc_mmr_shape(e, 3, MMR_NP_MIXED, m[1]);
        std::printf("%d %d %d %d %d %d", (int)s.staged, s.ntiles, s.ntr, s.mtiles, s.nkb, s.NL);
        for (const MmrShape &x : m)
            std::printf(" %d %d %d %d %d", (int)x.supported, x.ntiles, x.nr, x.nr_last, x.nstg);
        std::printf("\n");
    }
    return 0;
}
"""
SF = ("staged", "ntiles", "ntr", "mtiles", "nkb", "NL")
MM = ("supported", "ntiles", "nr", "nr_last", "nstg")


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    q.load()
    lib = q.library_path()
    d = tmp_path_factory.mktemp("shapes")
    (d / "drv.cu").write_text(DRIVER)
    subprocess.run([nvcc, "-std=c++17", "-I" + CSRC, str(d / "drv.cu"), "-o", str(d / "drv"), lib,
                    "-Xlinker", "-rpath=" + os.path.dirname(lib)], check=True, capture_output=True)

    def run(cases):
        text = "".join("%d %d %d %d\n" % c for c in cases)
        out = subprocess.run([str(d / "drv")], input=text, capture_output=True, text=True, check=True).stdout
        res = []
        for line in out.splitlines():
            v = [int(x) for x in line.split()]
            res.append((dict(zip(SF, v[:6])), dict(zip(MM, v[6:11])), dict(zip(MM, v[11:16]))))
        return res

    return run


def test_structure_factor_tilings_of_the_gpu_tests(shapes):
    # (kmax, charges) of test_gpu_recip_tc.py and of the cases named in test_gpu_recip_tilings.py
    small, k40 = shapes([(5, 5, 5, 36), (40, 40, 40, 36)])
    assert small[0]["staged"] and small[0]["ntiles"] == 1 and small[0]["nkb"] == 1
    assert k40[0]["staged"] and k40[0]["ntiles"] == 2
    names = list(CASES)
    got = dict(zip(names, shapes([CASES[n]["kmax"] + (3 * CASES[n]["n_waters"],) for n in names])))
    for name, want in (("unstaged", dict(staged=0, ntiles=1, ntr=64)), ("unstaged_two_ntiles", dict(staged=0, ntiles=2)),
                       ("two_ntiles", dict(staged=1, ntiles=2)), ("three_blocks", dict(staged=1, nkb=3))):
        for k, v in want.items():
            assert got[name][0][k] == v, (name, k)
    # charges dropped next to the QM atoms must not change the count of blocks of 1024
    assert 2 * 1024 + 100 < 3 * CASES["three_blocks"]["n_waters"] < 3 * 1024


def test_tilings_fit_the_hardware(shapes):
    cases = [(kx, ky, kz, 600) for kx in (1, 16, 40, 56) for ky in range(1, 57) for kz in range(1, 57)]
    smem = 232448
    for (kx, ky, kz, _), (sf, *mm) in zip(cases, shapes(cases)):
        NY, NZ = 2 * ky + 1, 2 * kz + 1
        assert sf["ntr"] % 16 == 0 and sf["ntr"] * sf["ntiles"] >= NZ and 7 * sf["ntr"] <= 512
        assert sf["NL"] == (2 * kx + 1) * NY and sf["mtiles"] * 128 >= sf["NL"]
        stage = 7 * (128 * 64 + sf["ntr"] * 64)
        rows = (127 // NY + 2 + NY) * 320  # phase rows of a chunk of 32 charges
        assert 2 * stage + 256 <= smem
        assert bool(sf["staged"]) == (2 * (stage + rows) + 256 <= smem)
        # where the phase rows are staged: everywhere up to ky = 45, beyond that unless the N tiles
        # are 64 rows wide
        assert bool(sf["staged"]) == (ky <= 45 or sf["ntr"] < 64), (ky, kz)
        for m, nacc, planes in zip(mm, (5, 3), (7, 5)):
            fits = 2 * (kx + 1) <= 512 // nacc // 16 * 16
            assert bool(m["supported"]) == (fits and NZ >= 8), (kx, kz)
            if m["supported"]:
                assert max(m["nr"], m["nr_last"]) * nacc <= 512
                need = m["nstg"] * planes * (4096 + m["nr"] * 32) + (NZ + 4 * 3) * 1040 + 256
                assert m["nstg"] in (2, 3) and need <= smem
