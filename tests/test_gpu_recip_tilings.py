"""Tilings of the tensor-core reciprocal sums that test_gpu_recip_tc.py's shapes do not reach: phase
rows read from global memory (one and two N tiles), two N tiles with staged rows, three blocks of 1024
charges, an odd last charge of a pair.  The tiling that each system takes is checked on the host in
test_recip_shapes.py.  Against the oracle, and the reciprocal part against the CUDA-core kernels with
test_gpu_recip_tc.py's bounds."""
import numpy as np
import pytest

import oracle
import workloads
from _gpuutil import TOL_FP64, gpu_all, grad_err, rel_max

pytestmark = pytest.mark.gpu

CASES = {
    "unstaged": dict(seed=51, n_waters=12, kmax=(4, 48, 24)),
    "unstaged_two_ntiles": dict(seed=52, n_waters=10, kmax=(3, 47, 49)),
    "two_ntiles": dict(seed=53, n_waters=12, kmax=(4, 4, 33)),
    "three_blocks": dict(seed=54, n_waters=800, box_A=31.0, kmax=(6, 5, 4)),
}


def _recip(name):
    def setup(h):
        import paper_2408_03273_gb300 as q
        h.set_recip_method(getattr(q, name))
    return setup


@pytest.mark.parametrize("name", list(CASES))
def test_tilings_against_oracle_and_cuda_cores(name):
    kw = dict(CASES[name])
    s = workloads.small_system(kw.pop("seed"), n_atoms=3, lmax=1, **kw)
    ref = oracle.energy(s)
    ref.update(oracle.forces(s))
    t = gpu_all(s, precision=0, setup=_recip("QMMM_RECIP_TENSOR"))
    assert rel_max(t["phi"], ref["phi"]) < TOL_FP64
    for k in ("dE_dRqm", "dE_dRmm", "dE_dq"):
        assert grad_err(t[k], ref, k, False) < TOL_FP64, k
    c = gpu_all(s, precision=0, setup=_recip("QMMM_RECIP_CUDA_CORES"))
    lr = oracle.ewald_phi(s, oracle.EW_LR)
    dq_lr, dR_lr = oracle.ewald_mm(s, oracle.multipoles(s), oracle.EW_LR)
    assert np.max(np.abs(t["phi"] - c["phi"])) < 1e-11 * np.max(np.abs(lr))
    assert np.max(np.abs(t["dE_dq"] - c["dE_dq"])) < 1e-11 * np.max(np.abs(dq_lr))
    assert np.max(np.abs(t["dE_dRmm"] - c["dE_dRmm"])) < 1e-11 * np.max(np.abs(dR_lr))
