"""The block sizes that the class sweeps launch (qmmm_sweep_threads): an installed one on a system of
few warps, the 128-thread default there, and the 256-thread default above four warps per SM; results
in every shape against the oracle."""
import numpy as np
import pytest

import oracle
import workloads
from _gpuutil import TOL_FP64, TOL_MIXED, check_V, gpu_all, grad_err

pytestmark = pytest.mark.gpu

KINDS = {0: (0, 2), 1: (1, 3)}  # precision -> (V sweep kind, adjoint sweep kind)
CHARGE_LANES = 3                # mixed adjoint: 256-thread blocks in every variant


@pytest.fixture(scope="module")
def small():
    # every angular class, some 40 tiles of 32 pairs and 39 charges: far below four warps per SM
    s = workloads.small_system(seed=111, n_atoms=4, lmax=3, nprim=(1, 4), n_waters=14)
    ref = oracle.energy(s)
    ref.update(oracle.forces(s))
    return s, ref


def _sizes(h, kind, size):
    return [size if n else 0 for n in h.info["n_prim_pairs_class"]]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", ["default", "256", "wide"])
def test_launched_block_sizes(small, precision, shape):
    s, ref = small

    def setup(h):
        for k in KINDS[precision]:
            wide = h.tuning(k)["wide"]
            if shape == "256":
                h.set_tuning(k, [256] * 10)
            elif shape == "wide":
                h.set_tuning(k, [w or 256 for w in wide])
            if k == CHARGE_LANES or shape == "256":
                want = _sizes(h, k, 256)
            elif shape == "default":
                want = _sizes(h, k, 128)
            else:
                want = [(w or 256) if n else 0 for w, n in zip(wide, h.info["n_prim_pairs_class"])]
            assert h.sweep_threads(k) == want, k

    g = gpu_all(s, precision=precision, screen_tol=0.0, setup=setup)
    tol = TOL_FP64 if precision == 0 else TOL_MIXED
    check_V(g["V"], ref["V"], precision)
    for key in ("dE_dRqm", "dE_dRmm", "dE_dq"):
        assert grad_err(g[key], ref, key, precision == 1) < tol, key


def test_default_blocks_of_a_large_sweep():
    import paper_2408_03273_gb300 as q
    h = q.Handle(workloads.config2_active_site())
    try:
        for k in range(4):
            assert h.sweep_threads(k) == _sizes(h, k, 256)
        with pytest.raises(q.QMMMError):
            h.sweep_threads(4)
    finally:
        h.close()


def test_plan_of_another_shape_replaces_the_installed_one(small):
    # an installed shape holds until it is replaced; the autotuner starts from the default again
    import paper_2408_03273_gb300 as q
    h = q.Handle(small[0])
    try:
        h.set_tuning(0, [256] * 10)
        assert h.sweep_threads(0) == _sizes(h, 0, 256)
        h.autotune(q.QMMM_TUNE_V)
        t = h.tuning(0)
        got = h.sweep_threads(0)
        for c, n in enumerate(h.info["n_prim_pairs_class"]):
            assert got[c] == (0 if not n else 128 if t["threads"][c] == 256 else t["wide"][c]), c
        assert np.all(np.isfinite(h.vpot()[0]))
    finally:
        h.close()
