"""The moment kernels (multipoles, octupoles, Fock term, Pulay gradient) at a density that is not
symmetric, against the oracle, which takes gamma_{nu mu} for the atom of mu: symmetric densities leave
the kernels' antisymmetric sums out.  Shell recipes cover one to ten components per shell (one to ten
warps per block) and pair counts around a multiple of 32."""
import numpy as np
import pytest

import oracle
import workloads
from _gpuutil import TOL_FP64, rel_max

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spec,natm", [("1s", 2), ("2s1p", 3), ("1s1p1d", 3), ("1s1p1d1f", 2), ("1d1f", 4)])
def test_moments_at_a_nonsymmetric_density(spec, natm):
    import paper_2408_03273_gb300 as q
    s = workloads.small_system(77 + natm, n_atoms=natm, lmax=3, shells_per_atom=spec)
    rng = np.random.default_rng(5)
    dm = s.dm + 0.3 * s.dm.std() * rng.standard_normal(s.dm.shape)
    h = q.Handle(s)
    try:
        h.vpot()
        _, M, F = h.ewald(dm, want_F=True)
        _, octu = h.octupole_error(dm, 3.0, 0.5, 4, want_octupoles=True)
        gq, _, _ = h.forces(dm)
        gq_sym, _, _ = h.forces(0.5 * (dm + dm.T))
    finally:
        h.close()
    phi = oracle.ewald_phi(s)
    assert rel_max(M, oracle.multipoles(s, dm)) < TOL_FP64
    assert rel_max(octu, oracle.octupoles(s, dm)) < TOL_FP64
    assert rel_max(F, oracle.fock_ii(s, phi)) < TOL_FP64
    # the region-I sweep sees gamma + gamma^T only: the difference is the multipole part's
    d = lambda x: oracle.pulay_grad(s, phi, x) + oracle.tensor_grad_qm(s, oracle.multipoles(s, x), phi)  # noqa: E731
    want = d(dm) - d(0.5 * (dm + dm.T))
    scale = np.max(np.abs(d(dm)))
    assert np.max(np.abs((gq - gq_sym) - want)) < TOL_FP64 * max(scale, np.max(np.abs(gq)))
