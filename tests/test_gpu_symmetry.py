"""V is symmetric bit for bit whatever the number of its contributions: shell pairs of 256 primitive
pairs (nine tiles of 32), several chunks of region-I charges, and the charge slices of a batch's mixed
frames, which all add into one matrix.  Repeated, since the order of the additions varies from run to
run; the values against the oracle."""
import numpy as np
import pytest

import oracle
import workloads
from _gpuutil import check_V

pytestmark = pytest.mark.gpu

CASES = {
    "nine_tiles": dict(seed=140, n_atoms=3, lmax=3, nprim=(16, 16), n_waters=8),
    # a width of region I beyond one chunk of 4096 charges
    "chunks": dict(seed=108, n_atoms=2, lmax=1, nprim=(3, 5), n_waters=5400, box_A=40.0, cutoff_A=19.5,
                   alpha_invA=0.3, kmax=(6, 6, 6)),
}


@pytest.fixture(scope="module", params=list(CASES))
def case(request):
    s = workloads.small_system(**CASES[request.param])
    return s, oracle.vpot(s)


@pytest.mark.parametrize("precision", [0, 1])
def test_v_is_symmetric(case, precision):
    import paper_2408_03273_gb300 as q
    s, ref = case
    h = q.Handle(s, precision=precision, screen_tol=0.0)
    try:
        for _ in range(8):
            V, _ = h.vpot()
            assert np.array_equal(V, V.T)
        check_V(V, ref, precision)
    finally:
        h.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_batch_v_is_symmetric(case, precision):
    torch = pytest.importorskip("torch")
    import paper_2408_03273_gb300 as q
    s, ref = case
    hs = [q.Handle(s, precision=precision, screen_tol=0.0) for _ in range(2)]
    try:
        dm = [torch.as_tensor(s.dm, device="cuda") for _ in hs]
        V = [torch.zeros_like(d) for d in dm]
        b = q.Batch(hs)
        try:
            for _ in range(4):
                b.run(dm, V)
                for v in V:
                    assert torch.equal(v, v.T)
                    check_V(v.cpu().numpy(), ref, precision)
        finally:
            b.close()
    finally:
        for h in hs:
            h.close()


@pytest.mark.parametrize("natm,lmax,nao", [(1, 0, 1), (32, 0, 32), (33, 0, 33), (9, 2, 90)])
def test_mirror_over_ragged_tiles(natm, lmax, nao):
    # orders of V around the mirror's 32 x 32 tiles, down to a single function
    import paper_2408_03273_gb300 as q
    s = workloads.small_system(seed=141 + natm, n_atoms=natm, lmax=lmax, nprim=(1, 2), n_waters=40, radius_A=3.0)
    assert s.nao == nao
    h = q.Handle(s, screen_tol=0.0)
    try:
        V, _ = h.vpot()
        assert np.array_equal(V, V.T)
        check_V(V, oracle.vpot(s), 0)
    finally:
        h.close()
