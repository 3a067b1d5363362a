"""A batch of FP64 frames whose sweep scratch a plain call has moved: the graph is recorded again for
the new buffer, and results stay those of the plain calls, on the recording run and on a replay."""
import pytest

import workloads
from test_gpu_batch import _close, _dev_outputs, _plain

pytestmark = pytest.mark.gpu

CLASSES = 10


def test_batch_after_a_plain_call_moved_the_scratch():
    torch = pytest.importorskip("torch")
    import paper_2408_03273_gb300 as q
    frames = [workloads.small_system(seed=130 + i, n_atoms=4 + i, lmax=2, nprim=(1, 3), n_waters=120) for i in range(2)]
    # one charge slice for every class but (s,s); then the model's weights, which cut every class into as
    # many slices as its charges allow: several times the pair sums, beyond the scratch sized for the
    # first plan
    coarse = ([256] * CLASSES, [1.0] + [1e-9] * (CLASSES - 1))
    hs = [q.Handle(s) for s in frames]
    try:
        for h in hs:
            h.set_tuning(0, *coarse)
        dm = [torch.as_tensor(s.dm, device="cuda") for s in frames]
        V, E, gq, gm, gc = _dev_outputs(torch, frames)
        b = q.Batch(hs)
        try:
            for _ in range(2):
                b.run(dm, V, E, gq, gm, gc)
            assert b.captures() == 1
            hs[0].set_tuning(0, [256] * CLASSES)
            hs[0].vpot()
            hs[0].set_tuning(0, *coarse)
            ref = [_plain(h, s, s.dm) for h, s in zip(hs, frames)]
            for replay in (False, True):
                for t in V + E + gq + gm + gc:
                    t.zero_()
                b.run(dm, V, E, gq, gm, gc)
                for i in range(2):
                    for got, key in ((V, "V"), (E, "E"), (gq, "gq"), (gm, "gm"), (gc, "gc")):
                        # same kernels; only the order of atomic additions differs
                        assert _close(got[i].cpu(), ref[i][key], 1e-12), (replay, i, key)
                assert b.captures() == 2
        finally:
            b.close()
    finally:
        for h in hs:
            h.close()
