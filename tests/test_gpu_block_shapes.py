"""The block sizes that the class sweeps really launch, from a trace of the kernels: those that
qmmm_get_tuning reports, on a system of few warps too, for the default, the 256-thread and the wide
shapes; results in every shape against the oracle."""
import json
import re

import pytest

import oracle
import workloads
from _gpuutil import TOL_FP64, TOL_MIXED, check_V, grad_err

pytestmark = pytest.mark.gpu

KERNELS = {0: "k_vpot_f64", 1: "k_vpot_f32", 2: "k_vgrad_f64"}  # sweep kind -> kernel
KINDS = {0: (0, 2), 1: (1,)}  # precision -> kinds (the mixed adjoint's charge lanes have one block size)


@pytest.fixture(scope="module")
def small():
    # every angular class, some 40 tiles of 32 pairs and 39 charges: far below four warps per SM
    s = workloads.small_system(seed=111, n_atoms=4, lmax=3, nprim=(1, 4), n_waters=14)
    ref = oracle.energy(s)
    ref.update(oracle.forces(s))
    return s, ref


def _traced(call, path):
    """The call's result and {(kernel, class): block sizes} of the sweep kernels that it launched."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(2):  # the first trace of a process can be empty: the tracer starts up in it
        torch.zeros(1, device="cuda")
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            out = call()
            torch.cuda.synchronize()
    prof.export_chrome_trace(str(path))
    sizes = {}
    for e in json.loads(path.read_text())["traceEvents"]:
        m = re.search(r"(k_v(?:pot|grad)_f\d\d)<(\d), (\d), \d+>", e.get("name", ""))
        if m and e.get("cat") == "kernel":
            la, lb = int(m.group(2)), int(m.group(3))
            sizes.setdefault((m.group(1), la * (la + 1) // 2 + lb), set()).add(e["args"]["block"][0])
    return out, sizes


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", ["default", "256", "wide"])
def test_launched_block_sizes(small, precision, shape, tmp_path):
    pytest.importorskip("torch")
    import paper_2408_03273_gb300 as q
    s, ref = small
    h = q.Handle(s, precision=precision, screen_tol=0.0)
    try:
        for k in KINDS[precision]:
            wide = h.tuning(k)["wide"]
            if shape != "default":
                h.set_tuning(k, [w if shape == "wide" and w else 256 for w in wide])
        (V, g), sizes = _traced(lambda: (h.vpot()[0], h.forces(s.dm)), tmp_path / "trace.json")
        if not sizes:
            pytest.skip("no kernel trace (another tool holds the tracer)")
        for k in KINDS[precision]:
            t = h.tuning(k)["threads"]
            for c, n in enumerate(h.info["n_prim_pairs_class"]):
                assert n == 0 or sizes[KERNELS[k], c] == {t[c]}, (k, c)
            assert shape != "wide" or any(x > 256 for x in t)
    finally:
        h.close()
    tol = TOL_FP64 if precision == 0 else TOL_MIXED
    check_V(V, ref["V"], precision)
    for got, key in zip(g, ("dE_dRqm", "dE_dRmm", "dE_dq")):
        assert grad_err(got, ref, key, precision == 1) < tol, key
