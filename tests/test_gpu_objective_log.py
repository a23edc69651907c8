"""A fit that fails midway has written the objective of every iteration that it
finished (they are kept on the device and copied several at a time)."""
import ctypes
import threading
import time

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"
LAUNCH = 2


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    yield skm
    skm.skm_inject_fault(LAUNCH, 0)


def test_objective_of_finished_iterations(skm):
    n, d, k = 3000, 32, 20
    X = synth.gmm_points(n, d, 20, seed=5).to(DEV)
    p = skm.Points(skm.REPR_SQ8, skm.skm_quantize(skm.REPR_SQ8, X)["codes"], d)
    idx = synth.forgy_indices(n, k, seed=5).to(DEV)
    ws = skm.workspace(skm.OP_FIT, p, k)
    C = torch.empty(k, d, dtype=torch.uint8, device=DEV)
    a = torch.empty(n, dtype=torch.int32, device=DEV)

    def fit(iters):  # status, objective, kernels launched
        obj = np.full(iters + 1, np.nan)
        st = skm.Stats()
        cfg = skm.FitConfig(k, iters, 0, 0, 0)
        before = skm.skm_kernel_launches()
        rc = skm.lib().skm_fit(ctypes.byref(cfg), ctypes.byref(p.ref), None, skm._ptr(idx), skm._ptr(C), skm._ptr(a),
                               None, obj.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), ctypes.byref(st),
                               skm._ptr(ws), ws.numel(), None)
        launches = skm.skm_kernel_launches() - before
        torch.cuda.synchronize()
        return rc, obj, launches

    # launches of a fit of no iteration, of one more iteration, and of the
    # statistics behind the last one
    rc, want, _ = fit(200)
    assert rc == 0 and np.isfinite(want).all()
    l0, l1, l2 = fit(0)[2], fit(1)[2], fit(2)[2]
    per = l2 - l1
    tail = 1  # the histogram of the final assignment
    first = l0 - tail
    assert l1 - l0 == per
    checked = 0
    for attempt in range(12):
        got = {}
        t = threading.Thread(target=lambda: got.update(zip(("rc", "obj", "launches"), fit(50000))))
        before = skm.skm_kernel_launches()
        t.start()
        while t.is_alive() and skm.skm_kernel_launches() - before < first + 40 * per + 37 * attempt:
            time.sleep(0.0002)
        skm.skm_inject_fault(LAUNCH, 1)
        t.join()
        assert got["rc"] == 3
        # the failed launch is the last; objectives whose sum came before it
        done = (got["launches"] - 1 - first) // per + 1
        written = int(np.isfinite(got["obj"]).sum())
        assert 0 < done < 50001
        assert np.isfinite(got["obj"][:done]).all(), (done, written)
        m = min(done, want.size)
        np.testing.assert_array_equal(got["obj"][:m], want[:m])
        checked += done % 32 != 0
    assert checked
