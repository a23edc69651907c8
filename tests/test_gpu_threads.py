"""Calls of different sizes from several host threads at once, each on its own
stream and workspace: kernels whose dynamic shared memory depends on the size
launch all the same, and every call gives what it gives alone."""
import ctypes
import threading

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    return skm


def _update(skm, kind, n, d, k, stream):
    """A library call (no Python work inside), its outputs, what it keeps alive."""
    if kind == "sq8":  # one-block sort: 4 (k + n) bytes
        p = skm.Points(skm.REPR_SQ8, torch.randint(0, 256, (n, d), dtype=torch.uint8, device=DEV), d)
    else:              # ring of rows: by d
        p = skm.Points(skm.REPR_F32, torch.randint(-9, 9, (n, d), device=DEV).float(), d)
    C = p.x[:k].clone()
    a = torch.arange(n, dtype=torch.int32, device=DEV) % k
    counts = torch.zeros(k, dtype=torch.int64, device=DEV)
    ws = torch.zeros(skm.skm_workspace_size(skm.OP_UPDATE, p, k), dtype=torch.uint8, device=DEV)
    args = (ctypes.byref(p.ref), skm._ptr(a), k, skm._ptr(C), skm._ptr(counts), None, skm._ptr(ws), ws.numel(),
            skm._stream(stream))
    return lambda: skm.lib().skm_update(*args), [C, counts], (p, a, ws)


def _assign(skm, kind, n, d, k, stream):  # centroid preparation: rows of d in shared memory
    X = synth.gmm_points(n, d, 8, seed=d).to(DEV)
    p = skm.rbq1_points(skm.skm_quantize(skm.REPR_RBQ1, X), d)
    C = X[:k].clone()
    a = torch.empty(n, dtype=torch.int32, device=DEV)
    dist = torch.empty(n, device=DEV)
    ws = torch.zeros(skm.skm_workspace_size(skm.OP_ASSIGN, p, k), dtype=torch.uint8, device=DEV)
    args = (ctypes.byref(p.ref), skm._ptr(C), k, None, skm._ptr(a), skm._ptr(dist), skm._ptr(ws), ws.numel(),
            skm._stream(stream))
    return lambda: skm.lib().skm_assign(*args), [a, dist], (p, C, ws)


@pytest.mark.parametrize("make,kind,sizes", [(_update, "sq8", [(20000, 16, 100), (13000, 16, 100)]),
                                             (_update, "f32", [(500, 72, 20), (500, 116, 20)]),
                                             (_assign, "rbq1", [(200, 2900, 10), (200, 4096, 10)])])
def test_sizes_side_by_side(skm, make, kind, sizes):
    torch.manual_seed(3)
    streams = [torch.cuda.Stream() for _ in range(4)]
    jobs = [make(skm, kind, *sizes[i % 2], s) for i, s in enumerate(streams)]
    torch.cuda.synchronize()
    wants = []
    for call, out, _ in jobs:
        assert call() == 0
        torch.cuda.synchronize()
        wants.append([t.clone() for t in out])
    failed = []

    def work(call):
        for _ in range(2000):
            rc = call()
            if rc != 0:
                failed.append((rc, skm.lib().skm_last_error()))
                return

    threads = [threading.Thread(target=work, args=(call,)) for call, _, _ in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for (_, out, _), want in zip(jobs, wants):
        assert all(torch.equal(x, y) for x, y in zip(out, want))
