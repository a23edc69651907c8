"""Entry points that hold an assignment's workspace inside their own take one
without the part that only makes small assignments faster (the shared centroid
tiles' row states), and give the same results with it."""
import ctypes

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


def _r256(b):
    return (b + 255) // 256 * 256


def test_hierarchical_fit(skm):
    n, d, k, m = 2000, 16, 320, 300
    X = synth.gmm_points(n, d, 100, seed=1).mul(8).round().to(DEV)  # small integers: exact sums
    p = skm.Points(skm.REPR_F32, X, d)
    idx = synth.forgy_indices(n, m, seed=1).to(DEV)
    cfg = skm.HierConfig(k, m, 2, 2, 0)
    full = skm.lib().skm_hier_workspace_size(ctypes.byref(cfg), ctypes.byref(p.ref))
    part = _r256(n * 2 * 10 * 4)  # two centroid tiles, ten words a row and share
    want = skm.skm_fit_hierarchical(p, k, m, idx, 2, 2)
    got = skm.skm_fit_hierarchical(p, k, m, idx, 2, 2, ws=torch.zeros(full - part, dtype=torch.uint8, device=DEV))
    assert torch.equal(got[2], want[2]) and got[3] == want[3] and torch.equal(got[1], want[1])
    with pytest.raises(skm.SkmError) as ei:
        skm.skm_fit_hierarchical(p, k, m, idx, 2, 2, ws=torch.zeros(full - part - 256, dtype=torch.uint8, device=DEV))
    assert ei.value.code == 4


@pytest.mark.parametrize("warm", [False, True])
def test_host_step(skm, warm):
    n, d, k, chunks = 4000, 16, 600, 2
    X = torch.randint(-9, 9, (n, d), generator=torch.Generator().manual_seed(2)).float().pin_memory()
    C = X[:k].clone().pin_memory()
    part = _r256(n // chunks * 3 * 10 * 4) * (chunks if warm else 1)  # three centroid tiles
    outs = []
    for less in (0, part):
        step = skm.LloydStepHost(skm.REPR_F32, X, d, k, chunks=chunks, warm=warm)
        step.ws = torch.zeros(step.ws.numel() - less, dtype=torch.uint8, device=DEV)
        Ch = C.clone().pin_memory()
        for _ in range(2):
            _, a, _, _ = step(Ch)
        outs.append((Ch.clone(), a.clone()))
    assert all(torch.equal(x, y) for x, y in zip(*outs))
    step.ws = torch.zeros(step.ws.numel() - 256, dtype=torch.uint8, device=DEV)
    with pytest.raises(skm.SkmError) as ei:
        step(C.clone().pin_memory())
    assert ei.value.code == 4
