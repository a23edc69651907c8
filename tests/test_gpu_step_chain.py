"""Steps queued back to back, whose kernels are placed on the chip before their
predecessors end: the same centroids, counts and assignments, bit for bit, as
with the device idle before every call and as replayed from a CUDA graph.  The
float points are small integers, so their sums are exact in any order."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    return skm


# small grids all along; the multi-block sort; grids around two blocks an SM and above
@pytest.mark.parametrize("n,d,k", [(300, 64, 7), (2500, 96, 300), (20000, 128, 100), (38900, 64, 304), (39100, 64, 2500),
                                   (120000, 256, 350)])
@pytest.mark.parametrize("kind", ["f32", "bf16", "sq8", "rbq1", "lvq4"])
def test_queued_steps_equal_separate_ones(skm, kind, n, d, k):
    g = torch.Generator().manual_seed(n + d)
    X = torch.randint(-8, 9, (n, d), generator=g).float()
    X += 4 * torch.randint(-8, 9, (40, d), generator=g).float()[torch.randint(0, 40, (n,), generator=g)]
    Xd = X.to(DEV)
    if kind == "f32":
        p = skm.Points(skm.REPR_F32, Xd, d)
    elif kind == "bf16":
        p = skm.Points(skm.REPR_BF16, Xd.to(torch.bfloat16).view(torch.int16), d)
    elif kind == "sq8":
        p = skm.Points(skm.REPR_SQ8, skm.skm_quantize(skm.REPR_SQ8, Xd)["codes"], d)
    elif kind == "rbq1":
        p = skm.rbq1_points(skm.skm_quantize(skm.REPR_RBQ1, Xd), d)
    else:
        p = skm.lvq4_points(skm.skm_quantize(skm.REPR_LVQ4, Xd), d)
    pick = torch.randperm(n, generator=g)[:k].to(DEV)
    C0 = p.x[pick].clone() if kind == "sq8" else Xd[pick].clone()
    ws = torch.zeros(skm.skm_workspace_size(skm.OP_ASSIGN, p, k), dtype=torch.uint8, device=DEV)
    ws_up = torch.zeros(skm.skm_workspace_size(skm.OP_UPDATE, p, k), dtype=torch.uint8, device=DEV)
    C = C0.clone()
    assign = torch.empty(n, dtype=torch.int32, device=DEV)
    dist = torch.empty(n, dtype=torch.float32, device=DEV)
    counts = torch.zeros(k, dtype=torch.int64, device=DEV)

    def steps(apart):
        for _ in range(4):
            if apart:
                torch.cuda.synchronize()
            skm.skm_assign(p, C, ws=ws, out=assign, dist_out=dist)
            if apart:
                torch.cuda.synchronize()
            skm.skm_update(p, assign, C, counts=counts.zero_(), ws=ws_up)

    def result():
        torch.cuda.synchronize()
        return [t.clone() for t in (C, assign, dist, counts)]

    steps(True)
    want = result()
    for _ in range(3):
        C.copy_(C0)
        steps(False)
        assert all(torch.equal(x, y) for x, y in zip(result(), want))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        steps(False)
    for _ in range(2):
        C.copy_(C0)
        graph.replay()
        assert all(torch.equal(x, y) for x, y in zip(result(), want))
