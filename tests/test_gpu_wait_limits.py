"""What a call leaves behind when a device wait runs out (the injected short wait,
before anything is loaded): nothing is read through an assignment that was never
written, and the next call is as before."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"
WAIT = 4


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    yield skm
    skm.skm_inject_fault(WAIT, 0)


# centroid tiles shared out to several blocks; one tile; several tiles, one block a point tile
@pytest.mark.parametrize("n,k,shared", [(2000, 1000, True), (2000, 200, False), (40000, 300, False)])
@pytest.mark.parametrize("kind", ["f32", "bf16"])
def test_distances_without_assignments(skm, kind, n, k, shared):
    d = 64
    X = synth.gmm_points(n, d, 30, seed=n + k).to(DEV)
    if kind == "bf16":
        p = skm.Points(skm.REPR_BF16, X.to(torch.bfloat16).view(torch.int16), d)
    else:
        p = skm.Points(skm.REPR_F32, X, d)
    C = X[:k].clone()
    ws = skm.workspace(skm.OP_ASSIGN, p, k)
    a0, d0 = skm.skm_assign(p, C, ws=ws)
    out = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    dist = torch.zeros(n, device=DEV)
    skm.skm_inject_fault(WAIT, 1)
    skm.skm_assign(p, C, ws=ws, out=out, dist_out=dist)
    torch.cuda.synchronize()
    assert skm.skm_fault_armed(WAIT) == 0
    assert (out == -1).all() and torch.isinf(dist).all()
    if shared:  # rows of shared tiles are set, whatever the array held
        out.fill_(k - 1)
        skm.skm_inject_fault(WAIT, 1)
        skm.skm_assign(p, C, ws=ws, out=out, dist_out=dist)
        assert (out == -1).all() and torch.isinf(dist).all()
    a1, d1 = skm.skm_assign(p, C, ws=ws)
    assert torch.equal(a1, a0) and torch.equal(d1, d0)


# packed codes with three point tiles or more a job stream, so that the converter
# warps come to wait for an expansion slot that is never freed
@pytest.mark.parametrize("k", [30, 300])
@pytest.mark.parametrize("kind", ["rbq1", "lvq4"])
def test_packed_codes(skm, kind, k):
    n, d = 152 * 128 * 7, 128
    X = synth.gmm_points(n, d, 30, seed=k).to(DEV)
    if kind == "rbq1":
        p = skm.rbq1_points(skm.skm_quantize(skm.REPR_RBQ1, X), d)
    else:
        p = skm.lvq4_points(skm.skm_quantize(skm.REPR_LVQ4, X), d)
    idx = synth.forgy_indices(n, k, seed=1).to(DEV)

    def fit():
        return skm.skm_fit(p, k, 1, init_idx=idx, want_objective=False, want_dist=False)[:2]

    C0, a0 = fit()
    skm.skm_inject_fault(WAIT, 1)
    with pytest.raises(skm.SkmError) as ei:
        fit()
    assert ei.value.code == 5 and skm.skm_fault_armed(WAIT) == 0
    C1, a1 = fit()
    assert torch.equal(C1, C0) and torch.equal(a1, a0)


# one tile; several row and column tiles a block; more tiles than blocks
@pytest.mark.parametrize("n,d,dout", [(100, 64, 16), (3000, 600, 300), (152 * 128 * 2 + 5, 128, 48)])
@pytest.mark.parametrize("bf16", [False, True])
def test_projection(skm, bf16, n, d, dout):
    g = torch.Generator().manual_seed(d)
    X, P = torch.randn(n, d, generator=g).to(DEV), torch.randn(d, dout, generator=g).to(DEV)
    dt = skm.DTYPE_BF16 if bf16 else skm.DTYPE_F32

    def project():
        Y = skm.skm_project(X, P, out_dtype=dt)
        return Y.view(torch.bfloat16) if bf16 else Y

    want = project()
    assert torch.isfinite(want).all()
    skm.skm_inject_fault(WAIT, 1)
    assert torch.isnan(project()).all()
    assert skm.skm_fault_armed(WAIT) == 0
    assert torch.equal(project(), want)
