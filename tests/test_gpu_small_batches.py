"""fp32 / bf16 assignment of few points, whose centroid tiles several CTAs share:
the same assignments and distances as without the shared buffer (a workspace
that ends before it), equal to the oracle's nearest centroid, through ties, rows
left to the fp32 scan and bounds kept between calls; and the cold centroid
preparation's fp64 path for centroids of extreme sizes."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    return skm


def _parts(n, k):
    nct, nrt = -(-k // 256), -(-n // 128)
    most = min(nct, 152 // nrt)
    return 1 if most < 2 else -(-nct // -(-nct // most))


@pytest.mark.parametrize("n,d,k", [(1, 64, 257), (129, 33, 512), (2000, 768, 1000), (6400, 100, 1100), (9728, 16, 600),
                                   (9729, 16, 600), (300, 1536, 5000)])
@pytest.mark.parametrize("kind", ["f32", "bf16"])
@pytest.mark.parametrize("close", [False, True])
def test_split_screen(skm, kind, n, d, k, close):
    X = synth.gmm_points(max(n, k), d, 30, seed=n + d, decay=True)
    g = torch.Generator().manual_seed(k)
    C = X[torch.randperm(max(n, k), generator=g)[:k]].clone()
    if close:  # near-copies and exact copies far apart in index: many rows undecided, ties
        C[k // 2:] = C[: k - k // 2] * (1.0 + 1e-6 * torch.randn(k - k // 2, d, generator=g))
        C[k - 1] = C[0]
    X = X[:n].contiguous()
    if kind == "bf16":
        Xb = X.to(torch.bfloat16)
        p = skm.Points(skm.REPR_BF16, Xb.view(torch.int16).to(DEV), d)
        X = Xb.float()
    else:
        p = skm.Points(skm.REPR_F32, X.to(DEV), d)
    Cd = C.to(DEV)
    S = _parts(n, k)
    full = skm.skm_workspace_size(skm.OP_ASSIGN, p, k)
    a, dist = skm.skm_assign(p, Cd, ws=torch.zeros(full, dtype=torch.uint8, device=DEV))
    less = full - (n * S * 40 if S > 1 else 0)
    a1, dist1 = skm.skm_assign(p, Cd, ws=torch.zeros(less, dtype=torch.uint8, device=DEV))
    assert torch.equal(a, a1) and torch.equal(dist, dist1)
    ao, best, second = oracle.assign_f32(X.numpy(), C.numpy())
    a = a.cpu().numpy()
    off = a != ao
    assert np.all((second - best)[off] <= 1e-5 * np.maximum(best[off], 1e-30))
    np.testing.assert_allclose(dist.cpu().numpy()[~off], best[~off], rtol=2e-5, atol=1e-6)
    # kept bounds: a second call on moved centroids, from the first's state
    pw = p.with_flags(skm.FLAG_WARM)
    ws = skm.workspace(skm.OP_ASSIGN, pw, k)
    skm.skm_assign(pw, Cd, ws=ws)
    C2 = (Cd * 1.001).contiguous()
    aw, dw = skm.skm_assign(pw, C2, ws=ws)
    ac, dc = skm.skm_assign(p, C2)
    assert torch.equal(aw, ac) and torch.equal(dw, dc)


@pytest.mark.parametrize("scale", [2.0 ** -60, 2.0 ** -25, 2.0 ** -19, 1.0, 2.0 ** 45, 2.0 ** 52])
def test_centroids_of_any_size(skm, scale):
    """Squares below 2^-40 or above 2^100 leave the fp32 preparation."""
    n, d, k = 700, 96, 300
    X = synth.gmm_points(n, d, 20, seed=1, decay=False)
    C = X[synth.forgy_indices(n, k, seed=2)] + 0.01
    C[5] = 0.0
    X, C = X * scale, C * scale
    a, dist = skm.skm_assign(skm.Points(skm.REPR_F32, X.to(DEV), d), C.to(DEV))
    ao, best, second = oracle.assign_f32(X.numpy(), C.numpy())
    off = a.cpu().numpy() != ao
    assert np.all((second - best)[off] <= 1e-5 * best[off])
    np.testing.assert_allclose(dist.cpu().numpy()[~off], best[~off], rtol=2e-5)
