"""Tensor-core projection at the edges of its tiles: rows and columns around 128
and 256, column tiles of uneven splits, dimensions around a 64-wide slice and
not a multiple of a vector load, points at an unaligned address, no mean.
Tolerance: the fp32-accuracy bound the projection is documented with, 2e-6 of
||x - mean|| for orthonormal columns."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    return skm


@pytest.mark.parametrize("n", [1, 127, 129, 20_000])
@pytest.mark.parametrize("d,dout", [(1, 1), (7, 7), (63, 15), (64, 17), (65, 64), (257, 256), (260, 257), (300, 272),
                                    (1030, 513), (4096, 40), (1536, 1536)])
def test_project_tile_edges(skm, n, d, dout):
    g = torch.Generator(device=DEV).manual_seed(n + d + dout)
    X = torch.randn(n, d, device=DEV, generator=g) + 3.0
    P = torch.linalg.qr(torch.randn(d, d, device=DEV, generator=g, dtype=torch.float64))[0][:, :dout]
    P = P.float().contiguous()
    mu = torch.randn(d, device=DEV, generator=g) + 3.0
    for mean in (mu, None):
        Z = X.double() - (mean.double() if mean is not None else 0.0)
        want = Z @ P.double()
        scale = Z.norm(dim=1, keepdim=True)
        Y = skm.skm_project(X, P, mean)
        assert bool(((Y.double() - want).abs() <= 2e-6 * scale).all())
        Yb = skm.skm_project(X, P, mean, out_dtype=skm.DTYPE_BF16)
        assert torch.equal(Yb, Y.to(torch.bfloat16))
    buf = torch.empty(n * d + 1, device=DEV)
    Xu = buf[1:].view(n, d)
    Xu.copy_(X)
    assert torch.equal(skm.skm_project(Xu, P, mu), skm.skm_project(X, P, mu))


def test_project_large_and_small_values(skm):
    """Rows 2^60 apart in size: each keeps its own accuracy."""
    n, d, dout = 300, 200, 96
    g = torch.Generator(device=DEV).manual_seed(1)
    X = torch.randn(n, d, device=DEV, generator=g) * torch.logspace(-30, 30, n, base=2, device=DEV).unsqueeze(1)
    P = torch.linalg.qr(torch.randn(d, d, device=DEV, generator=g, dtype=torch.float64))[0][:, :dout].float().contiguous()
    Y = skm.skm_project(X, P)
    err = (Y.double() - X.double() @ P.double()).abs() / X.double().norm(dim=1, keepdim=True)
    assert float(err.max()) <= 2e-6
    assert np.isfinite(Y.cpu().numpy()).all()
