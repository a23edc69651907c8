"""Distances of fp32 and bf16 rows of every length around the batches in which a
warp reads them, on small integers, where every order of the sum is exact."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    return skm


@pytest.mark.parametrize("d", [1, 2, 31, 32, 33, 100, 127, 128, 129, 160, 255, 256, 257, 383, 384, 385, 511, 512, 513,
                               640, 1025])
@pytest.mark.parametrize("kind", ["f32", "bf16"])
def test_exact_distances(skm, kind, d):
    n, k = 700, 37
    g = torch.Generator().manual_seed(d)
    x = torch.randint(-8, 9, (n, d), generator=g).double().to(DEV)
    c = torch.randint(-8, 9, (k, d), generator=g).double().to(DEV)
    x[:50] = c[torch.randint(0, k, (50,), generator=g).to(DEV)]  # some at distance zero
    full = (x * x).sum(1)[:, None] + (c * c).sum(1)[None, :] - 2.0 * x @ c.T  # whole numbers below 2^24
    if kind == "f32":
        p = skm.Points(skm.REPR_F32, x.float(), d)
    else:
        p = skm.Points(skm.REPR_BF16, x.to(torch.bfloat16).view(torch.int16), d)
    a, dist = skm.skm_assign(p, c.float())
    assert torch.equal(dist.double(), full.min(1).values)
    assert torch.equal(full.gather(1, a.long()[:, None])[:, 0], full.min(1).values)
