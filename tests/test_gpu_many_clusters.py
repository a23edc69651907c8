"""The update's scan of the member counts around its rounds of 4096 clusters, up to
the most clusters there are: counts, centroids and empty clusters, through the
one-block sort and the multi-block one."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    return skm


@pytest.mark.parametrize("k", [1, 4, 1023, 4095, 4096, 4097, 8193, 12288, 12289, 40000, 65536])
@pytest.mark.parametrize("n", [9000, 32769, 90000])
def test_counts_and_centroids(skm, n, k):
    d = 16
    g = torch.Generator().manual_seed(n + k)
    codes = torch.randint(0, 256, (n, d), generator=g)
    a = torch.randint(0, k, (n,), generator=g)
    a[torch.rand(n, generator=g) < 0.1] = k - 1
    a[torch.rand(n, generator=g) < 0.01] = -1
    p = skm.Points(skm.REPR_SQ8, codes.to(torch.uint8).to(DEV), d)
    C0 = torch.randint(0, 256, (k, d), generator=g)
    ok = a >= 0
    S = torch.zeros(k, d, dtype=torch.int64).index_add_(0, a[ok], codes[ok])
    co = torch.bincount(a[ok], minlength=k)
    m = co.clamp_min(1)[:, None]
    q, r = S // m, S % m
    q += ((2 * r > m) | ((2 * r == m) & (q % 2 == 1))).long()  # half to even
    want = torch.where(co[:, None] > 0, q, C0).to(torch.uint8)
    C, counts = skm.skm_update(p, a.to(torch.int32).to(DEV), C0.to(torch.uint8).to(DEV))
    assert torch.equal(counts.cpu(), co)
    assert torch.equal(C.cpu(), want)


@pytest.mark.parametrize("n,k", [(9000, 4097), (9000, 9000), (50000, 4096), (50000, 20000)])
def test_empty_clusters(skm, n, k):
    d = 16
    g = torch.Generator().manual_seed(k)
    p = skm.Points(skm.REPR_SQ8, torch.randint(0, 256, (n, d), generator=g).to(torch.uint8).to(DEV), d)
    C0 = torch.randint(0, 256, (k, d), generator=g).to(torch.uint8).to(DEV)
    a, _ = skm.skm_assign(p, C0)
    want = int((torch.bincount(a.long(), minlength=k) == 0).sum())
    assert want > 0
    stats = skm.skm_fit(p, k, 1, C_init=C0)[4]
    assert stats["empty_per_iter"] == [want]
