"""Updates of few clusters, whose runs are longer than the number of rows alone
would make them, against the oracle (codes) and exact sums (float rows of small
integers), finalised and as partial sums."""
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


# runs of 16 to 128 by n and k; rows below and above a lane's group and 1 KB of codes
@pytest.mark.parametrize("n,k", [(700, 1), (3001, 2), (20011, 1), (20011, 3), (40000, 1), (40000, 9), (90001, 2)])
@pytest.mark.parametrize("d", [33, 64, 300, 1040])
@pytest.mark.parametrize("kind", ["f32", "bf16", "sq8", "rbq1", "lvq4"])
def test_few_clusters(skm, kind, d, n, k):
    g = torch.Generator().manual_seed(n + d + k)
    a = torch.randint(0, k, (n,), generator=g, dtype=torch.int32)
    a[torch.rand(n, generator=g) < 0.02] = -1
    ok = (a >= 0).numpy()
    ao = a.numpy()[ok]
    co = np.bincount(ao, minlength=k)
    ints = torch.randint(-100, 101, (n, d), generator=g)
    if kind in ("f32", "bf16"):
        x = ints.float()
        p = skm.Points(skm.REPR_F32, x.to(DEV), d)
        if kind == "bf16":
            p = skm.Points(skm.REPR_BF16, x.to(torch.bfloat16).view(torch.int16).to(DEV), d)
        S = torch.zeros(k, d, dtype=torch.int64).index_add_(0, torch.from_numpy(ao).long(), ints[torch.from_numpy(ok)])
        want = (S.float() / torch.from_numpy(co)[:, None].float()).numpy()  # below 2^24: exact sums
        part, dt = S.double(), torch.float64
    elif kind == "sq8":
        codes = (ints + 100).to(torch.uint8)
        p = skm.Points(skm.REPR_SQ8, codes.to(DEV), d)
        want, _ = oracle.update_sq8(codes.numpy()[ok], ao, np.zeros((k, d), np.uint8))
        part = torch.zeros(k, d, dtype=torch.int64).index_add_(0, torch.from_numpy(ao).long(),
                                                               codes[torch.from_numpy(ok)].long())
        dt = torch.int64
    else:
        X = synth.gmm_points(n, d, 5, seed=d).to(DEV)
        q = skm.skm_quantize(skm.REPR_RBQ1 if kind == "rbq1" else skm.REPR_LVQ4, X)
        C0 = np.zeros((k, d), np.float32)
        part, dt = None, torch.int64
        if kind == "rbq1":
            p = skm.rbq1_points(q, d)
            want, _ = oracle.rbq1_update(q["codes"].cpu().numpy().view(np.uint32)[ok], q["F"].cpu().numpy()[ok], d,
                                         q["m"].cpu().numpy(), p.rbq1_exp, ao, C0)
        else:
            p = skm.lvq4_points(q, d)
            want, _ = oracle.lvq4_update(oracle.lvq4_unpack(q["codes"].cpu().numpy(), d)[ok],
                                         q["lvq"].cpu().numpy()[ok], p.rbq1_exp, ao, C0)
    C = torch.zeros(k, d, dtype=torch.uint8 if kind == "sq8" else torch.float32, device=DEV)
    C1, counts = skm.skm_update(p, a.to(DEV), C)
    np.testing.assert_array_equal(counts.cpu().numpy(), co)
    np.testing.assert_array_equal(C1.cpu().numpy(), want)
    P = torch.zeros(k, d + (kind in ("rbq1", "lvq4")), dtype=dt, device=DEV)
    counts = torch.zeros(k, dtype=torch.int64, device=DEV)
    skm.skm_update(p, a.to(DEV), C, counts=counts, partial=P)
    if part is not None:
        assert torch.equal(P.cpu(), part)
    C2 = torch.zeros_like(C1)
    skm.skm_update_finalize(p, P, counts, C2)
    assert torch.equal(C2, C1)
