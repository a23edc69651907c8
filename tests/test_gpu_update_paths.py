"""The update's size rules against the oracle: the one-block sort and the
multi-block one on both sides of its limits, short and long runs, 1-bit and
LVQ4 rows whose words are no multiple of a vector load or span several blocks,
assignments outside [0, k), empty clusters, and the objective sum's two forms."""
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


def _assign(n, k, seed):
    g = torch.Generator().manual_seed(seed)
    a = torch.randint(0, max(1, k - 1), (n,), generator=g, dtype=torch.int32)  # cluster k - 1 empty
    a[torch.rand(n, generator=g) < 0.3] = 0                                     # one large cluster
    bad = torch.rand(n, generator=g) < 0.01
    a[bad] = torch.where(torch.rand(int(bad.sum()), generator=g) < 0.5, -1, k).to(torch.int32)
    return a


SIZES = [(1, 33, 1), (31, 64, 3), (700, 96, 13), (32768, 32, 50), (32769, 32, 50), (33000, 100, 12288),
         (33000, 64, 12289), (5000, 1100, 40), (3000, 1536, 9), (900, 4096, 5), (60001, 200, 300), (2000, 300, 700)]


@pytest.mark.parametrize("n,d,k", SIZES)
@pytest.mark.parametrize("kind", ["f32", "bf16", "sq8", "rbq1", "lvq4"])
def test_update_sizes_vs_oracle(skm, kind, n, d, k):
    X = synth.gmm_points(n, d, 20, seed=n + d, decay=False)
    a = _assign(n, k, n + k)
    ok = ((a >= 0) & (a < k)).numpy()
    ao = a.numpy()[ok]
    C0 = torch.randn(k, d, generator=torch.Generator().manual_seed(3))
    if kind == "sq8":
        q = skm.skm_quantize(skm.REPR_SQ8, X.to(DEV))
        C0 = torch.randint(0, 256, (k, d), generator=torch.Generator().manual_seed(3)).to(torch.uint8)
        C, counts = skm.skm_update(skm.Points(skm.REPR_SQ8, q["codes"], d), a.to(DEV), C0.to(DEV))
        Co, co = oracle.update_sq8(q["codes"].cpu().numpy()[ok], ao, C0.numpy())
    elif kind == "rbq1":
        q = skm.skm_quantize(skm.REPR_RBQ1, X.to(DEV))
        p = skm.rbq1_points(q, d)
        C, counts = skm.skm_update(p, a.to(DEV), C0.to(DEV))
        Co, co = oracle.rbq1_update(q["codes"].cpu().numpy().view(np.uint32)[ok], q["F"].cpu().numpy()[ok], d,
                                    q["m"].cpu().numpy(), p.rbq1_exp, ao, C0.numpy())
    elif kind == "lvq4":
        q = skm.skm_quantize(skm.REPR_LVQ4, X.to(DEV))
        p = skm.lvq4_points(q, d)
        C, counts = skm.skm_update(p, a.to(DEV), C0.to(DEV))
        Co, co = oracle.lvq4_update(oracle.lvq4_unpack(q["codes"].cpu().numpy(), d)[ok], q["lvq"].cpu().numpy()[ok],
                                    p.rbq1_exp, ao, C0.numpy())
    else:
        if kind == "bf16":
            Xb = X.to(torch.bfloat16)
            p = skm.Points(skm.REPR_BF16, Xb.view(torch.int16).to(DEV), d)
            xs = Xb.float().numpy().astype(np.float64)
        else:
            p = skm.Points(skm.REPR_F32, X.to(DEV), d)
            xs = X.numpy().astype(np.float64)
        C, counts = skm.skm_update(p, a.to(DEV), C0.to(DEV))
        co = np.bincount(ao, minlength=k)
        S, A = np.zeros((k, d)), np.zeros((k, d))
        np.add.at(S, ao, xs[ok])
        np.add.at(A, ao, np.abs(xs[ok]))
        np.testing.assert_array_equal(counts.cpu().numpy(), co)
        Cg = C.cpu().numpy()
        np.testing.assert_array_equal(Cg[co == 0], C0.numpy()[co == 0])
        m = np.maximum(co, 1)[:, None]
        # any order of c fp32 additions: (c - 1) 2^-24 of the absolute sum, and the division's rounding
        bound = 2.0 ** -24 * ((m + 1) * A / m + np.abs(S) / m)
        assert np.all(np.abs(Cg - S / m)[co > 0] <= bound[co > 0])
        return
    np.testing.assert_array_equal(counts.cpu().numpy(), co)
    np.testing.assert_array_equal(C.cpu().numpy(), Co)


@pytest.mark.parametrize("n", [1, 1023, 65536, 65537, 200_001])
def test_fit_objective_sum(skm, n):
    """iters = 0: one assignment, whose objective is the fp64 sum of its fp32
    distances (an order's rounding is below n 2^-53 of it)."""
    d, k = 8, 1
    X = synth.gmm_points(n, d, 4, seed=n, decay=False).to(DEV)
    _, _, dist, obj, _ = skm.skm_fit(skm.Points(skm.REPR_F32, X, d), k, 0,
                                     init_idx=torch.zeros(1, dtype=torch.int64, device=DEV))
    want = float(dist.double().sum())
    assert abs(obj[0] - want) <= max(n, 2) * 2.0 ** -52 * want


@pytest.mark.parametrize("d", [64, 100, 101, 300, 512, 516, 515])
@pytest.mark.parametrize("offset", [0, 4, 1])
def test_bf16_sums_by_alignment(skm, d, offset):
    """Rows that start on 16, 8 and 2 bytes; integer points, so that the sums are exact."""
    n, k = 5003, 37
    g = torch.Generator().manual_seed(d + offset)
    X = torch.randint(-100, 101, (n, d), generator=g).float()
    a = _assign(n, k, d)
    ok = (a >= 0) & (a < k)
    buf = torch.zeros(n * d + 8, dtype=torch.int16, device=DEV)
    x = buf[offset : offset + n * d].view(n, d)
    x.copy_(X.to(torch.bfloat16).view(torch.int16))
    C0 = torch.randn(k, d, generator=g)
    C, counts = skm.skm_update(skm.Points(skm.REPR_BF16, x, d), a.to(DEV), C0.to(DEV))
    S = torch.zeros(k, d).index_add_(0, a[ok].long(), X[ok])
    co = torch.bincount(a[ok].long(), minlength=k)
    want = torch.where(co[:, None] > 0, S / co.clamp_min(1)[:, None].float(), C0)
    assert torch.equal(counts.cpu(), co) and torch.equal(C.cpu(), want)
