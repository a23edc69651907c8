"""Segmented assignment of 1-bit codes that are read packed (rows of whole 16-byte
groups), per group against the oracle bit for bit, and from the expanded copy."""
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


# groups below and above 96 centroids on average (128- and 256-column jobs), and
# one whose tiles fill more than the grid's first round
@pytest.mark.parametrize("sizes,ks", [([1, 127, 129, 300, 5, 1000, 64, 257, 2, 700], [1, 3, 200, 2, 40, 300, 7, 1, 2, 90]),
                                      ([700, 3, 1290], [257, 300, 31]),
                                      ([30000, 100, 50000, 33], [60, 33, 64, 100])])
@pytest.mark.parametrize("d", [100, 128, 384])
def test_rbq1_packed(skm, d, sizes, ks):
    group = np.repeat(np.arange(len(sizes)), sizes).astype(np.int32)
    base = np.concatenate([[0], np.cumsum(ks)]).astype(np.int32)
    n, k = group.size, int(base[-1])
    X = synth.gmm_points(n, d, 30, seed=n + d)
    C = synth.gmm_points(k, d, 30, seed=d)
    r = skm.skm_quantize(skm.REPR_RBQ1, X.to(DEV))
    p = skm.rbq1_points(r, d)
    g, b = torch.from_numpy(group).to(DEV), torch.from_numpy(base).to(DEV)
    a, est = skm.skm_assign_segmented(p, C.to(DEV), g, b)
    a2, est2 = skm.skm_assign_segmented(p.with_screen(), C.to(DEV), g, b)
    assert torch.equal(a, a2) and torch.equal(est, est2)
    h = {f: r[f].cpu().numpy() for f in ("codes", "nx2", "F", "popx", "m")}
    h["codes"] = h["codes"].view(np.uint32)
    rng = np.random.default_rng(n)
    for s in range(len(sizes)):
        rows = np.nonzero(group == s)[0]
        rows = rows if rows.size <= 2000 else np.sort(rng.choice(rows, 2000, replace=False))
        prep = oracle.rbq1_centroid_sq4(C.numpy()[base[s]:base[s + 1]], h["m"])
        ao, eo = oracle.rbq1_assign(h["codes"][rows], h["nx2"][rows], h["F"][rows], h["popx"][rows], d, prep)
        np.testing.assert_array_equal(a.cpu().numpy()[rows] - base[s], ao)
        np.testing.assert_array_equal(est.cpu().numpy()[rows], eo)
