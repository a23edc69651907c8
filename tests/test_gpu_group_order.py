"""Hierarchical fits whose fine phase works on rows ordered by group, against the
oracle bit for bit: rows around a block's 4096 and past 128 blocks, groups around
a warp's 32 and a block's 1024; and 1-bit codes whose expanded copy has whole rows
without padding, rows padded to 16 bytes, and rows of a multiple of 16 but not 32."""
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


@pytest.mark.parametrize("n,d,k,m", [(4095, 32, 70, 31), (4096, 32, 80, 33), (4097, 32, 40, 2), (8193, 32, 2300, 1025),
                                     (540001, 32, 300, 65)])
def test_sq8_fit(skm, n, d, k, m):
    q = skm.skm_quantize(skm.REPR_SQ8, synth.gmm_points(n, d, 3 * m, seed=n, decay=False).to(DEV))
    idx = synth.forgy_indices(n, m, seed=m)
    C, a, meso, kf, _ = skm.skm_fit_hierarchical(skm.Points(skm.REPR_SQ8, q["codes"], d), k, m, idx.to(DEV), 2, 2)
    Co, ao, amo, kfo = oracle.hierarchical("sq8", q["codes"].cpu().numpy(), k, m, idx.numpy(), 2, 2)
    assert kf == kfo
    np.testing.assert_array_equal(meso.cpu().numpy(), amo)
    np.testing.assert_array_equal(a.cpu().numpy(), ao)
    np.testing.assert_array_equal(C.cpu().numpy(), Co)


@pytest.mark.parametrize("d", [32, 100, 112, 128, 160])
def test_rbq1_copy(skm, d):
    n, k = 3001, 300
    X = synth.gmm_points(n, d, 40, seed=d, decay=True).to(DEV)
    p = skm.rbq1_points(skm.skm_quantize(skm.REPR_RBQ1, X), d)
    a, dist = skm.skm_assign(p, X[:k].contiguous())
    a2, dist2 = skm.skm_assign(p.with_screen(), X[:k].contiguous())
    assert torch.equal(a, a2) and torch.equal(dist, dist2)
