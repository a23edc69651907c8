"""Hierarchical fits at and just below the documented limit of 12288 groups,
against the oracle: the order by group keeps a counter a group in one block's
shared memory, next to the block's own words."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    return skm


@pytest.mark.parametrize("m", [12256, 12257, 12288])
def test_most_groups(skm, m):
    n, d, k = 12400, 32, 12300
    q = skm.skm_quantize(skm.REPR_SQ8, synth.gmm_points(n, d, 2000, seed=m, decay=False).to(DEV))
    idx = synth.forgy_indices(n, m, seed=m)
    C, a, meso, kf, _ = skm.skm_fit_hierarchical(skm.Points(skm.REPR_SQ8, q["codes"], d), k, m, idx.to(DEV), 1, 1)
    Co, ao, amo, kfo = oracle.hierarchical("sq8", q["codes"].cpu().numpy(), k, m, idx.numpy(), 1, 1)
    assert kf == kfo
    np.testing.assert_array_equal(meso.cpu().numpy(), amo)
    np.testing.assert_array_equal(a.cpu().numpy(), ao)
    np.testing.assert_array_equal(C.cpu().numpy(), Co)
