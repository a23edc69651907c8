"""The RabitQ mean (exact fixed point) against the oracle, bit for bit, on both
sides of the one-pass rule's limits and where the sampled rows' maximum names
the wrong scale: one power of two too small, more than one, or none at all."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    return skm


def _mean(skm, X):
    return skm.skm_quantize(skm.REPR_RBQ1, X)["m"].cpu().numpy()


@pytest.mark.parametrize("n,d", [(65536, 64), (65537, 4), (65537, 64), (70001, 10), (131072, 100), (131073, 96),
                                 (70000, 768), (66000, 2052), (300_001, 8), (257, 768), (1, 4), (2049, 33)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -60, 3e-37, 1e30])
def test_mean_matches_the_oracle(skm, n, d, scale):
    g = torch.Generator().manual_seed(n + d)
    X = ((torch.randn(n, d, generator=g) + 0.1) * scale).float()
    X[torch.rand(n, generator=g) < 0.2] *= 2.0 ** -30  # values far below the largest
    np.testing.assert_array_equal(_mean(skm, X.to(DEV)), oracle.rbq1_mean(X.numpy()))


@pytest.mark.parametrize("factor", [1.0, 2.0, 4.0, 2.0 ** 40, -3.0])
@pytest.mark.parametrize("base", [0.75, 0.0])
def test_mean_with_an_outlier_outside_the_sample(skm, factor, base):
    n, d = 100_000, 64
    X = torch.rand(n, d, generator=torch.Generator().manual_seed(3)) * base
    X[12345, 7] = 0.9 * factor  # row 12345 is not i n / 2048 for any i
    assert all(i * n // 2048 != 12345 for i in range(2048))
    np.testing.assert_array_equal(_mean(skm, X.to(DEV)), oracle.rbq1_mean(X.numpy()))


def test_mean_of_an_unaligned_array(skm):
    n, d = 70_000, 32
    buf = torch.randn(n * d + 1, generator=torch.Generator().manual_seed(4)).to(DEV)
    X = buf[1:].view(n, d)
    np.testing.assert_array_equal(_mean(skm, X), oracle.rbq1_mean(X.cpu().numpy()))
