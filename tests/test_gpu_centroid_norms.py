"""The screen's record of a centroid, ||c||^2 rounded to fp32, is the rounding of
a sum held to 53 bits or more, with and without kept bounds: here the last of
three squares, 2^-52 of the first, decides a tie."""
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


@pytest.mark.parametrize("flags", ["cold", "warm"])
@pytest.mark.parametrize("order", [[0, 1, 2, 3], [1, 2, 0, 3], [2, 3, 1, 0]])
@pytest.mark.parametrize("stride", [1, 8, 32, 40])  # squares in neighbouring lanes, in one lane, in both
def test_tie_decided_by_the_last_bits(skm, flags, order, stride):
    d = 128
    c = torch.zeros(2, d)
    for place, i in enumerate(order):
        c[0, place * stride % d + (place * stride >= d)] = [1.0, 2.0**-12, 2.0**-26, 0.0][i]
    c[1, :4] = torch.tensor([2.0, 1.0, 1.0, 1.0])
    p = skm.Points(skm.REPR_F32, torch.randn(300, d, generator=torch.Generator().manual_seed(1)).to(DEV), d)
    if flags == "warm":
        p = p.with_flags(skm.FLAG_WARM)
    ws = torch.zeros(skm.skm_workspace_size(skm.OP_ASSIGN, p, 2), dtype=torch.uint8, device=DEV)
    skm.skm_assign(p, c.to(DEV), ws=ws)
    w = ws[: ws.numel() // 16 * 16].cpu().numpy().view(np.float32).reshape(-1, 4)
    rec = w[(w[:, 1] == 7.0) & (np.abs(w[:, 0] - 1.0) < 1e-6)]
    assert rec.shape[0] == 1
    assert rec[0, 0] == np.float32(1.0 + 2.0**-23)
