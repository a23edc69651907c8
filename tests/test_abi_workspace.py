"""Workspace sizes hold what the call can use (host only: sizes are formed without
a device)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def skm():
    from paper_2608_14648_gb300 import build as b

    b.build()
    import paper_2608_14648_gb300 as skm

    return skm


@pytest.mark.parametrize("d", [1536, 4096])
@pytest.mark.parametrize("op", [0, 2])
@pytest.mark.parametrize("kind", ["rbq1", "lvq4"])
def test_codes_that_cannot_be_read_packed_get_no_expansion_slots(skm, kind, op, d):
    def size(addr):
        x = skm.Data(skm.REPR_RBQ1 if kind == "rbq1" else skm.REPR_LVQ4, d, 20000, addr, 0x100, 0x100, 0x100, 0x100,
                     0, 0)
        x.lvq = 0x100
        return skm.lib().skm_workspace_size(op, ctypes.byref(x), 100)

    assert size(0x1000) > size(0x1004)  # 16-byte aligned codes: with the tensor-core buffers
    assert size(None) == size(0x1000)   # no address yet: as for aligned ones


def test_projection_holds_the_parts_of_p(skm):
    for n, d, dout in [(1000, 64, 32), (100000, 1024, 256), (5, 7, 3)]:
        x = skm.Data(skm.REPR_F32, d, n, 0x1000, None, None, None, None, 0, 0)
        dp = (d + 7) // 8 * 8
        want = 256 + 3 * dout * dp * 2  # the flag, then three bf16 parts
        for op in (6, 7):
            got = skm.lib().skm_workspace_size(op, ctypes.byref(x), dout)
            assert want <= got < want + 512
