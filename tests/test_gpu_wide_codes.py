"""1-bit and LVQ4 assignment of rows longer than 1024 dimensions, bit for bit
against the oracle: on the tensor cores (rows of whole 16-byte groups at an
aligned address), with code sums near their largest, and on CUDA cores where
the tensor-core path does not apply (other row sizes, an unaligned address, a
workspace that ends before its buffers)."""
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


def _case(skm, kind, X, C, sym=False):
    """(points, the oracle's assignment and distances)"""
    d = X.shape[1]
    if kind == "lvq4":
        q = skm.skm_quantize(skm.REPR_LVQ4, X.to(DEV))
        codes = oracle.lvq4_unpack(q["codes"].cpu().numpy(), d)
        return q, skm.lvq4_points(q, d), oracle.lvq4_assign(codes, q["lvq"].cpu().numpy(), oracle.lvq4_encode(C.numpy()))
    q = skm.skm_quantize(skm.REPR_RBQ1, X.to(DEV))
    h = {n: v.cpu().numpy() for n, v in q.items()}
    codes = h["codes"].view(np.uint32)
    p = skm.rbq1_points(q, d)
    if sym:
        return q, p.with_flags(skm.FLAG_SYMMETRIC), oracle.rbq1_assign_sym(
            codes, h["nx2"], h["F"], d, oracle.rbq1_centroid_sym(C.numpy(), h["m"]))
    return q, p, oracle.rbq1_assign(codes, h["nx2"], h["F"], h["popx"], d, oracle.rbq1_centroid_sq4(C.numpy(), h["m"]))


def _check(got, want):
    np.testing.assert_array_equal(got[0].cpu().numpy(), want[0])
    np.testing.assert_array_equal(got[1].cpu().numpy(), want[1])


@pytest.mark.parametrize("kind,sym", [("rbq1", False), ("rbq1", True), ("lvq4", False)])
@pytest.mark.parametrize("n,d,k", [(129, 1152, 1), (700, 1530, 257), (1500, 1536, 300), (300, 2048, 33), (260, 4096, 40),
                                   (200, 1100, 20), (200, 1026, 20)])
def test_wide_assign_vs_oracle(skm, kind, sym, n, d, k):
    X = synth.gmm_points(n, d, 20, seed=n + d, decay=False)
    C = X[synth.forgy_indices(n, k, seed=3)] + 0.1
    q, p, want = _case(skm, kind, X, C, sym)
    _check(skm.skm_assign(p, C.to(DEV)), want)


@pytest.mark.parametrize("kind", ["rbq1", "lvq4"])
@pytest.mark.parametrize("d", [1536, 4096])
def test_wide_large_code_sums_exact(skm, kind, d):
    rng = np.random.default_rng(d)
    n, k = 300, 260
    X = np.ones((n, d), np.float32)
    X[np.arange(n), rng.integers(0, d, n)] = 0.0          # one code 0, the rest 15
    X[: n // 2] -= rng.integers(0, 2, (n // 2, d)).astype(np.float32) / 15.0
    if kind == "rbq1":
        X[n // 2:] = np.where(np.arange(n - n // 2)[:, None] % 2 == 0, X[n // 2:], -X[n // 2:])  # all bits 1 or 0
    C = np.ones((k, d), np.float32)
    C[np.arange(k), rng.integers(0, d, k)] = 0.0
    C[k // 2:] -= rng.integers(0, 3, (k - k // 2, d)).astype(np.float32) / 15.0
    q, p, want = _case(skm, kind, torch.from_numpy(X), torch.from_numpy(C))
    _check(skm.skm_assign(p, torch.from_numpy(C).to(DEV)), want)


@pytest.mark.parametrize("kind", ["rbq1", "lvq4"])
def test_wide_without_the_tensor_core_buffers(skm, kind):
    """A workspace of the size before the tensor-core path's buffers, and codes
    at an address that is no multiple of 16 bytes: the same results."""
    n, d, k = 400, 1536, 50
    X = synth.gmm_points(n, d, 20, seed=5, decay=False)
    C = X[synth.forgy_indices(n, k, seed=3)] + 0.1
    q, p, want = _case(skm, kind, X, C)
    W = q["codes"].shape[1]
    side = k * W * 16 + k * 16 if kind == "rbq1" else k * W * 4 + k * 16  # the CUDA-core kernel's centroid side
    small = torch.zeros(side + 2048, dtype=torch.uint8, device=DEV)
    assert small.numel() < skm.skm_workspace_size(skm.OP_ASSIGN, p, k)
    _check(skm.skm_assign(p, C.to(DEV), ws=small), want)
    buf = torch.empty(n * W + 4, dtype=torch.int32, device=DEV)
    off = buf[1: 1 + n * W].view(n, W)
    off.copy_(q["codes"])
    q2 = dict(q, codes=off)
    p2 = skm.lvq4_points(q2, d) if kind == "lvq4" else skm.rbq1_points(q2, d)
    _check(skm.skm_assign(p2, C.to(DEV)), want)
    # both in one size: what an unaligned address asks for also serves an aligned one
    ws = skm.workspace(skm.OP_ASSIGN, p2, k)
    _check(skm.skm_assign(p, C.to(DEV), ws=ws), want)
    with pytest.raises(skm.SkmError):
        skm.skm_assign(p, C.to(DEV), ws=torch.zeros(512, dtype=torch.uint8, device=DEV))


@pytest.mark.parametrize("kind", ["rbq1", "lvq4"])
def test_wide_fit_trajectory(skm, kind):
    n, d, k, iters = 2000, 1536, 20, 4
    X = synth.gmm_points(n, d, 30, seed=9, decay=True)
    idx = synth.forgy_indices(n, k, seed=9)
    if kind == "lvq4":
        q = skm.skm_quantize(skm.REPR_LVQ4, X.to(DEV))
        p, codes, fac = skm.lvq4_points(q, d), oracle.lvq4_unpack(q["codes"].cpu().numpy(), d), q["lvq"].cpu().numpy()
        C0 = oracle.lvq4_decode_points(codes, fac, p.rbq1_exp, idx.numpy())
        Co, ao = oracle.lloyd_lvq4(codes, fac, C0, iters, p.rbq1_exp)[:2]
    else:
        q = skm.skm_quantize(skm.REPR_RBQ1, X.to(DEV))
        h = {a: v.cpu().numpy() for a, v in q.items()}
        codes, p = h["codes"].view(np.uint32), skm.rbq1_points(q, d)
        C0 = oracle.rbq1_decode_points(codes, h["F"], d, h["m"], p.rbq1_exp, idx.numpy())
        Co, ao = oracle.lloyd_rbq1(codes, h["nx2"], h["F"], h["popx"], d, h["m"], C0, iters, p.rbq1_exp)[:2]
    C, a, _, _, _ = skm.skm_fit(p, k, iters, init_idx=idx.to(DEV))
    np.testing.assert_array_equal(a.cpu().numpy(), ao)
    np.testing.assert_array_equal(C.cpu().numpy(), Co)
