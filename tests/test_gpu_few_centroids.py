"""Assignments whose centroids fit one tile, and segmented ones whose groups are
narrower than a tile: equal to the same centroids listed twice (two tiles; ties go
to the lower index) and to every group assigned by itself.  Codes: bit for bit.
fp32 / bf16: a row that the screen decides goes to its exact nearest centroid, one
that it leaves open (as every copy does) to the nearest by fp32 distances, so the
two may part where both distances agree within such a sum's rounding."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"
KINDS = ["f32", "bf16", "sq8", "rbq1", "lvq4"]


@pytest.fixture(scope="module")
def skm(cuda_ok):
    import paper_2608_14648_gb300 as skm

    skm.lib()
    return skm


def _points(skm, kind, X):
    """The points and a function that takes some of their rows."""
    d = X.shape[1]
    if kind == "f32":
        x = X.to(DEV)
        return lambda r: skm.Points(skm.REPR_F32, x[r].contiguous(), d)
    if kind == "bf16":
        x = X.to(torch.bfloat16).view(torch.int16).to(DEV)
        return lambda r: skm.Points(skm.REPR_BF16, x[r].contiguous(), d)
    q = skm.skm_quantize({"sq8": skm.REPR_SQ8, "rbq1": skm.REPR_RBQ1, "lvq4": skm.REPR_LVQ4}[kind], X.to(DEV))
    if kind == "sq8":
        return lambda r: skm.Points(skm.REPR_SQ8, q["codes"][r].contiguous(), d)
    rows = ("codes", "nx2", "F", "popx") if kind == "rbq1" else ("codes", "lvq")
    whole = (skm.rbq1_points if kind == "rbq1" else skm.lvq4_points)(q, d)

    def take(r):
        p = {f: v[r].contiguous() if f in rows else v for f, v in q.items()}
        return (skm.rbq1_points if kind == "rbq1" else skm.lvq4_points)(p, d, e=whole.rbq1_exp)

    return take


def _centroids(kind, X, pts, k, g):
    pick = torch.randperm(X.shape[0], generator=g)[:k]
    return pts(pick.to(DEV)).x.clone() if kind == "sq8" else (X[pick] * 0.9).to(DEV)


def _same(kind, X, C, a, dist, a2, dist2):
    if kind in ("f32", "bf16"):
        off = (a != a2).nonzero().flatten()
        x = (X.to(torch.bfloat16) if kind == "bf16" else X)[off.cpu()].double()
        c = C.cpu().double()
        e, e2 = ((x - c[t[off].long().cpu()]).square().sum(1) for t in (a, a2))
        # d subtractions, squares and additions in fp32, on either side
        bound = 2 * (X.shape[1] + 2) * 2.0 ** -24
        assert bool(((e - e2).abs() <= bound * torch.maximum(e, e2)).all())
        a2, dist2 = torch.where(a != a2, a, a2), torch.where(a != a2, dist, dist2)
    assert torch.equal(a, a2) and torch.equal(dist, dist2)


@pytest.mark.parametrize("k", [1, 31, 33, 63, 64, 65, 96, 97, 128, 129, 200, 255, 256])
@pytest.mark.parametrize("n,d", [(700, 96), (45000, 128), (20011, 200)])
@pytest.mark.parametrize("kind", KINDS)
def test_one_tile_equals_two(skm, kind, n, d, k):
    g = torch.Generator().manual_seed(n + k)
    X = synth.gmm_points(n, d, 30, seed=n + d, decay=True)
    pts = _points(skm, kind, X)
    p = pts(slice(None))
    C = _centroids(kind, X, pts, k, g)
    a, dist = skm.skm_assign(p, C)
    a2, dist2 = skm.skm_assign(p, C.repeat(257 // k + 2, 1))
    _same(kind, X, C, a, dist, a2, dist2)


@pytest.mark.parametrize("sizes", [[63] * 6, [5, 120, 1, 30, 95, 129, 33], [97, 300, 128, 260, 64, 513, 31, 2]])
@pytest.mark.parametrize("d", [64, 200])
@pytest.mark.parametrize("kind", KINDS)
def test_groups_equal_separate_calls(skm, kind, d, sizes):
    g = torch.Generator().manual_seed(d + len(sizes))
    counts = [int(c) for c in torch.randint(1, 900, (len(sizes),), generator=g)]
    counts[1] = 40  # several groups in one point tile
    counts[2] = 3
    n, k = sum(counts), sum(sizes)
    X = synth.gmm_points(max(n, k), d, 30, seed=n, decay=True)
    pts = _points(skm, kind, X)
    C = _centroids(kind, X, pts, k, g)
    group = torch.cat([torch.full((c,), i, dtype=torch.int32) for i, c in enumerate(counts)]).to(DEV)
    base = torch.tensor([0] + sizes).cumsum(0).to(torch.int32).to(DEV)
    a, dist = skm.skm_assign_segmented(pts(slice(0, n)), C, group, base)
    at = 0
    for i, c in enumerate(counts):
        lo, hi = int(base[i]), int(base[i + 1])
        ag, dg = skm.skm_assign(pts(slice(at, at + c)), C[lo:hi].contiguous())
        _same(kind, X[at : at + c], C[lo:hi], a[at : at + c] - lo, dist[at : at + c], ag, dg)
        at += c
