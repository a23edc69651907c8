"""What a user of the library has it do, as cases that can be timed: single
Lloyd steps (assign + update) in every point representation, the steps that
prepare the points (projection, encoding), the assignment of a small batch of
new points, and whole fits.

Points are Gaussian mixtures shaped like text and image embeddings (a decaying
spectrum, unit norm), the kind of data the paper clusters.  Everything a case
needs is drawn and encoded here with plain torch, so the inputs depend on the
seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2608_14648_gb300 as skm

# dimensions of embeddings in use: word vectors (100, 200, 300), descriptors
# (96, 128, 960), image and text encoders (384, 512, 768, 1024, 1536)
DIMS = (64, 96, 100, 128, 192, 200, 256, 300, 384, 512, 768, 960, 1024, 1536)
REPRS = {"f32": 0, "sq8": 1, "rbq1": 2, "bf16": 3, "lvq4": 4}
PRUNE = 1  # skm_data.flags: exact dimension pruning


def listed():
    return [
        # a small data set clustered in one call: launches and their gaps count
        {"name": "fit_sq8_20k_d128", "kind": "fit", "repr": "sq8", "n": 20_000, "d": 128, "k": 100, "iters": 10},
        # a batch of new points put into the clusters of an index that exists:
        # no copy of them is kept, and the distances are wanted too
        {"name": "batch_f32_2k_d768", "kind": "batch", "n": 2_000, "d": 768, "k": 1000},
        # Lloyd steps on full-precision embeddings at the size of a million
        {"name": "step_f32_1m_d768", "kind": "step", "repr": "f32", "n": 1_000_000, "d": 768, "k": 1000},
        # projected points kept in bf16, k = 4 sqrt(n) as the paper takes it, at a
        # size that is a multiple of nothing
        {"name": "step_bf16_700k_d192", "kind": "step", "repr": "bf16", "n": 700_001, "d": 192, "k": 3347},
        # ten million PCA-256 points once the centroids have settled: exact pruning
        # seeded with the previous step's assignment (the largest)
        {"name": "step_pruned_10m_d256", "kind": "pruned", "n": 10_000_000, "d": 256, "k": 10_000},
        # 8-bit codes, a million embeddings
        {"name": "step_sq8_1m_d1024", "kind": "step", "repr": "sq8", "n": 1_000_000, "d": 1024, "k": 1024},
        # 1-bit codes of millions of embeddings, read packed
        {"name": "step_rbq1_4m_d1024", "kind": "step", "repr": "rbq1", "n": 4_000_000, "d": 1024, "k": 3162},
        # 1-bit codes of the longer embeddings that text encoders give
        {"name": "step_rbq1_200k_d1536", "kind": "step", "repr": "rbq1", "n": 200_000, "d": 1536, "k": 1789},
        # 4-bit codes with a scale and a bias for each point, read packed
        {"name": "step_lvq4_1m_d768", "kind": "step", "repr": "lvq4", "n": 1_000_000, "d": 768, "k": 1000},
        # PCA projection of a million embeddings to bf16, before clustering
        {"name": "project_1m_d1024_256", "kind": "project", "n": 1_000_000, "d": 1024, "d_out": 256, "out": "bf16"},
        # 1-bit encoding of a million embeddings, the mean fitted on them
        {"name": "encode_rbq1_1m_d768", "kind": "encode", "repr": "rbq1", "n": 1_000_000, "d": 768},
        # hierarchical clustering of 1-bit codes into many clusters, one call
        {"name": "hier_rbq1_1m_d768", "kind": "hier", "n": 1_000_000, "d": 768, "k": 4000, "m": 63, "iters": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit", "batch", "step", "step", "step", "step", "step", "pruned", "project", "encode", "hier"])
    d = rng.choice(DIMS)
    if kind == "fit":
        n = _log(rng, 2_000, 200_000)
        return {"kind": kind, "repr": rng.choice(["sq8", "rbq1", "lvq4"]), "n": n, "d": min(d, 768),
                "k": max(8, int(rng.uniform(0.5, 2.0) * math.sqrt(n))),
                "iters": rng.randint(4, 12)}
    if kind == "batch":
        return {"kind": kind, "n": _log(rng, 64, 20_000), "d": d, "k": _log(rng, 256, 8192)}
    if kind == "pruned":
        n = _log(rng, 300_000, 2_000_000)
        return {"kind": kind, "n": n, "d": rng.choice([256, 320, 384, 512]), "k": int(rng.uniform(2.0, 4.0) * math.sqrt(n))}
    if kind == "project":
        n = _log(rng, 20_000, 1_000_000)
        d = max(d, 256)
        return {"kind": kind, "n": n, "d": d, "d_out": rng.choice([d // 4, 128, 192, d // 2, d]),
                "out": rng.choice(["f32", "bf16"])}
    if kind == "encode":
        return {"kind": kind, "repr": rng.choice(["sq8", "rbq1", "lvq4"]), "n": _log(rng, 20_000, 1_500_000), "d": d}
    if kind == "hier":
        n = _log(rng, 100_000, 1_000_000)
        return {"kind": kind, "n": n, "d": min(d, 1024), "k": int(4 * math.sqrt(n)), "m": int(2 * n ** 0.25),
                "iters": rng.randint(4, 10)}
    repr_ = rng.choice(["f32", "bf16", "sq8", "rbq1", "lvq4"])
    n = _log(rng, 20_000, 4_000_000)
    if d > 1024 and repr_ not in ("f32", "bf16"):
        n = min(n, _log(rng, 20_000, 200_000))
    c = rng.uniform(1.0, 4.0)
    while 2.0 * n * max(16, int(c * math.sqrt(n))) * d > 1.2e13:
        n = int(0.8 * n)
    return {"kind": kind, "repr": repr_, "n": n, "d": d, "k": max(16, int(c * math.sqrt(n)))}


# ---- inputs ------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _chunks(n, rows):
    for lo in range(0, n, rows):
        yield lo, min(n, lo + rows)


def _embeddings(n, d, comps, g, rotated=True):
    """Unit-norm mixture points float32 [n, d].  rotated: the decaying spectrum
    is spread over all dimensions (raw embeddings), else it lies along them in
    falling order (PCA's output)."""
    scale = (torch.arange(d, device="cuda", dtype=torch.float64) + 1).pow(-0.25).float()
    mix = torch.randn(d, d, device="cuda", generator=g) * (scale / math.sqrt(d)).unsqueeze(1) if rotated else None
    mu = torch.randn(comps, d, device="cuda", generator=g)
    x = torch.empty(n, d, device="cuda")
    for lo, hi in _chunks(n, 1 << 18):
        y = torch.randn(hi - lo, d, device="cuda", generator=g).mul_(0.3)
        y += mu[torch.randint(0, comps, (hi - lo,), device="cuda", generator=g)]
        y = y @ mix if rotated else y * scale
        x[lo:hi] = y / torch.linalg.vector_norm(y, dim=1, keepdim=True).clamp_min(1e-30)
    return x


def _nearest(x, c):
    """About the nearest centroid (tf32 products): the state of a run, not a result."""
    out = torch.empty(x.shape[0], dtype=torch.int64, device="cuda")
    cn, ct = c.square().sum(1), c.t().contiguous()
    was = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = True
    try:
        for lo, hi in _chunks(x.shape[0], 1 << 16):
            out[lo:hi] = torch.addmm(cn, x[lo:hi].float(), ct, alpha=-2).argmin(1)
    finally:
        torch.backends.cuda.matmul.allow_tf32 = was
    return out


def _settled(x, k, rounds, g):
    """Centroids after some Lloyd rounds from k of the points, and the last
    round's assignment.  The sums are integers, so their order does not matter."""
    c = x[torch.randperm(x.shape[0], device="cuda", generator=g)[:k]].float()
    a = None
    for _ in range(rounds):
        a = _nearest(x, c)
        s = torch.zeros(k, x.shape[1], dtype=torch.int64, device="cuda")
        for lo, hi in _chunks(x.shape[0], 1 << 18):
            s.index_add_(0, a[lo:hi], (x[lo:hi].float() * 2.0 ** 30).long())
        cnt = torch.bincount(a, minlength=k)
        c = torch.where(cnt.unsqueeze(1) > 0, (s.double() / (cnt.clamp_min(1).double() * 2.0 ** 30).unsqueeze(1)).float(), c)
    return c, a


def _sq8(x):
    b, hi = x.amin(0), x.amax(0)
    s = (hi - b) / 255
    s = torch.where(s > 0, s, torch.ones_like(s))
    codes = torch.empty(x.shape, dtype=torch.uint8, device="cuda")
    for lo, top in _chunks(x.shape[0], 1 << 18):
        codes[lo:top] = ((x[lo:top] - b) / s).round().clamp_(0, 255).to(torch.uint8)
    return codes, b, s


def _pack(bits, per):
    """[rows, d] small integers -> int32 words, `per` of them a word, lowest first."""
    rows, d = bits.shape
    w = -(-d // per)
    v = torch.zeros(rows, w * per, dtype=torch.int64, device="cuda")
    v[:, :d] = bits
    v = (v.view(rows, w, per) << (torch.arange(per, device="cuda") * (32 // per))).sum(2)
    return torch.where(v >= 1 << 31, v - (1 << 32), v).to(torch.int32)


def _unpack(words, d, per):
    v = words.long().unsqueeze(2) >> (torch.arange(per, device="cuda") * (32 // per))
    return (v & ((1 << (32 // per)) - 1)).reshape(words.shape[0], -1)[:, :d]


def _rbq1(x):
    n, d = x.shape
    m = sum(x[lo:hi].double().sum(0) for lo, hi in _chunks(n, 1 << 18)).div(n).float()
    codes = torch.empty(n, -(-d // 32), dtype=torch.int32, device="cuda")
    nx2, f = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    pop = torch.empty(n, dtype=torch.int32, device="cuda")
    for lo, hi in _chunks(n, 1 << 17):
        r = x[lo:hi] - m
        codes[lo:hi] = _pack(r > 0, 32)
        pop[lo:hi] = (r > 0).sum(1).int()
        r = r.double()
        q, l1 = r.square().sum(1), r.abs().sum(1)
        nx2[lo:hi] = q.float()
        f[lo:hi] = (math.sqrt(d) * q / l1.clamp_min(1e-300)).float()
    return {"codes": codes, "m": m, "nx2": nx2, "F": f, "popx": pop}


def _lvq4_terms(x, sums64=False):
    """Codes 0..15 and (s, b, N, A) of each row."""
    b = x.amin(1)
    s = (x.amax(1) - b) / 15
    s = torch.where(s > 0, s, torch.ones_like(s))
    codes = ((x - b.unsqueeze(1)) / s.unsqueeze(1)).round().clamp_(0, 15)
    t, q, sd, bd = codes.double().sum(1), codes.double().square().sum(1), s.double(), b.double()
    terms = torch.stack([sd, bd, sd * sd * q + 2 * bd * sd * t + x.shape[1] * bd * bd, sd * t + x.shape[1] * bd], 1)
    return codes, terms if sums64 else terms.float()


def _lvq4(x):
    n, d = x.shape
    codes = torch.empty(n, -(-d // 8), dtype=torch.int32, device="cuda")
    lvq = torch.empty(n, 4, device="cuda")
    for lo, hi in _chunks(n, 1 << 17):
        c, lvq[lo:hi] = _lvq4_terms(x[lo:hi])
        codes[lo:hi] = _pack(c.long(), 8)
    return {"codes": codes, "lvq": lvq}


def _comps(case):
    return min(10_000, max(32, 2 * case.get("k", 1000)))


def _inputs(case, seed):
    """What a case's points and centroids are, from the seed alone."""
    g = _gen(seed)
    n, d, kind = case["n"], case["d"], case["kind"]
    if kind == "pruned":
        x = _embeddings(n, d, case["k"], g, rotated=False).to(torch.bfloat16)
        c, a = _settled(x, case["k"], 4, g)
        return {"x": x, "C": c, "prev": a.int()}
    if kind == "batch":  # the index was built on other points of the same kind
        x = _embeddings(n + 16 * case["k"], d, _comps(case), g)
        return {"x": x[:n].clone(), "C": _settled(x[n:], case["k"], 2, g)[0]}
    x = _embeddings(n, d, _comps(case), g)
    if kind == "project":
        p = torch.linalg.qr(torch.randn(d, d, generator=torch.Generator().manual_seed(seed)))[0][:, :case["d_out"]]
        return {"x": x, "mean": x[: 1 << 16].mean(0), "P": p.contiguous().cuda()}
    if kind == "encode":
        return {"x": x}
    if kind in ("fit", "hier"):
        v = {"init": torch.randperm(n, device="cuda", generator=g)[:case["k" if kind == "fit" else "m"]]}
        r = case.get("repr", "rbq1")
        return {**v, "x": _sq8(x)[0]} if r == "sq8" else {**v, "q": _lvq4(x) if r == "lvq4" else _rbq1(x)}
    if case["repr"] == "bf16":
        x = x.to(torch.bfloat16)
    c, _ = _settled(x, case["k"], 2, g)
    if case["repr"] == "sq8":
        codes, b, s = _sq8(x)
        return {"x": codes, "C": ((c - b) / s).round().clamp_(0, 255).to(torch.uint8)}
    if case["repr"] == "rbq1":
        return {"q": _rbq1(x), "C": c}
    if case["repr"] == "lvq4":
        return {"q": _lvq4(x), "C": c}
    return {"x": x, "C": c}


def _points(case, v):
    r, d = case.get("repr"), case["d"]
    if case["kind"] == "pruned":
        return skm.Points(skm.REPR_BF16, v["x"].view(torch.int16), d, flags=PRUNE)
    if case["kind"] == "hier" or r == "rbq1":
        return skm.rbq1_points(v["q"], d)
    if r == "lvq4":
        return skm.lvq4_points(v["q"], d)
    if r == "bf16":
        return skm.Points(skm.REPR_BF16, v["x"].view(torch.int16), d)
    return skm.Points(REPRS[r] if r else skm.REPR_F32, v["x"], d)


def prepare(case, seed):
    v = _inputs(case, seed)
    s = {"case": case, "v": v}
    kind, n = case["kind"], case["n"]
    if kind in ("step", "pruned"):
        p = _points(case, v)
        if kind == "step" and case["repr"] in ("f32", "bf16", "sq8"):
            p = p.with_screen()  # built once for a data set: the points stay the same in all steps
        s.update(pts=p, ws=skm.workspace(skm.OP_ASSIGN, p, case["k"]), ws_up=skm.workspace(skm.OP_UPDATE, p, case["k"]),
                 assign=torch.empty(n, dtype=torch.int32, device="cuda"), next=v["C"].clone(),
                 counts=torch.zeros(case["k"], dtype=torch.int64, device="cuda"))
    elif kind == "fit":
        s["pts"] = _points(case, v)
        s["ws"] = skm.workspace(skm.OP_FIT, s["pts"], case["k"])
    elif kind == "encode":
        dummy = skm.Points(skm.REPR_F32, v["x"], case["d"])
        s["ws"] = skm.workspace(skm.OP_QUANTIZE, dummy, 1)
    elif kind == "hier":
        s["pts"] = _points(case, v)
    return s


def run(s):
    case, v = s["case"], s["v"]
    kind = case["kind"]
    if kind in ("step", "pruned"):
        a, _ = skm.skm_assign(s["pts"], v["C"], prev_assign=v.get("prev"), want_dist=False, ws=s["ws"], out=s["assign"])
        c, counts = skm.skm_update(s["pts"], a, s["next"], counts=s["counts"], ws=s["ws_up"])
        return {"assign": a, "C": c, "counts": counts}
    if kind == "batch":
        a, dist = skm.skm_assign(skm.Points(skm.REPR_F32, v["x"], case["d"]), v["C"])
        return {"assign": a, "dist": dist}
    if kind == "project":
        return skm.skm_project(v["x"], v["P"], v["mean"], skm.DTYPE_BF16 if case["out"] == "bf16" else skm.DTYPE_F32)
    if kind == "encode":
        return skm.skm_quantize(REPRS[case["repr"]], v["x"], ws=s["ws"])
    if kind == "fit":
        c, a, dist, obj, _ = skm.skm_fit(s["pts"], case["k"], case["iters"], init_idx=v["init"], ws=s["ws"])
        return {"C": c, "assign": a, "dist": dist, "objective": np.array(obj)}
    c, a, meso, fine, _ = skm.skm_fit_hierarchical(s["pts"], case["k"], case["m"], v["init"], case["iters"], case["iters"])
    return {"C": c, "assign": a, "meso": meso, "fine": np.array(fine)}


def work(case):
    n, d, k, kind = case["n"], case["d"], case.get("k", 0), case["kind"]
    row = {"f32": 4 * d, "bf16": 2 * d, "sq8": d, "rbq1": 4 * (-(-d // 32)) + 12, "lvq4": 4 * (-(-d // 8)) + 16}
    if kind in ("step", "pruned"):
        r = case.get("repr", "bf16")
        el = 1 if r == "sq8" else 4
        # pruned: every pair is looked at over the first dimensions, few beyond them
        return {"bytes": n * (row[r] + 4) + 2 * k * d * el, "flops": 2.0 * n * k * (128 if kind == "pruned" else d)}
    if kind == "batch":
        return {"bytes": n * (4 * d + 8) + 4 * k * d, "flops": 2.0 * n * k * d}
    if kind == "fit":
        return {"bytes": n * (row[case["repr"]] + 8) + 4 * k * d, "flops": 2.0 * n * k * d * (case["iters"] + 1)}
    if kind == "project":
        return {"bytes": n * (4 * d + (2 if case["out"] == "bf16" else 4) * case["d_out"]) + 4 * d * case["d_out"],
                "flops": 2.0 * n * d * case["d_out"]}
    if kind == "encode":
        return {"bytes": n * (4 * d + row[case["repr"]]), "flops": 2.0 * n * d}
    fine = 2.0 * n * (k / case["m"]) * d * (case["iters"] + 1)
    return {"bytes": n * (row["rbq1"] + 8) + 4 * k * d, "flops": 2.0 * n * case["m"] * d * (case["iters"] + 1) + fine}


# ---- the same in 64 bits, in plain torch --------------------------------------
def _argmin64(x, c):
    """The nearest centroid by 64-bit distances of the four nearest in fp32 products."""
    k = c.shape[0]
    c64, ct = c.double(), c.float().t().contiguous()
    cn = c.float().square().sum(1)
    a = torch.empty(x.shape[0], dtype=torch.int64, device="cuda")
    dist = torch.empty(x.shape[0], dtype=torch.float64, device="cuda")
    for lo, hi in _chunks(x.shape[0], 1 << 15):
        cand = torch.addmm(cn, x[lo:hi].float(), ct, alpha=-2).topk(min(4, k), 1, largest=False)[1].sort(1)[0]
        e = torch.stack([(x[lo:hi].double() - c64[cand[:, j]]).square().sum(1) for j in range(cand.shape[1])], 1)
        dist[lo:hi], j = e.min(1)
        a[lo:hi] = cand.gather(1, j.unsqueeze(1)).squeeze(1)
    return a, dist


def _mean64(rows, n, a, c):
    """Means of the members (rows(lo, hi): 64-bit rows); an empty cluster keeps its centroid."""
    s = torch.zeros(c.shape, dtype=torch.float64, device="cuda")
    for lo, hi in _chunks(n, 1 << 17):
        s.index_add_(0, a[lo:hi], rows(lo, hi))
    cnt = torch.bincount(a, minlength=c.shape[0]).unsqueeze(1)
    return torch.where(cnt > 0, s / cnt.clamp_min(1), c.double())


def _exact_codes(case, v):
    q, c, d = v["q"], v["C"], case["d"]
    n, k = q["codes"].shape[0], c.shape[0]
    a = torch.empty(n, dtype=torch.int64, device="cuda")
    one_bit = case["repr"] == "rbq1"
    if one_bit:
        rho = c - q["m"]
        b = rho.amin(1)
        s = (rho.amax(1) - b) / 15
        s = torch.where(s > 0, s, torch.ones_like(s))
        y = ((rho - b.unsqueeze(1)) / s.unsqueeze(1)).round().clamp_(0, 15)
        ny2, sy = rho.double().square().sum(1), y.double().sum(1)
        b, s = b.double() / math.sqrt(d), s.double() / math.sqrt(d)
    else:
        y, t = _lvq4_terms(c, sums64=True)
        gy = t[:, 0] * y.double().sum(1)
    yt = y.t().contiguous()
    for lo, hi in _chunks(n, 1 << 15):
        # small integers: these products and sums are exact in fp32
        p = (_unpack(q["codes"][lo:hi], d, 32 if one_bit else 8).float() @ yt).double()
        if one_bit:
            u = s * (2 * p - sy) + b * (2 * q["popx"][lo:hi].double() - d).unsqueeze(1)
            key = ny2 - 2 * q["F"][lo:hi].double().unsqueeze(1) * u
        else:
            f = q["lvq"][lo:hi].double()
            key = t[:, 2] - 2 * (f[:, 3:4] * t[:, 1] + f[:, 1:2] * gy + f[:, 0:1] * (t[:, 0] * p))
        a[lo:hi] = key.argmin(1)

    def rows(lo, hi):
        x = _unpack(q["codes"][lo:hi], d, 32 if one_bit else 8).double()
        if one_bit:
            return q["m"].double() + (2 * x - 1) * (q["F"][lo:hi].double() / math.sqrt(d)).unsqueeze(1)
        return x * q["lvq"][lo:hi, 0:1].double() + q["lvq"][lo:hi, 1:2].double()

    return {"assign": None, "C": _mean64(rows, n, a, c), "counts": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fit", "hier") or (kind == "step" and case["repr"] == "sq8"):
        return None  # chains of roundings to codes, or whole numbers only
    v = _inputs(case, seed)
    if kind == "step" and case["repr"] in ("rbq1", "lvq4"):
        return _exact_codes(case, v)
    x = v["x"]
    n, d = x.shape
    if kind in ("step", "pruned"):
        a, _ = _argmin64(x, v["C"])
        return {"assign": None, "C": _mean64(lambda lo, hi: x[lo:hi].double(), n, a, v["C"]), "counts": None}
    if kind == "batch":
        return {"assign": None, "dist": _argmin64(x, v["C"])[1]}
    if kind == "project":
        p, m = v["P"].double(), v["mean"].double()
        return torch.cat([(x[lo:hi].double() - m) @ p for lo, hi in _chunks(n, 1 << 17)])
    if case["repr"] == "sq8":
        b, hi = x.amin(0).double(), x.amax(0).double()
        return {"codes": None, "b": b, "s": torch.where(hi > b, (hi - b) / 255, torch.ones_like(b))}
    if case["repr"] == "lvq4":
        return {"codes": None, "lvq": torch.cat([_lvq4_terms(x[lo:hi], sums64=True)[1] for lo, hi in _chunks(n, 1 << 17)])}
    m = sum(x[lo:hi].double().sum(0) for lo, hi in _chunks(n, 1 << 18)) / n
    nx2, f = [], []
    for lo, hi in _chunks(n, 1 << 17):
        r = x[lo:hi].double() - m
        nx2.append(r.square().sum(1))
        f.append(math.sqrt(d) * nx2[-1] / r.abs().sum(1))
    return {"codes": None, "m": m, "nx2": torch.cat(nx2), "F": torch.cat(f), "popx": None}
