"""The calls that the library's performance is measured on.

A case is one call of the public binding as a user's program makes it: an EMST, an HDBSCAN* (tree,
core distances, ordered dendrogram and reachability plot), or a batch of independent instances.
Sizes and point distributions are those of the repository's own configurations: the scale suite
(10^7 points, uniform and variable-density blobs), the HDBSCAN* benchmark workload (10^6
Gaussian-mixture points in 3-D, minPts 10), the FP64 EMST of 10^4 points in the plane, the batched
mix (n log-uniform in [64, 65536]) and the served mix (host arrays, n in [10^3, 2x10^6], d in
{2, 3, 5, 7}, minPts in {10, 50}).
"""
import math

import numpy as np
import torch

import paper_2104_01126_gb300 as wm

_TORCH = {"f32": torch.float32, "f64": torch.float64}
_EXACT_MAX = 12_000   # points up to which the O(n^2) reference below stays within seconds


def listed():
    return [
        # a request of the smallest served size: latency, launches and host round trips
        dict(name="emst-gmm-1k-3d", call="emst", gen="gmm", n=1_000, d=3, dtype="f32"),
        # the paper-sized toy problem in FP64 coordinates (inexact FP32 screen copies)
        dict(name="emst-uniform-10k-2d-f64", call="emst", gen="uniform", n=10_000, d=2, dtype="f64"),
        # scale suite: low dimension, even density
        dict(name="emst-uniform-10m-3d", call="emst", gen="uniform", n=10_000_000, d=3, dtype="f32"),
        # scale suite: low dimension, density over three decades
        dict(name="emst-varden-10m-2d", call="emst", gen="varden", n=10_000_000, d=2, dtype="f32"),
        # scale suite: middle dimension, where the separation tests get expensive
        dict(name="emst-uniform-10m-5d", call="emst", gen="uniform", n=10_000_000, d=5, dtype="f32"),
        # scale suite: the hardest set, high dimension and variable density
        dict(name="emst-varden-10m-7d", call="emst", gen="varden", n=10_000_000, d=7, dtype="f32"),
        # a data set kept as FP64 columns, solved without the FP32 screen
        dict(name="emst-gmm-1m-3d-f64-columns", call="emst", gen="gmm", n=1_000_000, d=3, dtype="f64", layout="soa",
             precision="fp64"),
        # a small clustering job at an odd size
        dict(name="hdbscan-gmm-5003-5d-f64", call="hdbscan", gen="gmm", n=5_003, d=5, dtype="f64", min_pts=10,
             start=17),
        # the HDBSCAN* benchmark workload
        dict(name="hdbscan-gmm-1m-3d", call="hdbscan", gen="gmm", n=1_000_000, d=3, dtype="f32", min_pts=10, start=0),
        # a served clustering job with long neighbour lists in high dimension, ragged size
        dict(name="hdbscan-varden-300k-7d-k50", call="hdbscan", gen="varden", n=300_007, d=7, dtype="f32", min_pts=50,
             start=5),
        # a served clustering job as it arrives: host arrays in, host arrays out
        dict(name="hdbscan-gmm-200k-2d-host", call="hdbscan", gen="gmm", n=200_003, d=2, dtype="f32", min_pts=10,
             start=0, host=True),
        # many small independent instances, EMST and HDBSCAN* mixed
        dict(name="batch-192", call="batch", count=192, mix=1),
    ]


def draw(rng):
    """One more case of the same ranges: every field is drawn on its own, sizes over their logarithm."""
    call = rng.choice(["emst", "emst", "emst", "hdbscan", "hdbscan", "batch"])
    if call == "batch":
        return dict(call="batch", count=_log_int(rng, 12, 192), mix=rng.randrange(1 << 30))
    d = rng.choice([2, 3, 5, 7])
    gen = rng.choice(["uniform", "gmm", "varden"])
    dtype = rng.choice(["f32", "f32", "f64"])
    if call == "emst":
        case = dict(call="emst", gen=gen, n=_log_int(rng, 1_000, 9_000_000), d=d, dtype=dtype)
    else:
        n = _log_int(rng, 1_000, 1_000_000 if d <= 3 else 300_000)
        case = dict(call="hdbscan", gen=gen, n=n, d=d, dtype=dtype, min_pts=rng.choice([5, 10, 10, 50]),
                    start=rng.randrange(n))
    if rng.random() < 0.2:
        case["layout"] = "soa"
    if rng.random() < 0.15:
        case["precision"] = "fp64"
    if case["n"] <= 500_000 and rng.random() < 0.2:
        case["host"] = True
    return case


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# ------------------------------------------------------------------------------ point sets
def _points(gen, n, d, dtype, g):
    """n points on the GPU, rows in no particular order."""
    def rand(*shape):
        return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64 if dtype == "f64" else torch.float32)

    def randn(*shape):
        return torch.randn(*shape, generator=g, device="cuda",
                           dtype=torch.float64 if dtype == "f64" else torch.float32)

    if gen == "uniform":
        return rand(n, d)
    if gen == "gmm":
        # 50 isotropic Gaussians of random weight and width in a box of side 100, 5 % uniform noise
        k, noise = 50, round(0.05 * n)
        centre, width = 100 * rand(k, d), 0.1 * 50 ** rand(k)
        weight = -torch.log(1 - rand(k).double())
        label = torch.multinomial(weight, n - noise, replacement=True, generator=g)
        x = torch.cat([centre[label] + width[label, None] * randn(n - noise, d), 100 * rand(noise, d)])
        return x[torch.randperm(n, generator=g, device="cuda")]
    # 1000 Gaussian blobs in the unit cube, widths over three decades, sizes after Zipf (s = 1.1)
    k = 1000
    centre, width = rand(k, d), 1e-4 * 1000 ** rand(k)
    share = torch.arange(1, k + 1, device="cuda", dtype=torch.float64) ** -1.1
    edges = torch.cumsum(share / share.sum(), 0)
    label = torch.searchsorted(edges, torch.rand(n, generator=g, device="cuda", dtype=torch.float64)).clamp_(max=k - 1)
    return centre[label] + width[label, None] * randn(n, d)


def _instances(case):
    """(generator, n, d, min_pts, start) of every instance of a batch (a property of the case)."""
    g = np.random.default_rng([case["mix"], case["count"]])
    out = []
    for i in range(case["count"]):
        n = int(round(math.exp(g.uniform(math.log(64), math.log(65536)))))
        min_pts = int(g.choice([5, 10, 50])) if i % 2 else 1
        out.append((str(g.choice(["uniform", "gmm"])), n, int(g.choice([2, 3, 5])), min_pts, int(g.integers(n))))
    return out


def prepare(case, seed):
    wm.load()
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["call"] == "batch":
        inst = [(_points(gen, n, d, "f32", g), min_pts, start) for gen, n, d, min_pts, start in _instances(case)]
        return {"call": "batch", "instances": inst}
    x = _points(case["gen"], case["n"], case["d"], case["dtype"], g)
    layout = case.get("layout", "aos")
    if layout == "soa":
        x = x.t().contiguous()
    if case.get("host"):
        x = x.cpu().numpy()
    kw = {"precision": case.get("precision", "fp32"), "layout": layout}
    if case["call"] == "hdbscan":
        kw.update(min_pts=case["min_pts"], start=case["start"])
    return {"call": case["call"], "points": x, "options": kw}


def run(state):
    if state["call"] == "batch":
        # every field of all instances end to end, as the program hands them on
        res = wm.batch(state["instances"])
        out = {"total": np.array([r["total"] for r in res if "total" in r])}
        for key in ("u", "v", "w", "cd", "left", "right", "height", "size", "order", "reach"):
            out[key] = torch.cat([r[key] for r in res if key in r])
        return out
    if state["call"] == "emst":
        return wm.emst(state["points"], **state["options"])
    return wm.hdbscan(state["points"], **state["options"])


# ------------------------------------------------------------------------- necessary work
def _work_one(n, d, itemsize, min_pts):
    """Points read once, outputs written once; a comparison per coordinate and level of a spatial
    index, and per point its minPts (at least one) neighbour distances."""
    hdb = min_pts > 1
    bytes_ = n * d * itemsize + 16 * (n - 1) + ((8 + 4 + 8) * n + 20 * (n - 1) if hdb else 0)
    flops = n * d * math.ceil(math.log2(max(n, 2))) + 3 * d * n * max(min_pts, 1)
    return bytes_, flops


def work(case):
    if case["call"] == "batch":
        parts = [_work_one(n, d, 4, min_pts) for _, n, d, min_pts, _ in _instances(case)]
    else:
        parts = [_work_one(case["n"], case["d"], 4 if case["dtype"] == "f32" else 8, case.get("min_pts", 1))]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


# -------------------------------------------------------------------- 64-bit reference
def exact(case, seed):
    """Prim's algorithm on all point pairs in FP64.  Of the sizes in these ranges only the small
    ones can be answered this way in seconds."""
    if case["call"] == "batch" or case["n"] > _EXACT_MAX:
        return None
    host = case.get("host", False)
    x = prepare(case, seed)["points"]
    x = torch.as_tensor(x, device="cuda").double()
    if case.get("layout") == "soa":
        x = x.t()
    n, d = x.shape
    min_pts = case.get("min_pts", 1)
    cd2 = torch.zeros(n, device="cuda", dtype=torch.float64)
    if case["call"] == "hdbscan":
        for a in range(0, n, 1024):
            d2 = torch.zeros(min(1024, n - a), n, device="cuda", dtype=torch.float64)
            for k in range(d):
                t = x[a:a + 1024, k, None] - x[None, :, k]
                d2 += t * t
            cd2[a:a + 1024] = torch.kthvalue(d2, min_pts, dim=1).values
    ids = torch.arange(n, device="cuda")
    key = torch.full((n,), math.inf, device="cuda", dtype=torch.float64)    # best weight to the tree
    pair = torch.full((n,), 1 << 62, device="cuda", dtype=torch.int64)      # its (min id, max id)
    out = torch.zeros(n, device="cuda", dtype=torch.bool)
    w2 = torch.zeros(n, device="cuda", dtype=torch.float64)
    cur = torch.tensor(case.get("start", 0), device="cuda")
    for i in range(1, n):
        out[cur] = True
        key[cur] = math.inf
        d2 = torch.zeros(n, device="cuda", dtype=torch.float64)
        for k in range(d):
            t = x[:, k] - x[cur, k]
            d2 += t * t
        if case["call"] == "hdbscan":
            d2 = torch.maximum(d2, torch.maximum(cd2, cd2[cur]))
        p = torch.minimum(ids, cur) * (1 << 31) + torch.maximum(ids, cur)
        better = ~out & ((d2 < key) | ((d2 == key) & (p < pair)))
        key = torch.where(better, d2, key)
        pair = torch.where(better, p, pair)
        m = key.min()
        cur = torch.where(key == m, pair, 1 << 62).argmin()
        w2[i] = m
    bars = torch.sqrt(w2)
    w = torch.sort(bars[1:]).values
    if case["call"] == "emst":
        res = {"u": None, "v": None, "w": w, "total": float(w.sum())}
    else:
        bars[0] = math.inf
        res = {"u": None, "v": None, "w": w, "cd": torch.sqrt(cd2), "left": None, "right": None, "height": w.clone(),
               "size": None, "order": None, "reach": bars}
    if host:
        res = {k: v.cpu().numpy() if isinstance(v, torch.Tensor) else v for k, v in res.items()}
    return res
