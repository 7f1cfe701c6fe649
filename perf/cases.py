"""Performance cases: the pair counts that users of this framework run, through its public
entry points (``countpairs_xi``, ``countpairs_rp_pi``, ``countpairs_xi_noalloc``, ``Batch``).

A case is a dict of plain values.  The catalogues are those of the benchmark: a
Neyman-Scott stand-in for a galaxy catalogue (20 children per parent, sigma 2, listed
parent by parent) and uniform randoms, in a box of side 420 unless the case says
otherwise; they are drawn on the GPU from the seed alone.

Fields: entry ("xi", "rppi", "noalloc" or "batch"), n (points of the first catalogue),
n2 (points of the second, 0 for an auto-correlation), points ("clustered" or "uniform";
a second catalogue is uniform, as randoms are), dtype of the inputs, host (inputs in
page-locked host memory), mode, periodic, box, edges ("log" from 0.1 or "linear" from 0),
rmax, nbins, pimax, npibins, weighted, ravg; for a batch: jobs, scale, shapes (the seed
of the jobs' sizes).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1911_08275_gb300 as cf
from paper_1911_08275_gb300 import synth

CHILDREN, SIGMA = 20, 2.0

_DEFAULT = dict(entry="xi", n=0, n2=0, points="clustered", dtype="float64", host=False,
                mode="fp32_recheck", periodic=True, box=420.0, edges="log", rmax=25.0, nbins=20,
                pimax=0.0, npibins=0, weighted=False, ravg=False)


def _case(**kw) -> dict:
    return {**_DEFAULT, **kw}


def listed() -> list:
    return [
        # a mock or jackknife region of a few thousand to tens of thousands of points: latency
        _case(name="xi_20k", n=20_000, points="uniform"),
        # small scales of a whole catalogue kept in float32
        _case(name="xi_1.2M_r10_f32", n=1_198_890, dtype="float32", rmax=10.0),
        # the benchmark's headline: DD(r) of a 1.2M-point periodic box
        _case(name="xi_1.2M_r25", n=1_198_890),
        # the same from page-locked host memory, as a loader hands it over
        _case(name="xi_1.2M_r25_host", n=1_198_890, host=True),
        # large scales: the most pairs an unweighted count of this catalogue has
        _case(name="xi_1.2M_r50", n=1_198_890, rmax=50.0),
        # the same count asked for in binary64
        _case(name="xi_1.2M_r25_fp64", n=1_198_890, mode="fp64"),
        # wp(rp): 14 log rp bins, pimax 40 in unit bins
        _case(name="rppi_1.2M", entry="rppi", n=1_198_890, nbins=14, pimax=40.0, npibins=40),
        # the DR of a survey: weighted data against ten times as many weighted randoms, open
        # box, with the mean separation of each bin
        _case(name="dr_1.2Mx12M_w_ravg", n=1_198_890, n2=12_000_000, periodic=False, weighted=True,
              ravg=True),
        # weighted DD(r) of a volume-limited sample (odd size, float64, periodic)
        _case(name="xi_300k_w", n=301_237, weighted=True),
        # weighted wp's DR with the mean rp of each bin
        _case(name="rppi_dr_150kx300k_w_ravg", entry="rppi", n=150_001, n2=300_007, periodic=False,
              nbins=14, pimax=40.0, npibins=40, weighted=True, ravg=True),
        # many small jobs (sub-boxes, resamplings): DD(r) and DD(rp, pi), both modes
        _case(name="batch_480_small", entry="batch", jobs=480, scale=0.004, shapes=1000),
        # an analysis' list of uneven catalogues in one batch
        _case(name="batch_48_mixed", entry="batch", jobs=48, scale=0.25, shapes=1000),
    ]


def _loguniform(rng: random.Random, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# most unordered pairs in range that a drawn case may have, by what a pair costs
_MOST = {"plain": 5.0e9, "fp64": 6.0e8, "sums": 5.0e9, "sums_rppi": 4.0e8, "sums_fp64": 1.0e8}


def _class(c: dict) -> str:
    if c["weighted"] or c["ravg"]:
        return "sums_fp64" if c["mode"] == "fp64" else "sums_rppi" if c["entry"] == "rppi" else "sums"
    return "fp64" if c["mode"] == "fp64" else "plain"


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["xi", "xi", "xi", "xi_small", "xi_small", "rppi", "rppi", "fp64", "sums",
                       "sums", "sums_rppi", "noalloc", "batch"])
    if kind == "batch":
        jobs = int(_loguniform(rng, 8, 480))
        return _case(entry="batch", jobs=jobs, scale=min(0.25, 4.0 / jobs) * _loguniform(rng, 0.2, 1.0),
                     shapes=rng.randrange(1, 10 ** 6))
    c = _case(points=rng.choice(["clustered", "clustered", "uniform"]),
              dtype=rng.choice(["float64", "float64", "float32"]),
              rmax=round(_loguniform(rng, 5.0, 60.0), 2), nbins=rng.randint(8, 40),
              edges=rng.choice(["log", "log", "linear"]), periodic=rng.random() < 0.6)
    lo, hi = {"xi_small": (2e3, 6e4), "noalloc": (4e3, 1.3e5)}.get(kind, (4e4, 2e6))
    c["n"] = int(_loguniform(rng, lo, hi)) | 1
    if kind == "noalloc":
        c["entry"] = "noalloc"
    if kind in ("rppi", "sums_rppi") or (kind == "fp64" and rng.random() < 0.5):
        c.update(entry="rppi", pimax=round(rng.uniform(10.0, 60.0), 1), npibins=rng.randint(4, 60),
                 nbins=rng.randint(8, 20))
    if kind == "fp64" or (kind == "xi_small" and rng.random() < 0.2):
        c["mode"] = "fp64"
    if kind in ("sums", "sums_rppi"):
        c["weighted"], c["ravg"] = rng.choice([(True, False), (True, True), (True, True), (False, True)])
        if rng.random() < 0.15:
            c["mode"] = "fp64"
    if rng.random() < (0.6 if kind in ("sums", "sums_rppi") else 0.25):
        c["n2"] = c["n"] * (1 if kind == "noalloc" else rng.randint(1, 8)) - rng.randint(0, 3)
    if kind == "xi" and rng.random() < 0.3:
        c["host"] = True
    while _pairs(c) > _MOST[_class(c)]:
        c["n"] = int(c["n"] * 0.7) | 1
        c["n2"] = int(c["n2"] * 0.7)
    return c


# ---------------------------------------------------------------- inputs
def _generator(seed: int, stream: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + stream) % (1 << 62))
    return g


def _points(n: int, points: str, box: float, dtype: str, g: torch.Generator) -> list:
    if points == "uniform":
        p = torch.rand((3, n), generator=g, device="cuda", dtype=torch.float64) * box
    else:
        parents = max(1, n // CHILDREN)
        owner = torch.randint(parents, (n,), generator=g, device="cuda").sort().values
        centre = torch.rand((3, parents), generator=g, device="cuda", dtype=torch.float64) * box
        p = centre[:, owner]
        p += SIGMA * torch.randn((3, n), generator=g, device="cuda", dtype=torch.float64)
        p = torch.remainder(p, box)
    p = p.to(getattr(torch, dtype))
    p[p >= box] = 0.0  # a coordinate that rounds up to the side of the box
    return [p[a].contiguous() for a in range(3)]


def _weights(n: int, g: torch.Generator) -> torch.Tensor:
    return 0.5 + torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _edges(c: dict) -> np.ndarray:
    return (synth.log_edges(0.1, c["rmax"], c["nbins"]) if c["edges"] == "log"
            else synth.linear_edges(0.0, c["rmax"], c["nbins"]))


def _jobs(c: dict) -> list:
    """Sizes and options of a batch's jobs (those of the 48-job workload, scaled)."""
    r = random.Random(c["shapes"])
    jobs = []
    for j in range(c["jobs"]):
        box = _loguniform(r, 100.0, 1000.0)
        rmax = float(min(round(_loguniform(r, 5.0, 40.0)), int(box / 2.0) - 1))
        n = max(2, int(_loguniform(r, 5e4, 2e6) * c["scale"]))
        rppi = (j // 2) % 2 == 1
        job = _case(entry="rppi" if rppi else "xi", n=n, points="uniform" if j % 2 else "clustered",
                    mode="fp64" if (j // 4) % 2 else "fp32_recheck", box=box, rmax=rmax)
        if rppi:
            job.update(nbins=14, pimax=rmax, npibins=int(rmax))
        jobs.append(job)
    return jobs


def _inputs(c: dict, seed: int) -> tuple:
    """The catalogues on the GPU: (coordinates, weights) of each."""
    g = _generator(seed, 1)
    cats = [(_points(c["n"], c["points"], c["box"], c["dtype"], g), None)]
    if c["n2"]:
        cats.append((_points(c["n2"], "uniform", c["box"], c["dtype"], g), None))
    if c["weighted"]:
        cats = [(p, _weights(p[0].numel(), g)) for p, _ in cats]
    return tuple(cats)


def prepare(case: dict, seed: int) -> dict:
    c = _case(**case)
    if c["entry"] == "batch":
        b, results = cf.Batch(), []
        for k, job in enumerate(_jobs(c)):
            x = _points(job["n"], job["points"], job["box"], job["dtype"], _generator(seed, 100 + k))
            kw = dict(boxsize=job["box"], mode=job["mode"])
            results.append(b.add_rp_pi(*x, _edges(job), job["pimax"], job["npibins"], **kw)
                           if job["entry"] == "rppi" else b.add_xi(*x, _edges(job), **kw))
        return {"batch": b, "results": results}
    cats = _inputs(c, seed)
    if c["host"]:
        cats = tuple(([v.cpu().pin_memory() for v in p], None if w is None else w.cpu().pin_memory())
                     for p, w in cats)
    args = [*cats[0][0], _edges(c)]
    kw = dict(periodic=c["periodic"], boxsize=c["box"], mode=c["mode"])
    if len(cats) > 1:
        kw.update(x2=cats[1][0][0], y2=cats[1][0][1], z2=cats[1][0][2])
    if c["entry"] != "noalloc":
        kw["want_ravg"] = c["ravg"]
        if c["weighted"]:
            kw["w"] = cats[0][1]
            if len(cats) > 1:
                kw["w2"] = cats[1][1]
    if c["entry"] == "rppi":
        args += [c["pimax"], c["npibins"]]
    call = {"xi": cf.countpairs_xi, "rppi": cf.countpairs_rp_pi, "noalloc": cf.countpairs_xi_noalloc}
    return {"call": call[c["entry"]], "args": args, "kw": kw}


def run(state: dict):
    if "batch" in state:
        state["batch"].run()
        return {"npairs": np.concatenate([r.npairs.ravel() for r in state["results"]])}
    r = state["call"](*state["args"], **state["kw"])
    out = {"npairs": r.npairs}
    if r.wsum is not None:
        out["wsum"] = r.wsum
    if r.ravg is not None:
        out["ravg"] = r.ravg
    return out


# ---------------------------------------------------------------- what a pass needs
def _pairs(c: dict) -> float:
    """Expected pairs in range (each unordered pair of an auto-correlation once)."""
    vol = (math.pi * c["rmax"] ** 2 * 2.0 * c["pimax"] if c["entry"] == "rppi"
           else 4.0 / 3.0 * math.pi * c["rmax"] ** 3) / c["box"] ** 3
    if c["n2"]:
        return float(c["n"]) * c["n2"] * vol
    pairs = 0.5 * float(c["n"]) ** 2 * vol
    if c["points"] == "clustered":  # pairs of children of one parent
        pairs += 0.5 * c["n"] * CHILDREN
    return pairs


def work(case: dict) -> dict:
    c = _case(**case)
    parts = _jobs(c) if c["entry"] == "batch" else [c]
    nbytes = flops = 0.0
    for p in parts:
        points = p["n"] + p["n2"]
        size = 4 if p["dtype"] == "float32" else 8
        slots = p["nbins"] * max(1, p["npibins"])
        nbytes += points * (3 * size + (8 if p["weighted"] else 0))
        nbytes += slots * 8 * (1 + int(p["weighted"]) + int(p["ravg"]))
        # three differences, three squares, two sums; a weight product and two sums, a root
        per = 8 + (2 if p["weighted"] else 0) + (3 if p["ravg"] else 0)
        flops += per * _pairs(p)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- 64-bit values
_MOST_TESTED = 6.0e10  # candidate pairs beyond which the values would take too long


def _count(c: dict, cats: tuple) -> dict:
    """Counts and sums in binary64 torch operations: primaries in blocks sorted by z against
    the slab of secondaries within reach (periodic images of the slab listed explicitly)."""
    auto = not c["n2"]
    edges = _edges(c)
    e2 = torch.from_numpy(edges * edges).cuda()
    rppi = c["entry"] == "rppi"
    npi = c["npibins"] if rppi else 1
    slots = c["nbins"] * npi
    reach = c["pimax"] if rppi else float(edges[-1])
    pe = torch.tensor([c["pimax"] * m / npi for m in range(npi)] + [c["pimax"]],
                      dtype=torch.float64, device="cuda") if rppi else None
    a = torch.stack([v.double() for v in cats[0][0]])
    wa = cats[0][1] if c["weighted"] else torch.ones_like(a[0])
    b, wb = (a, wa) if auto else (torch.stack([v.double() for v in cats[1][0]]),
                                  cats[1][1] if c["weighted"] else None)
    if wb is None:
        wb = torch.ones_like(b[0])
    box = c["box"]
    order = torch.argsort(a[2])
    key, idx = b[2], torch.arange(b.shape[1], device="cuda")
    if c["periodic"]:
        up, down = idx[b[2] < reach], idx[b[2] >= box - reach]
        key = torch.cat([key, b[2][up] + box, b[2][down] - box])
        idx = torch.cat([idx, up, down])
    s = torch.argsort(key)
    key, idx = key[s], idx[s]
    n = torch.zeros(slots, dtype=torch.int64, device="cuda")
    ws = torch.zeros(slots, dtype=torch.float64, device="cuda")
    rs = torch.zeros(slots, dtype=torch.float64, device="cuda")
    k0 = 0
    while k0 < order.numel():
        k1 = min(order.numel(), k0 + 256)
        ia = order[k0:k1]
        za = a[2][ia]
        pad = 1e-6 * box
        lo, hi = torch.searchsorted(key, torch.stack([za[0] - reach - pad, za[-1] + reach + pad])).tolist()
        k0 = k1
        step = max(1, 60_000_000 // max(1, ia.numel()))
        for j0 in range(lo, hi, step):
            jb = idx[j0:min(hi, j0 + step)]
            d = []
            for ax in range(3):
                v = b[ax][jb][None, :] - a[ax][ia][:, None]
                if c["periodic"]:
                    v = torch.where(v > 0.5 * box, v - box, torch.where(v < -0.5 * box, v + box, v))
                d.append(v)
            s2 = d[0] * d[0] + d[1] * d[1]
            pi = d[2].abs()
            if not rppi:
                s2 = s2 + d[2] * d[2]
            ok = (s2 >= e2[0]) & (s2 < e2[-1])
            if rppi:
                ok &= pi < c["pimax"]
            if auto:
                ok &= jb[None, :] != ia[:, None]
            at = ok.nonzero(as_tuple=True)
            s2 = s2[at]
            slot = torch.bucketize(s2, e2, right=True) - 1
            if rppi:
                slot = slot * npi + torch.bucketize(pi[at], pe, right=True) - 1
            w = wa[ia][at[0]] * wb[jb][at[1]]
            n += torch.bincount(slot, minlength=slots)
            ws += torch.bincount(slot, weights=w, minlength=slots)
            if c["ravg"]:
                rs += torch.bincount(slot, weights=w * s2.sqrt(), minlength=slots)
    out = {"npairs": n.cpu().numpy().astype(np.uint64)}
    shape = (c["nbins"], npi) if rppi else (c["nbins"],)
    out["npairs"] = out["npairs"].reshape(shape)
    if c["weighted"]:
        out["wsum"] = ws.cpu().numpy().reshape(shape)
    if c["ravg"]:
        out["ravg"] = torch.where(n > 0, rs / ws.clamp(min=1e-300), rs).cpu().numpy().reshape(shape)
    return out


def exact(case: dict, seed: int):
    c = _case(**case)
    if c["entry"] == "batch":
        return None  # counts only, of too many jobs
    reach = c["pimax"] if c["entry"] == "rppi" else c["rmax"]
    tested = float(c["n"]) * (c["n2"] or c["n"]) * min(1.0, 2.2 * reach / c["box"])
    if tested > _MOST_TESTED:
        return None
    return _count(c, _inputs(c, seed))
