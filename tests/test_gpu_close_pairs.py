"""Float32 mean separations of points closer than their coordinates' float32 rounding.

Two float64 points 1e-8 apart may round to float32 neighbours 3e-5 apart (box of 420) or to
the same value: the separation then comes from the rounding residuals alone.  Per pair
r may be off by 1e-10 (a few residuals of at most 1e-4, each rounded to 2^-24 of itself),
by a few float32 roundings of r and, where only the squared distance is corrected, by
3e-6 of r; DD(r) rounds r w to a grid of at most
e_{k+1} max(w w) 2^-19, so by half of that (weights within [0.5, 1.5]: 9 times as much
relative to the weight).  wsum has the documented 1e-5.
"""
import numpy as np
import pytest

import oracle
import paper_1911_08275_gb300 as cf

pytestmark = pytest.mark.gpu

BOX = 420.0


def close_points():
    """Pairs 1e-8 to 1e-5 apart, around float32 rounding boundaries and elsewhere, some
    across the faces of the box, equal points, and a background."""
    rng = np.random.default_rng(301)
    c = rng.uniform(1.0, BOX - 1.0, (300, 3))
    f = c.astype(np.float32)
    half = f.astype(np.float64) * 0.5 + np.nextafter(f, np.float32(1e9)).astype(np.float64) * 0.5
    c[:200] = half[:200]
    c[190:230, 0] = 0.0
    off = 10.0 ** rng.uniform(-8, -5, (300, 1)) * rng.normal(size=(300, 3))
    p = np.concatenate([np.stack([c - off, c + off], 1).reshape(-1, 3), np.repeat(c[:20], 2, axis=0),
                        rng.uniform(0, BOX, (1500, 3))])
    p = np.where(p < 0.0, p + BOX, p)
    return p[(p < BOX).all(axis=1)]


@pytest.mark.parametrize("edges", [(0.0, 5.0, 20.0), (0.0, 1e-5, 1e-3, 20.0)])
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("cross", [False, True])
@pytest.mark.parametrize("kind", ["xi", "rppi"])
def test_ravg_of_close_pairs(cuda_device, kind, cross, weighted, periodic, edges):
    import torch
    p = close_points()
    w = np.random.default_rng(302).uniform(0.5, 1.5, len(p))
    e = np.array(edges)
    kw, okw, cols = {}, dict(periodic=periodic, box=BOX, want_r=True), []
    for s, x in ((slice(None, None, 2), "xyz"), (slice(1, None, 2), ("x2", "y2", "z2"))) if cross else ((slice(None), "xyz"),):
        v = [np.ascontiguousarray(p[s, k]) for k in range(3)]
        d = [torch.from_numpy(a).cuda() for a in v]
        ww = np.ascontiguousarray(w[s])
        if x == "xyz":
            cols, dev = v, d
        else:
            kw.update(zip(x, d))
            okw.update(zip(x, v), autocorr=False)
        if weighted:
            kw["w" if x == "xyz" else "w2"] = torch.from_numpy(ww).cuda()
            okw["w1" if x == "xyz" else "w2"] = ww
    if kind == "xi":
        r = cf.countpairs_xi(*dev, e, boxsize=BOX, periodic=periodic, want_ravg=True, **kw)
        n, ws, rs = oracle.xi(*cols, edges=e, **okw)
        grid = e[1:] * 2.0 ** -20 * (9.0 if weighted else 1.0)
    else:
        r = cf.countpairs_rp_pi(*dev, e, 20.0, 4, boxsize=BOX, periodic=periodic, want_ravg=True, **kw)
        n, ws, rs = oracle.rppi(*cols, rp_edges=e, pimax=20.0, npibins=4, **okw)
        grid = 0.0
    assert np.array_equal(r.npairs, n) and n.ravel()[0] > 0
    den = ws if weighted else n.astype(float)
    ref = np.divide(rs, den, out=np.zeros_like(rs), where=den != 0.0)
    assert np.all(np.abs(r.ravg - ref) <= grid + 1e-10 + 1e-5 * ref)
