"""Counts whose windows are cut into slices: few primaries against many secondaries, and
small catalogues with a reach of nearly half the box (a column pairs with itself, under
several images).  Counts are exact, sums within the documented 1e-5 (float32) and 1e-12.
"""
import numpy as np
import pytest

import oracle
import paper_1911_08275_gb300 as cf
from paper_1911_08275_gb300 import synth

pytestmark = pytest.mark.gpu

BOX = 60.0
EDGES = {"few": np.linspace(0.0, 25.0, 10), "many": np.linspace(0.0, 25.0, 31), "narrow": np.linspace(22.0, 25.0, 6)}


def dev(*arrays):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def catalogues(n1, n2):
    a = synth.uniform_box(n1, BOX, seed=331 + n1)
    b = synth.neyman_scott(n2 // 20, 20.0, 2.0, BOX, seed=332) if n2 else None
    return a, b


@pytest.mark.parametrize("edges", list(EDGES))
@pytest.mark.parametrize("mode", ["fp32_recheck", "fp64"])
@pytest.mark.parametrize("n1,n2", [(1, 20000), (33, 20000), (700, 20000), (6001, 0)])
def test_counts(cuda_device, n1, n2, mode, edges):
    a, b = catalogues(n1, n2)
    e = EDGES[edges]
    for periodic in (True, False):
        kw, okw = dict(boxsize=BOX, periodic=periodic, mode=mode), dict(periodic=periodic, box=BOX)
        if n2:
            kw.update(zip(("x2", "y2", "z2"), dev(b.x, b.y, b.z)))
            okw.update(x2=b.x, y2=b.y, z2=b.z, autocorr=False)
        xyz = dev(a.x, a.y, a.z)
        want = oracle.xi(a.x, a.y, a.z, edges=e, **okw)[0]
        assert np.array_equal(cf.countpairs_xi(*xyz, e, **kw).npairs, want)
        shards = [cf.countpairs_xi(*xyz, e, shard=(k, 3), **kw).npairs for k in range(3)]
        assert np.array_equal(sum(shards), want)
        want = oracle.rppi(a.x, a.y, a.z, rp_edges=e, pimax=28.0, npibins=7, **okw)[0]
        assert np.array_equal(cf.countpairs_rp_pi(*xyz, e, 28.0, 7, **kw).npairs, want)


@pytest.mark.parametrize("ravg", [False, True])
@pytest.mark.parametrize("mode", ["fp32_recheck", "fp64"])
@pytest.mark.parametrize("n1,n2", [(33, 20000), (6001, 0)])
def test_sums(cuda_device, n1, n2, mode, ravg):
    a, b = catalogues(n1, n2)
    rng = np.random.default_rng(333)
    wa, wb = rng.uniform(0.5, 1.5, a.n), rng.uniform(0.5, 1.5, b.n if n2 else 1)
    e = EDGES["narrow" if ravg else "few"]
    kw = dict(boxsize=BOX, mode=mode, want_ravg=ravg, w=dev(wa)[0])
    okw = dict(periodic=True, box=BOX, w1=wa, want_r=ravg)
    if n2:
        kw.update(zip(("x2", "y2", "z2", "w2"), dev(b.x, b.y, b.z, wb)))
        okw.update(x2=b.x, y2=b.y, z2=b.z, w2=wb, autocorr=False)
    xyz, tol = dev(a.x, a.y, a.z), 1e-12 if mode == "fp64" else 1e-5
    for r, ref in ((cf.countpairs_xi(*xyz, e, **kw), oracle.xi(a.x, a.y, a.z, edges=e, **okw)),
                   (cf.countpairs_rp_pi(*xyz, e, 28.0, 7, **kw),
                    oracle.rppi(a.x, a.y, a.z, rp_edges=e, pimax=28.0, npibins=7, **okw))):
        assert np.array_equal(r.npairs, ref[0]) and np.allclose(r.wsum, ref[1], rtol=tol, atol=0.0)
        if ravg:
            mean = np.divide(ref[2], ref[1], out=np.zeros_like(ref[2]), where=ref[1] != 0.0)
            assert np.allclose(r.ravg, mean, rtol=tol, atol=0.0)


@pytest.mark.parametrize("mode", ["fp32_recheck", "fp64"])
def test_few_primaries_take_about_as_long_as_the_other_order(cuda_device, mode):
    # 1,001 x 2M points, a reach of a seventh of the box: whole windows took 15 times (binary64
    # 35 times) as long as 2M x 1,001 (4.5 against 0.29 ms), slices 1.1 and 1.7 times
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(334)
    p = torch.rand((3, 2_001_001), generator=g, device="cuda", dtype=torch.float64) * 420.0
    a, b = ([p[k, s].contiguous() for k in range(3)] for s in (slice(0, 1001), slice(1001, None)))
    e = synth.log_edges(0.1, 60.0, 20)
    one = [cf.countpairs_xi(*a, e, x2=b[0], y2=b[1], z2=b[2], mode=mode) for _ in range(5)]
    two = [cf.countpairs_xi(*b, e, x2=a[0], y2=a[1], z2=a[2], mode=mode) for _ in range(5)]
    assert np.array_equal(one[0].npairs, two[0].npairs)
    assert min(r.kernel_ms for r in one) < 5.0 * min(r.kernel_ms for r in two)
