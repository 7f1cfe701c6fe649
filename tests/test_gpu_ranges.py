"""Both sides of the sizes at which a count changes kernels: the last number of bins whose
float32 rows of weights and mean separations fit shared memory, and the secondaries up to
which one histogram word takes two pairs (fewer where the stencil is wider than the grid).
"""
import numpy as np
import pytest

import oracle
import paper_1911_08275_gb300 as cf
from paper_1911_08275_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(*arrays):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


@pytest.mark.parametrize("dtype", [np.float64, np.float32])  # with and without residuals
@pytest.mark.parametrize("nbins", [58, 59, 60, 64])
def test_weighted_ravg_around_the_last_float32_layout(cuda_device, nbins, dtype):
    cat = synth.neyman_scott(120, 20.0, 2.0, 80.0, seed=341).astype(dtype)
    w = np.random.default_rng(342).uniform(0.5, 1.5, cat.n)
    e = np.linspace(0.0, 25.0, nbins + 1)
    x, y, z, wd = dev(cat.x, cat.y, cat.z, w)
    r = cf.countpairs_xi(x, y, z, e, w=wd, boxsize=80.0, want_ravg=True)
    a = [v.astype(np.float64) for v in (cat.x, cat.y, cat.z)]
    n, ws, rs = oracle.xi(*a, edges=e, w1=w, periodic=True, box=80.0, want_r=True)
    assert np.array_equal(r.npairs, n) and np.allclose(r.wsum, ws, rtol=1e-5, atol=0.0)
    k = ws > 0
    # r w is rounded to a grid of at most e_{k+1} max(w w) 2^-19: bin 0 alone feels it
    grid = e[1:][k] * 2.0 ** -20 * n[k] * 2.25 / ws[k]
    assert np.all(np.abs(r.ravg[k] - rs[k] / ws[k]) <= 1e-5 * rs[k] / ws[k] + grid)


@pytest.mark.parametrize("box,rmax,n2", [(420.0, 20.0, 2 ** 23), (420.0, 20.0, 2 ** 23 + 1),
                                         (60.0, 25.0, 2 ** 23 // 9), (60.0, 25.0, 2 ** 23 // 9 + 1)])
def test_secondaries_around_the_paired_histogram(cuda_device, box, rmax, n2):
    a = synth.uniform_box(41, box, seed=343)
    b = synth.uniform_box(n2, box, seed=344).astype(np.float32)
    a = a.astype(np.float32)
    e = np.linspace(0.0, rmax, 12)
    x2, y2, z2 = dev(b.x, b.y, b.z)
    r = cf.countpairs_xi(*dev(a.x, a.y, a.z), e, x2=x2, y2=y2, z2=z2, boxsize=box)
    f = lambda c: [v.astype(np.float64) for v in (c.x, c.y, c.z)]  # noqa: E731
    xb, yb, zb = f(b)
    assert np.array_equal(r.npairs, oracle.xi(*f(a), x2=xb, y2=yb, z2=zb, edges=e, autocorr=False, periodic=True,
                                              box=box)[0])
