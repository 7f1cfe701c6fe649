"""The chunk-task kernels at the sizes where they can go wrong, against the oracle.

A column is padded to 32 entries and a warp takes 32 of them, so catalogues of one
column around 32, 64 and 192 points (chunk, two chunks, ring) cover the ragged ends;
bin counts around 23 cover the choice between one histogram word per pair and per two
pairs, and dense cells, -0.0 coordinates, empty second catalogues and mixed-sign
weights the other branches.  Counts are exact.  A float32 weight sum may be off
by half a unit of 2^-21 max|w_i w_j| per pair and by four float32 roundings
(2^-24 each) of every term.
"""
import threading

import numpy as np
import pytest

import oracle
import paper_1911_08275_gb300 as cf
from paper_1911_08275_gb300 import synth

pytestmark = pytest.mark.gpu

MODES = ["fp32_recheck", "fp64"]


def dev(*arrays):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def points(cat):
    return dev(cat.x, cat.y, cat.z)


@pytest.mark.parametrize("nbins", [1, 20, 22, 23, 24, 25])
@pytest.mark.parametrize("edges", ["log", "narrow"])
def test_bins_around_the_paired_histogram(cuda_device, nbins, edges):
    # log edges give table cells linear in d2, a narrow range cells on float bits
    e = synth.log_edges(0.1, 24.0, nbins) if edges == "log" else np.linspace(14.0, 18.0, nbins + 1)
    a = synth.neyman_scott(600, 20.0, 2.0, 150.0, seed=201)
    b = synth.uniform_box(5003, 150.0, seed=202)
    for periodic in (True, False):
        r = cf.countpairs_xi(*points(a), e, boxsize=150.0, periodic=periodic)
        assert np.array_equal(r.npairs, oracle.xi(a.x, a.y, a.z, edges=e, periodic=periodic, box=150.0)[0])
        x2, y2, z2 = points(b)
        r = cf.countpairs_xi(*points(a), e, x2=x2, y2=y2, z2=z2, boxsize=150.0, periodic=periodic)
        ref = oracle.xi(a.x, a.y, a.z, x2=b.x, y2=b.y, z2=b.z, edges=e, autocorr=False, periodic=periodic,
                        box=150.0)[0]
        assert np.array_equal(r.npairs, ref)


def test_paired_histogram_on_a_lattice(cuda_device):
    # every separation of a lattice sits on a bin edge: all pairs are flagged and settled
    g = np.arange(12) * 8.0
    x, y, z = (v.ravel().copy() for v in np.meshgrid(g, g, g, indexing="ij"))
    e = np.arange(0, 5) * 8.0
    r = cf.countpairs_xi(*dev(x, y, z), e, boxsize=96.0)
    assert np.array_equal(r.npairs, oracle.xi(x, y, z, edges=e, periodic=True, box=96.0)[0])


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 191, 192, 193, 1025])
def test_ragged_columns(cuda_device, mode, n):
    cat = synth.uniform_box(n, 60.0, seed=210 + n)
    other = synth.uniform_box(max(1, n - 7), 60.0, seed=211 + n)
    e = synth.log_edges(0.5, 25.0, 9)
    x2, y2, z2 = points(other)
    for periodic in (True, False):
        kw = dict(boxsize=60.0, periodic=periodic, mode=mode)
        okw = dict(periodic=periodic, box=60.0)
        r = cf.countpairs_xi(*points(cat), e, **kw)
        assert np.array_equal(r.npairs, oracle.xi(cat.x, cat.y, cat.z, edges=e, **okw)[0])
        r = cf.countpairs_rp_pi(*points(cat), e, 20.0, 5, **kw)
        ref = oracle.rppi(cat.x, cat.y, cat.z, rp_edges=e, pimax=20.0, npibins=5, **okw)[0]
        assert np.array_equal(r.npairs.ravel(), np.asarray(ref).ravel())
        r = cf.countpairs_xi(*points(cat), e, x2=x2, y2=y2, z2=z2, **kw)
        ref = oracle.xi(cat.x, cat.y, cat.z, x2=other.x, y2=other.y, z2=other.z, edges=e, autocorr=False,
                        **okw)[0]
        assert np.array_equal(r.npairs, ref)


@pytest.mark.parametrize("mode", MODES)
def test_dense_cells_and_signed_zeros(cuda_device, mode):
    # one cell of more entries than a warp ranks at once, repeated points, and -0.0
    rng = np.random.default_rng(220)
    p = np.concatenate([50.0 + rng.normal(0, 0.01, (700, 3)), rng.uniform(0, 100.0, (900, 3)),
                        np.full((40, 3), 50.0)])
    p[::97] = np.array([-0.0, 0.0, -0.0])
    x, y, z = (np.ascontiguousarray(p[:, k]) for k in range(3))
    e = synth.log_edges(1e-3, 20.0, 16)
    for dt in (np.float64, np.float32):
        a = [v.astype(dt) for v in (x, y, z)]
        a64 = [v.astype(np.float64) for v in a]
        for periodic in (True, False):
            r = cf.countpairs_xi(*dev(*a), e, boxsize=100.0, periodic=periodic, mode=mode)
            assert np.array_equal(r.npairs, oracle.xi(*a64, edges=e, periodic=periodic, box=100.0)[0])


@pytest.mark.parametrize("kind", ["xi", "rppi"])
@pytest.mark.parametrize("mode", MODES)
def test_counts_at_the_reach(cuda_device, kind, mode):
    # separations at, one ulp below and one ulp above Rmax and pimax, across the box's faces
    rng = np.random.default_rng(230)
    L, R, pm = 64.0, 16.0, 12.0
    base = rng.uniform(0, L, (400, 3))
    steps = [np.nextafter(R, 0), R, np.nextafter(R, 99), np.nextafter(pm, 0), pm, np.nextafter(pm, 99)]
    more = [np.mod(base + s * np.eye(3)[ax], L) for s in steps for ax in range(3)]
    p = np.concatenate([base] + more)
    p = p[(p < L).all(axis=1)]
    x, y, z = (np.ascontiguousarray(p[:, k]) for k in range(3))
    e = np.linspace(0.0, R, 9)
    if kind == "xi":
        got = cf.countpairs_xi(*dev(x, y, z), e, boxsize=L, mode=mode).npairs
        ref = oracle.xi(x, y, z, edges=e, periodic=True, box=L)[0]
    else:
        got = cf.countpairs_rp_pi(*dev(x, y, z), e, pm, 6, boxsize=L, mode=mode).npairs
        ref = oracle.rppi(x, y, z, rp_edges=e, pimax=pm, npibins=6, periodic=True, box=L)[0]
    assert np.array_equal(np.ravel(got), np.ravel(ref))


@pytest.mark.parametrize("kind", ["xi", "rppi"])
@pytest.mark.parametrize("n", [33, 3001])
def test_sums_of_mixed_weights(cuda_device, kind, n):
    cat = synth.uniform_box(n, 60.0, seed=240)
    rng = np.random.default_rng(241)
    w = rng.normal(0, 1, n) * 10.0 ** rng.uniform(-3, 0, n)
    w[::5] = 0.0
    e = synth.log_edges(0.5, 20.0, 8)
    x, y, z, wd = dev(cat.x, cat.y, cat.z, w)
    okw = dict(periodic=True, box=60.0)
    if kind == "xi":
        r = cf.countpairs_xi(x, y, z, e, w=wd, boxsize=60.0)
        f, okw = oracle.xi, dict(okw, edges=e)
    else:
        r = cf.countpairs_rp_pi(x, y, z, e, 20.0, 4, w=wd, boxsize=60.0)
        f, okw = oracle.rppi, dict(okw, rp_edges=e, pimax=20.0, npibins=4)
    cnt, ref, _ = f(cat.x, cat.y, cat.z, w1=w, **okw)
    size = np.ravel(f(cat.x, cat.y, cat.z, w1=np.abs(w), **okw)[1])
    cnt = np.ravel(cnt)
    assert np.array_equal(np.ravel(r.npairs), cnt)
    tol = cnt * 2.0 ** -22 * np.max(np.abs(w)) ** 2 + 4 * 2.0 ** -24 * size
    assert np.all(np.abs(np.ravel(r.wsum) - np.ravel(ref)) <= tol)


@pytest.mark.parametrize("njobs", [1, 3, 200])
def test_batch_of_uneven_jobs(cuda_device, njobs):
    # CTAs move between jobs of one point and of thousands, of both kinds and modes
    b, want = cf.Batch(), []
    for j in range(njobs):
        n = [1, 33, 700, 6000][j % 4] if njobs > 3 else 4000
        cat = synth.uniform_box(n, 80.0, seed=250 + j)
        kw = dict(boxsize=80.0, mode=MODES[(j // 2) % 2], periodic=j % 3 != 2)
        e = synth.log_edges(0.2, 20.0, 5 + j % 20)
        xyz = points(cat)
        if j % 2:
            want.append((b.add_rp_pi(*xyz, e, 15.0, 3, **kw), cf.countpairs_rp_pi(*xyz, e, 15.0, 3, **kw)))
        else:
            want.append((b.add_xi(*xyz, e, **kw), cf.countpairs_xi(*xyz, e, **kw)))
    for _ in range(2):
        b.run()
        assert all(np.array_equal(got.npairs, ref.npairs) for got, ref in want)
    b.close()


def test_calls_from_threads_on_their_own_streams(cuda_device):
    # the gridding's grid-wide barriers beside other calls' kernels
    import torch
    e = synth.log_edges(0.1, 25.0, 20)
    jobs = []
    for t in range(4):
        cat = synth.neyman_scott([500, 3000, 15000, 40][t], 20.0, 2.0, 200.0, seed=260 + t)
        xyz = points(cat)
        kw = dict(boxsize=200.0, mode=MODES[t % 2], periodic=t != 3)
        jobs.append((xyz, kw, cf.countpairs_xi(*xyz, e, **kw).npairs))
    torch.cuda.synchronize()
    bad = []

    def work(xyz, kw, ref):
        try:
            s = torch.cuda.Stream()
            for _ in range(25):
                if not np.array_equal(cf.countpairs_xi(*xyz, e, stream=s.cuda_stream, **kw).npairs, ref):
                    bad.append("counts")
        except Exception as err:  # noqa: BLE001 (a thread's failure is reported below)
            bad.append(repr(err))

    threads = [threading.Thread(target=work, args=j) for j in jobs for _ in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


@pytest.mark.parametrize("n2", [599_999, 600_000])
def test_binary64_evaluation_widths(cuda_device, n2):
    # a few primaries against more secondaries than the size where DD(r) goes from two
    # pairs per lane and evaluation to one, with sums (tolerance: order of summation)
    a = synth.uniform_box(301, 200.0, seed=270)
    b = synth.uniform_box(n2, 200.0, seed=271)
    rng = np.random.default_rng(272)
    w, w2 = rng.uniform(0.5, 1.5, a.n), rng.uniform(0.5, 1.5, b.n)
    e = synth.log_edges(0.5, 12.0, 9)
    x, y, z, wd = dev(a.x, a.y, a.z, w)
    x2, y2, z2, wd2 = dev(b.x, b.y, b.z, w2)
    r = cf.countpairs_xi(x, y, z, e, x2=x2, y2=y2, z2=z2, boxsize=200.0, mode="fp64")
    s = cf.countpairs_xi(x, y, z, e, w=wd, x2=x2, y2=y2, z2=z2, w2=wd2, boxsize=200.0, mode="fp64")
    cnt, ref, _ = oracle.xi(a.x, a.y, a.z, w1=w, x2=b.x, y2=b.y, z2=b.z, w2=w2, edges=e, autocorr=False,
                            periodic=True, box=200.0)
    assert np.array_equal(r.npairs, cnt) and np.array_equal(s.npairs, cnt)
    assert np.allclose(s.wsum, ref, rtol=1e-12, atol=0.0)
