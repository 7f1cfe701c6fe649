"""The one-launch gridding beside other work: it waits for no other stream and no block that
is not running, gives up cleanly, and the no-alloc entry point makes no CUDA object.
"""
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

import oracle
import paper_1911_08275_gb300 as cf
from paper_1911_08275_gb300 import synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def points(cat):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (cat.x, cat.y, cat.z)]


@pytest.mark.parametrize("cross", [False, True])
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("mode", ["fp32_recheck", "fp64"])
def test_gridding_that_gives_up_then_exact_counts(cuda_device, mode, periodic, cross):
    # the stages wait for a block that does not exist, 1 ms at most; no kernel after it runs
    # over the unfinished grid, and the next call on the same context is exact
    a = synth.neyman_scott(300, 20.0, 2.0, 90.0, seed=321)
    b = synth.uniform_box(5001, 90.0, seed=322)
    e = synth.log_edges(0.2, 15.0, 9)
    kw, okw = dict(boxsize=90.0, periodic=periodic, mode=mode), dict(periodic=periodic, box=90.0)
    if cross:
        kw.update(zip(("x2", "y2", "z2"), points(b)))
        okw.update(x2=b.x, y2=b.y, z2=b.z, autocorr=False)
    xyz = points(a)
    want = oracle.xi(a.x, a.y, a.z, edges=e, **okw)[0]
    for _ in range(2):
        for call in (lambda f: cf.countpairs_xi(*xyz, e, flags=f, **kw),
                     lambda f: cf.countpairs_rp_pi(*xyz, e, 10.0, 4, flags=f, **kw),
                     lambda f: cf.countpairs_xi(*xyz, e, flags=f, want_ravg=True, **kw)):
            t0 = time.perf_counter()
            with pytest.raises(cf.CfError) as ei:
                call(cf.CF_FLAG_DEBUG_STALL_GRID)
            assert ei.value.status == cf.CF_ETIMEOUT and time.perf_counter() - t0 < 5.0
        assert np.array_equal(cf.countpairs_xi(*xyz, e, **kw).npairs, want) and want.sum() > 0


def test_a_call_does_not_wait_for_another_stream(cuda_device):
    # stream a is busy for most of a second before its call's gridding can start; a call on
    # stream b returns long before that
    import torch
    cat = synth.uniform_box(20000, 200.0, seed=323)
    e = synth.log_edges(0.1, 20.0, 10)
    xyz = points(cat)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for s in (a, b, a, b):  # allocations of both streams
        ref = cf.countpairs_xi(*xyz, e, boxsize=200.0, stream=s.cuda_stream).npairs
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        torch.cuda._sleep(1_600_000_000)
    end = {}

    def call(name, s):
        n = cf.countpairs_xi(*xyz, e, boxsize=200.0, stream=s.cuda_stream).npairs
        end[name] = (time.perf_counter(), np.array_equal(n, ref))

    ta = threading.Thread(target=call, args=("a", a))
    t0 = time.perf_counter()
    ta.start()
    time.sleep(0.1)
    call("b", b)
    ta.join()
    assert end["a"][1] and end["b"][1]
    assert end["a"][0] - t0 > 0.3, "stream a was not busy long enough for the test to tell"
    assert end["b"][0] - t0 < 0.2


SHIM = r"""
#include <dlfcn.h>
#include <stddef.h>
static long made;
static void *real(const char *name)
{
    void *h = dlopen("libcudart.so.13", RTLD_NOLOAD | RTLD_LAZY);
    return h ? dlsym(h, name) : NULL;
}
#define WRAP(name, args, call) int name args { ++made; return ((int (*) args)real(#name)) call; }
WRAP(cudaMalloc, (void **p, size_t n), (p, n))
WRAP(cudaMallocAsync, (void **p, size_t n, void *s), (p, n, s))
WRAP(cudaHostAlloc, (void **p, size_t n, unsigned f), (p, n, f))
WRAP(cudaEventCreate, (void **e), (e))
WRAP(cudaEventCreateWithFlags, (void **e, unsigned f), (e, f))
WRAP(cudaStreamCreateWithFlags, (void **s, unsigned f), (s, f))
long made_so_far(void) { return made; }
"""

NOALLOC = r"""
import ctypes, sys
import numpy as np, torch
import paper_1911_08275_gb300 as cf
made = ctypes.CDLL(sys.argv[1]).made_so_far
made.restype = ctypes.c_long
rng = np.random.default_rng(324)
xyz = [torch.from_numpy(rng.uniform(0, 60.0, 3000)).cuda() for _ in range(3)]
e = np.linspace(0.0, 10.0, 6)
torch.cuda.synchronize()
stream = torch.cuda.current_stream().cuda_stream
for periodic in (True, False):
    n0 = made()
    r = cf.countpairs_xi_noalloc(*xyz, e, boxsize=60.0, periodic=periodic, stream=stream)
    assert made() == n0, f"{made() - n0} objects made"
n0 = made()
assert np.array_equal(cf.countpairs_xi(*xyz, e, boxsize=60.0, periodic=False, stream=stream).npairs, r.npairs)
assert made() > n0, "the calls of the library are not seen"
"""


def test_noalloc_makes_no_cuda_object(cuda_device, tmp_path):
    # counted by wrappers of the runtime's allocating calls, from the first call on
    src, so = tmp_path / "made.c", tmp_path / "made.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so), str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", NOALLOC, str(so)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, LD_PRELOAD=str(so)))
    assert r.returncode == 0, r.stderr[-2000:]
