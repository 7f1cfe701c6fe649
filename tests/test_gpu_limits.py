"""A planned batch keeps the shared memory it was planned with, whatever runs meanwhile.

A kernel's dynamic shared-memory limit is raised when a call needs more; a batch asks
only when it is planned.  A process that has used many of the library's kernels (every
shape, option and kind of sums) and then plans a batch with a large and one with a small
histogram must still be able to run the first.  A process of its own: the limits are kept
for the life of the process.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = r"""
import numpy as np, torch
import paper_1911_08275_gb300 as cf

rng = np.random.default_rng(311)
f64 = [torch.from_numpy(rng.uniform(0, 60.0, 300)).cuda() for _ in range(3)]
f32 = [v.float() for v in f64]
w = torch.from_numpy(rng.uniform(0.5, 1.5, 300)).cuda()
linear, narrow = np.linspace(0.0, 20.0, 9), np.linspace(14.0, 15.0, 9)
for e in (linear, narrow):
    for flags in (0, cf.CF_FLAG_COUNT_EVALS):
        kw = dict(boxsize=60.0, flags=flags)
        for chunk, pp in ((8, 1), (16, 1), (32, 1), (8, 2), (16, 2), (8, 4)):
            cf.countpairs_xi(*f64, e, pair_chunk=chunk, pair_pp=pp, **kw)
        for xyz in (f32, f64):
            for sums in (dict(), dict(w=w), dict(want_ravg=True), dict(w=w, want_ravg=True)):
                for mode in ("fp32_recheck", "fp64"):
                    cf.countpairs_xi(*xyz, e, mode=mode, **sums, **kw)
                    cf.countpairs_rp_pi(*xyz, e, 20.0, 2, mode=mode, **sums, **kw)
large, small = cf.Batch(), cf.Batch()
a = large.add_rp_pi(*f64, linear, 20.0, 512, boxsize=60.0)
b = small.add_rp_pi(*f64, linear, 20.0, 2, boxsize=60.0)
for batch in (large, small, large, small):
    batch.run(use_graph=False)
for r, npi in ((a, 512), (b, 2)):
    assert np.array_equal(r.npairs, cf.countpairs_rp_pi(*f64, linear, 20.0, npi, boxsize=60.0).npairs)
"""


def test_batch_launches_after_many_other_kernels(cuda_device):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
