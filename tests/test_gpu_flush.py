"""The overflow flushes of the counts' shared words, which only runs of some 1e12 pairs reach:
a build that flushes a million times as often repeats the comparisons with the oracle.
"""
import os
import subprocess
import sys

import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import os, sys
import paper_1911_08275_gb300.build as b
b.OUTDIR = sys.argv[1]
b.LIB = os.path.join(b.OUTDIR, "libcfgpu.so")
b.build(force=True, extra=["-DCF_FLUSH_SHIFT=20"])
import pytest
import paper_1911_08275_gb300 as cf
assert cf.lib()._name == b.LIB
sys.exit(pytest.main(["-q", "-x", "-m", "gpu", "-p", "no:cacheprovider"] + [os.path.join("tests", f) for f in (
    "test_gpu_xi.py", "test_gpu_rppi.py", "test_gpu_tasks.py", "test_gpu_slices.py", "test_gpu_batch.py")]))
"""


def test_counts_with_frequent_flushes(cuda_device, tmp_path):
    r = subprocess.run([sys.executable, "-c", SCRIPT, str(tmp_path)], cwd=ROOT, capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-1000:]
    assert " passed" in r.stdout
