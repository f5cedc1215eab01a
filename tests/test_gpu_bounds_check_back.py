"""The wide back-transform under the bounds-checked debug build: its kernels' indices
against their buffers, scratch poisoned with NaN, a canary after it.  An index out of
range, a changed canary or a read of unwritten scratch makes X NaN.  Shapes with a
ragged last block, one block, several chunks of columns; the panels' reads of H (the
sweep's own launches here) are checked by the same build."""
import os
import subprocess
import sys

import pytest

from paper_1708_06290_gb300 import build

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import numpy as np, torch
import workloads as W
from paper_1708_06290_gb300 import ssv
from tests.gpu_util import dev, shifts_dev
lib = ssv.load()
assert ssv.lib_path() != lib._name, "the debug copy must be the one loaded"
for n, m, s in [(256, 4, 176), (257, 1, 710), (385, 16, 40), (700, 2, 560)]:
    sysr = W.random_system(n, m, 1, seed=8400 + n)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    sd = shifts_dev(1j * np.logspace(-2, 2, s))
    X, st, _ = h.solve(sd, mode="x", precision="split")
    ref = h.apply_q(h.solve(sd, mode="xhat", precision="split")[0])
    torch.cuda.synchronize()
    assert (st == 0).all(), (n, m, s)
    nrm = torch.linalg.vector_norm
    assert float((nrm(X - ref, dim=0) / nrm(ref, dim=0)).max()) < 5e-15, (n, m, s)
    h.close()
print("bounds-checked back-transform ok")
'''


def test_wide_back_transform_passes_the_bounds_checked_build():
    lib = build.build(variant="check")
    env = dict(os.environ, SSV_LIBRARY=lib, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "bounds-checked back-transform ok" in r.stdout
