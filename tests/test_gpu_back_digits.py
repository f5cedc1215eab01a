"""The wide back-transform by digit products (mode x of the precisions below FP64),
column by column against ssv_apply_q of the same Xhat on the FP64 pipe, at ragged
last blocks, several chunks of columns, more and fewer columns than a tile; shifts
over 15 decades, so the columns' norms differ as much.

Tolerance: either product of n reflectors leaves at most a few eps of a column per
block of reflectors, adding up as a random walk; n <= 1400 gives 1.5e-15 a side, and
5e-15 is what two digit levels fewer (2^-42) exceed by far.

Columns of a shift that is not finite are NaN and leave the others' bits alone.
"""
import numpy as np
import pytest
import torch

import workloads as W
from tests.gpu_util import dev, shifts_dev

pytestmark = pytest.mark.gpu


def columns_differ(x, y):
    """Largest relative difference of a column, over real and imaginary parts."""
    nrm = torch.linalg.vector_norm
    return float((nrm(x - y, dim=0) / nrm(y, dim=0)).max())


@pytest.mark.parametrize("n,m,s,prec,pad", [(256, 4, 176, "split", 0), (257, 1, 710, "mixed", 3),
                                            (500, 20, 18, "dfloat", 0), (769, 3, 79, "mixed", 0),
                                            (1100, 2, 530, "split", 1), (1400, 16, 9, "mixed", 0)])
def test_columns_against_the_fp64_path(n, m, s, prec, pad):
    from paper_1708_06290_gb300 import ssv
    assert n * m * s >= 180000
    sysr = W.random_system(n, m, 1, seed=8200 + n + m)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    sig = 1j * np.logspace(-3, 12, s)
    buf = torch.zeros((s * m, n + pad), dtype=torch.complex128, device="cuda")
    X = buf.t()[:n]
    _, st, _ = h.solve(shifts_dev(sig), mode="x", precision=prec, out=X)
    xhat = h.solve(shifts_dev(sig), mode="xhat", precision=prec)[0]
    ref = h.apply_q(xhat)
    torch.cuda.synchronize()
    assert (st == 0).all()
    assert columns_differ(X, ref) < 5e-15
    if pad:
        assert float(buf[:, n:].abs().max()) == 0.0
    # shifts that are not finite, in the first, a middle and the last place
    bad = [0, s // 2, s - 1]
    sig2 = sig.copy()
    sig2[bad] = [complex(np.nan, 0), complex(0, np.inf), complex(np.nan, np.nan)]
    X2, st2, _ = h.solve(shifts_dev(sig2), mode="x", precision=prec)
    torch.cuda.synchronize()
    good = [j for j in range(s) if j not in bad]
    blk = lambda a, js: a.reshape(n, s, m)[:, js]  # noqa: E731
    assert torch.isnan(blk(X2, bad).real).all()
    assert (st2[bad] != 0).all() and (st2[good] == 0).all()
    assert torch.equal(blk(X2, good), blk(X, good))
    h.close()
