"""Back-transform X = Q Xhat in blocks of reflectors: on the FP64 pipe every
grouping of columns and rows (1-4 columns per cluster, 1-8 CTAs per cluster),
on the tensor cores several column chunks, in both a ragged last block and more
and fewer reflectors of Q_B than a block, against the definition of Q: Q^T Q = I,
B = Q R, A Q = Q H.

Tolerance: a product of n Householder reflectors in compact WY form has a
backward error of a small multiple of n eps per column; 50 n eps as for the
oracle's own reduction pins.
"""
import numpy as np
import pytest
import torch

import workloads as W
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,ncols,pad", [(2, 1, 1, 0), (33, 1, 1, 0), (34, 2, 3, 1), (97, 32, 5, 0),
                                           (65, 40, 2, 3), (300, 5, 40, 0), (300, 3, 153, 0), (290, 16, 305, 7),
                                           (1100, 4, 24, 0), (2300, 2, 2, 5), (700, 8, 620, 0),
                                           # wide: digit products on the tensor cores
                                           (256, 4, 704, 0), (384, 1, 720, 0), (769, 3, 365, 2), (1153, 130, 240, 0),
                                           (800, 2, 1100, 1), (1500, 16, 330, 0)])
def test_apply_q_definition(n, m, ncols, pad):
    from paper_1708_06290_gb300 import ssv
    sysr = W.random_system(n, m, 1, seed=5200 + n + m + ncols)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    H, R, _ = h.reduced()
    rng = np.random.default_rng(5201)
    tol = 50 * n * np.finfo(float).eps
    x = rng.standard_normal((n, ncols)) + 1j * rng.standard_normal((n, ncols))
    buf = torch.zeros((ncols, n + pad), dtype=torch.complex128, device="cuda")
    X = buf.t()[:n]
    X.copy_(torch.from_numpy(x))
    Y = h.apply_q(X)
    # in place, with a leading dimension
    h.apply_q(X, out=X)
    torch.cuda.synchronize()
    assert torch.equal(X, Y)
    if pad:
        assert float(buf[:, n:].abs().max()) == 0.0
    xt = torch.from_numpy(x).cuda()
    nrm = torch.linalg.vector_norm
    # isometry, column inner products included
    assert float(nrm(Y.mH @ Y - xt.mH @ xt) / nrm(xt.mH @ xt)) < tol
    # A Q x = Q H x
    A = torch.from_numpy(sysr.A).cuda().to(torch.complex128)
    QHx = h.apply_q(ssv.colmajor(H.to(torch.complex128) @ xt))
    assert float(nrm(A @ Y - QHx) / (nrm(A) * nrm(xt))) < tol
    # B = Q R
    QR = h.apply_q(ssv.colmajor(R.to(torch.complex128)))
    B = torch.from_numpy(sysr.B).cuda()
    assert float(nrm(QR - B) / nrm(B)) < tol
    h.close()
