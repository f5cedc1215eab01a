"""FP64 reduction with one-column panels (m = 1): rows within and beyond what a thread
keeps in registers, the smallest systems, an exact zero column, and the step from B's
last group of one reflector to a wide panel (m = 9, 17). Q^T Q = I and A Q = Q H, B = Q R
on random vectors, 50 n eps."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,zero", [(2, 1, False), (3, 1, False), (33, 1, False), (512, 1, False), (514, 1, True),
                                      (700, 9, False), (300, 17, False), (4200, 1, False)])
def test_invariants(n, m, zero):
    from paper_1708_06290_gb300 import ssv
    sysr = W.random_system(n, m, 2, seed=8700 + n + m)
    A = sysr.A.copy()
    if zero:  # a column that is annihilated already, mid-way: two uncoupled halves
        A[n // 2:, :n // 2] = 0.0
        sysr.B[n // 2:] = 0.0
    h = ssv.reduce(dev(A), dev(sysr.B), dev(sysr.C))
    H, R, Ct = h.reduced()
    rng = np.random.default_rng(8701)
    x = torch.from_numpy(rng.standard_normal((n, 3)) + 1j * rng.standard_normal((n, 3))).cuda()
    x = ssv.colmajor(x)
    Qx = h.apply_q(x)
    nrm = torch.linalg.vector_norm
    tol = 50 * n * np.finfo(float).eps
    assert float(nrm(Qx.mH @ Qx - x.mH @ x) / nrm(x.mH @ x)) < tol
    Ad, c = torch.from_numpy(A).cuda().to(torch.complex128), lambda t: t.to(torch.complex128)
    assert float(nrm(Ad @ Qx - h.apply_q(ssv.colmajor(c(H) @ x))) / (nrm(Ad) * nrm(x))) < tol
    B = torch.from_numpy(sysr.B).cuda()
    assert float(nrm(h.apply_q(ssv.colmajor(c(R))) - B) / nrm(B)) < tol
    C = torch.from_numpy(sysr.C).cuda()
    assert float(nrm(c(Ct) @ x - c(C) @ Qx) / (nrm(C) * nrm(x))) < tol
    h.close()
