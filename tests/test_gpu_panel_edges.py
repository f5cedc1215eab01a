"""The window panel in sub-blocks (every sweep) and its surroundings at the
sizes where the blocking can go wrong: one row, a sub-block less, exactly and
one more, a block less, exactly and one more, for every class of m and m at the
edge of a class; row counts of Ct around what is staged; and the grouping of
shifts in the tensor-core residual at ragged group sizes.

Tolerances: the parity tolerance of the sweeps, relative error <= 1e-10 against
the oracle's dense solve (the spectra lie in the disk of radius 1 about -2, the
shifts outside twice that, so kappa < 100); for the residual the
one derived in test_gpu_resid_tc: 5e-15 plus 1e-9 relative.
"""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from paper_1708_06290_gb300 import ssv
from tests.gpu_util import blocks, dev, relerr, shifts_dev

pytestmark = pytest.mark.gpu

SIG = np.array([0.4j, -0.9 + 1.7j, 3.0j, 0.2 + 0.05j])


def _check(sysr, h, sig, precision, nb=0):
    m = sysr.B.shape[1]
    o, st, _ = h.solve(shifts_dev(sig), mode="g", precision=precision, nb=nb)
    assert (st.cpu().numpy() == 0).all()
    X, _ = oracle.dense_solve(sysr.A, sysr.B, sig)
    Go = oracle.transfer(sysr.C, X)
    G = blocks(o, m)
    assert max(relerr(G[j], Go[j]) for j in range(len(sig))) <= 1e-10


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 8, 9, 12, 16, 17, 32])
@pytest.mark.parametrize("rows", [1, 15, 17, 29, 33, 127, 128, 129, 161])
def test_every_precision_at_block_edges(m, rows):
    n = m + rows
    sysr = W.random_system(n, m, 2, seed=8100 + 40 * m + rows)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    precs = ["fp64", "dfloat"] + (["split", "mixed"] if m <= 16 else [])
    for prec in precs:
        _check(sysr, h, SIG, prec)
    for nb in (1, 16, 17, 128):
        _check(sysr, h, SIG[:2], "fp64", nb=nb)
        _check(sysr, h, SIG[:2], "dfloat", nb=nb)
    # the tangential and transposed sweeps carry a right-hand side through the panel
    rng = np.random.default_rng(rows)
    b = rng.standard_normal((m, len(SIG))) + 1j * rng.standard_normal((m, len(SIG)))
    c = rng.standard_normal((2, len(SIG))) + 1j * rng.standard_normal((2, len(SIG)))
    x, _ = h.solve_rhs(shifts_dev(SIG), dev(b, torch.complex128), mode="x")
    y, _ = h.solve_trans(shifts_dev(SIG), dev(c, torch.complex128), mode="x")
    xo, _ = oracle.dense_solve_vec(sysr.A, (sysr.B @ b).T, SIG)
    yo, _ = oracle.dense_solve_vec(sysr.A, (sysr.C.T @ c).T, SIG, trans=True)
    for j in range(len(SIG)):
        assert relerr(x[:, j].cpu().numpy(), xo[j]) <= 1e-10
        assert relerr(y[:, j].cpu().numpy(), yo[j]) <= 1e-10
    h.close()


@pytest.mark.parametrize("m,p", [(1, 30), (2, 113), (8, 24), (8, 25), (16, 17), (16, 40), (20, 33)])
def test_rows_of_c(m, p):
    n = 300
    sysr = W.random_system(n, m, p, seed=8400 + m + p)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    for prec in ["fp64", "dfloat"] + (["split", "mixed"] if m <= 16 else []):
        _check(sysr, h, SIG, prec)


@pytest.mark.parametrize("m", [1, 2, 3, 4, 7, 8, 16])
@pytest.mark.parametrize("s", [1, 15, 17, 33])
def test_residual_groups(m, s):
    n = 150
    sysr = W.random_system(n, m, 1, seed=8600 + m)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    sig = 1j * np.logspace(-1, 1, s) - 0.1
    sd = shifts_dev(sig)
    X, _, _ = h.solve(sd, mode="xhat")
    rng = np.random.default_rng(s)
    for scale in (0.0, 1e-8):
        Xp = X.cpu().numpy()
        Xp = Xp * (1 + scale * rng.standard_normal(Xp.shape))
        Xd = dev(Xp, torch.complex128)
        a = h.backward_error(sd, Xd, method="tensor").cpu().numpy()
        b = h.backward_error(sd, Xd, method="fp64").cpu().numpy()
        assert np.all(np.abs(a - b) <= 1e-9 * b + 5e-15), (scale, a, b)


@pytest.mark.parametrize("n,m", [(2791, 8), (2800, 8), (2810, 3), (64, 40), (90, 17)])
def test_fp64_reduction_panel_in_and_out_of_shared_memory(n, m):
    """Panels of up to 22272 entries stay in shared memory (2784 rows of 8)."""
    rng = np.random.default_rng(n)
    A, B, C = rng.standard_normal((n, n)) / np.sqrt(n), rng.standard_normal((n, m)), rng.standard_normal((2, n))
    h = ssv.reduce(dev(A), dev(B), dev(C))
    H, R, Ct = h.reduced()
    x = dev(rng.standard_normal((n, 3)), torch.complex128)
    tol = 50 * n * np.finfo(float).eps
    Qx = h.apply_q(x)
    nrm = torch.linalg.vector_norm
    At = dev(A, torch.complex128)
    QHx = h.apply_q(ssv.colmajor(H.to(torch.complex128) @ x))
    assert float(nrm(At @ Qx - QHx) / (nrm(At) * nrm(x))) < tol
    QR = h.apply_q(ssv.colmajor(R.to(torch.complex128)))
    assert float(nrm(QR - dev(B, torch.complex128)) / np.linalg.norm(B)) < tol
    assert float(nrm(dev(C, torch.complex128) @ Qx - Ct.to(torch.complex128) @ x) / (np.linalg.norm(C) * nrm(x))) < tol
    h.close()
