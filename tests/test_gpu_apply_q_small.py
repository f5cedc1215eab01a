"""Back-transform of systems up to two warps of rows (n <= 64), and just above, against
Q from the oracle's reduction (column signs fixed): ragged column counts, a leading
dimension, in place.  50 n eps as for the other back-transform tests."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from tests.gpu_util import dev, sign_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,ncols,pad", [(1, 1, 3, 0), (2, 1, 1, 0), (2, 2, 700, 1), (5, 3, 9, 0), (8, 8, 64, 0),
                                           (31, 1, 17, 2), (32, 5, 2001, 0), (32, 32, 8, 0), (33, 5, 40, 0), (63, 2, 300, 3), (64, 1, 33, 0),
                                           (64, 20, 1200, 0), (65, 4, 40, 0)])
def test_small_systems(n, m, ncols, pad):
    from paper_1708_06290_gb300 import ssv
    sysr = W.random_system(n, m, 1, seed=8600 + n + m + ncols)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    H, R, _ = [t.cpu().numpy() for t in h.reduced()]
    Ho, Ro, _, Qo = oracle.reduce(sysr.A, sysr.B, sysr.C, want_q=True)
    Q = Qo * sign_matrix(R, H, Ro, Ho, m)[None, :]
    rng = np.random.default_rng(8601)
    x = rng.standard_normal((n, ncols)) + 1j * rng.standard_normal((n, ncols))
    buf = torch.zeros((ncols, n + pad), dtype=torch.complex128, device="cuda")
    X = buf.t()[:n]
    X.copy_(torch.from_numpy(x))
    Y = h.apply_q(X)
    h.apply_q(X, out=X)
    torch.cuda.synchronize()
    assert torch.equal(X, Y)
    if pad:
        assert float(buf[:, n:].abs().max()) == 0.0
    want = Q @ x
    assert np.linalg.norm(Y.cpu().numpy() - want) <= 50 * n * np.finfo(float).eps * np.linalg.norm(want)
    h.close()
