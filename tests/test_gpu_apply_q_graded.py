"""ssv_apply_q keeps the small entries of a graded column: on a system of two
uncoupled halves the reflectors of one have exact zeros in the rows of the other,
so X's lower half depends on Xhat's lower half alone, and scaling that by a power
of two scales it exactly (FP64 sums of products with exact zeros between).  Narrow
and wide X, in and out of place."""
import numpy as np
import pytest
import torch

from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ncols", [(600, 5), (600, 299), (600, 300), (600, 400), (300, 1100)])
def test_lower_half_scales_exactly(n, ncols):
    from paper_1708_06290_gb300 import ssv
    rng = np.random.default_rng(8100 + ncols)
    k, m = n // 2, 2
    A = np.zeros((n, n))
    A[:k, :k] = rng.standard_normal((k, k)) / np.sqrt(k) - 2 * np.eye(k)
    A[k:, k:] = rng.standard_normal((k, k)) / np.sqrt(k) - 2 * np.eye(k)
    B = np.zeros((n, m))
    B[:k] = rng.standard_normal((k, m))
    h = ssv.reduce(dev(A), dev(B), dev(rng.standard_normal((1, n))))
    x = rng.standard_normal((n, ncols)) + 1j * rng.standard_normal((n, ncols))
    y = x.copy()
    y[k:] *= 2.0 ** -30
    X = h.apply_q(dev(x, torch.complex128))
    Yd = dev(y, torch.complex128)
    Y = h.apply_q(Yd)
    assert torch.equal(Y[:k], X[:k])
    assert torch.equal(Y[k:], X[k:] * 2.0 ** -30)
    h.apply_q(Yd, out=Yd)
    assert torch.equal(Yd, Y)
    h.close()
