"""A bounded wait that gives up inside the wide back-transform is reported: X is NaN,
shifts that were certified become non-finite with NaN backward errors, others keep
their status.  The error word is set from the host; nothing waits or stalls."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.gpu_util import dev, shifts_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,s", [(256, 4, 176), (400, 1, 2100)])
def test_a_wait_that_gave_up_is_reported(n, m, s):
    from paper_1708_06290_gb300 import ssv
    sysr = W.random_system(n, m, 1, seed=8300 + n)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    sd = shifts_dev(1j * np.logspace(-2, 2, s))
    xhat, st, eta = h.solve(sd, mode="xhat", precision="mixed", want_resid=True)
    X, stx, etax = h.solve(sd, mode="x", precision="mixed", want_resid=True)
    st[1], stx[1] = ssv.SHIFT_SINGULAR, ssv.SHIFT_SINGULAR
    Y, sty, etay = xhat.clone(), st.clone(), eta.clone()
    Y = ssv.colmajor(Y)
    # no wait gave up: the product of mode x, nothing else touched
    ssv.selftest_backtransform(h, Y, sty, etay)
    torch.cuda.synchronize()
    assert torch.equal(Y, X)
    assert torch.equal(sty, st) and torch.equal(etay, eta) and torch.equal(st, stx)
    # one did
    ssv.selftest_backtransform(h, Y, sty, etay, gave_up=True)
    torch.cuda.synchronize()
    assert torch.isnan(Y.real).all() and torch.isnan(Y.imag).all()
    assert torch.isnan(etay).all()
    want = torch.full_like(st, ssv.SHIFT_NONFINITE)
    want[1] = ssv.SHIFT_SINGULAR
    assert torch.equal(sty, want)
    ssv.selftest_backtransform(h, ssv.colmajor(xhat), gave_up=True)  # neither array
    torch.cuda.synchronize()
    h.close()
