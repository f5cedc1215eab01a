"""Default block width of the sweeps: 64 rows below n = 1024, 128 from there on,
in FP64 and in double-float alike (128 rows double the typical error of a
double-float solution at n = 600).  The default gives the bits of the explicit
width, in ssv_solve and in the many-systems launch."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.gpu_util import dev, shifts_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nb", [(255, 64), (256, 64), (600, 64), (1023, 64), (1024, 128)])
@pytest.mark.parametrize("prec", ["fp64", "dfloat"])
def test_default_block_width(n, nb, prec):
    from paper_1708_06290_gb300 import ssv
    sysr = W.random_system(n, 4, 2, seed=6100 + n)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    sd = shifts_dev(np.concatenate([W.imag_axis_logspace(-2, 2, 3), [-1.7 + 0.4j]]))
    default = h.solve(sd, mode="xhat", precision=prec)[0]
    explicit = h.solve(sd, mode="xhat", precision=prec, nb=nb)[0]
    many = ssv.solve_many([h], [sd], mode="xhat", precision=prec)[0][0]
    torch.cuda.synchronize()
    assert torch.equal(default, explicit)
    assert torch.equal(default, many)
    h.close()
