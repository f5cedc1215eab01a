"""Sweeps whose shifts are shared by the CTAs of a cluster (few shifts): the same
bits as with one CTA per shift, for every team size (1 to 15 shifts: eight CTAs,
to 31: four, to 76: two), every output mode and both arithmetics.  The sums of
a row do not depend on who forms them, so the comparison is exact; the solves
with one CTA per shift are compared with the oracle in the other tests.
"""
import numpy as np
import pytest
import torch

import workloads as W
from paper_1708_06290_gb300 import ssv
from tests.gpu_util import dev, shifts_dev

pytestmark = pytest.mark.gpu

MANY = 200


@pytest.mark.parametrize("n,m,p,nb", [(256, 4, 3, 0), (257, 5, 1, 16), (700, 2, 2, 0), (1030, 8, 20, 0),
                                      (1100, 16, 3, 0), (200, 20, 2, 0)])
def test_same_bits_for_every_team(n, m, p, nb):
    sysr = W.random_system(n, m, p, seed=9000 + n)
    h = ssv.reduce(dev(sysr.A), dev(sysr.B), dev(sysr.C))
    sig = 1j * np.logspace(-1, 1, MANY) + 0.1
    rng = np.random.default_rng(n)
    b = rng.standard_normal((m, MANY)) + 1j * rng.standard_normal((m, MANY))
    c = rng.standard_normal((p, MANY)) + 1j * rng.standard_normal((p, MANY))

    def runs(s):
        sd = shifts_dev(sig[:s])
        bd, cd = dev(b[:, :s], torch.complex128), dev(c[:, :s], torch.complex128)
        out = [h.solve(sd, mode=mode, precision=prec, nb=nb)[:2]
               for prec in ("fp64", "dfloat") for mode in ("g", "xhat")]
        out.append(h.solve_rhs(sd, bd, mode="xhat", nb=nb))
        out.append(h.solve_trans(sd, cd, mode="xhat", nb=nb))
        g, st, eta = h.solve(sd, mode="g", precision="fp64", nb=nb, want_resid=True)
        return out + [(g, st)], eta

    many, eta_many = runs(MANY)
    for s in (1, 15, 16, 31, 32, 76, 77):
        few, eta = runs(s)
        for (x, st), (y, _) in zip(few, many):
            assert (st.cpu().numpy() == 0).all()
            assert torch.equal(x, y[:, :x.shape[1]])
        assert float(eta.max()) <= 1e-14 and float(eta_many.max()) <= 1e-14
