"""The Peng-Robinson root (Section 2, Eq. equ:PR) just above the pressures where the vapour
root of a subcritical fluid meets the middle one and both disappear: one real root is left,
far from the start that the closed form in FP32 may give, and Newton from beside the lost
pair goes anywhere. Every state has an admissible root, and a finite residual and Jacobian."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import eos
from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev

pytestmark = pytest.mark.gpu


def _lost_pair(fluid, lo, hi):
    """The pressure in (lo, hi) at which the cubic's discriminant changes sign (extended precision)."""
    L = np.longdouble
    a, b = (L(v) for v in eos.pr_constants(fluid))

    def disc(p):
        A, B = eos.AB(p, a, b, fluid.R, fluid.T)
        c2, c1, c0 = -(1 - B), A - 3 * B * B - 2 * B, -(A * B - B * B - B ** 3)
        return 18 * c2 * c1 * c0 - 4 * c2 ** 3 * c0 + c2 * c2 * c1 * c1 - 4 * c1 ** 3 - 27 * c0 * c0
    lo, hi = L(lo), L(hi)
    s = np.sign(disc(lo))
    assert s != np.sign(disc(hi))
    for _ in range(90):
        m = (lo + hi) / 2
        lo, hi = (m, hi) if np.sign(disc(m)) == s else (lo, m)
    return float(hi)


@pytest.mark.parametrize("tr,lo,hi", [(0.7, 1.3e6, 1.6e6), (0.9, 2.9e6, 3.2e6), (0.95, 3.6e6, 3.8e6),
                                      (0.999, 4.5735e6, 4.58e6)])
def test_states_beside_the_lost_pair(tr, lo, hi):
    from paper_2007_13966_gb300 import ras
    fluid = syn.Fluid(T=190.6 * tr)
    r = _lost_pair(fluid, lo, hi)
    n = 1 << 20
    res = dataclasses.replace(syn.small_3d(n, 1, 1, seed=1), fluid=fluid)
    gp = ras.Problem(res)
    rng = np.random.default_rng(5)
    for _ in range(4):
        p = r * (1.0 + 10.0 ** -rng.uniform(2, 14, n))
        F = torch.zeros(n, dtype=torch.float64, device="cuda")
        q = dev(p)
        gp.residual_eval(q, 0.9 * q, 0.9 * q, res.dt, 1, F, gp.J, want_norm=True)   # (raises RAS_ENOROOT)
        assert torch.isfinite(F).all() and torch.isfinite(gp.J[0]).all()
