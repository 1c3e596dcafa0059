"""Coarse operators with a zero or small diagonal inside a 4 x 4 pivot block (Section 3.2,
the exact coarse solve): piecewise-constant interpolation (interp_order 1) of a 4-cell line
whose pairs of cells cancel gives A_c = [[e, h], [h, e]]. The FP32 elimination takes the
block whatever e is, 0 and 2^-16 beside h = 1/2 among them; the FP64 one, whose pivots are
single values, refuses e = 0 with RAS_EZEROPIVOT and takes the rest. A singular block is
refused by both."""
import numpy as np
import pytest
import torch

from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev, host

pytestmark = pytest.mark.gpu

RAS_EZEROPIVOT = -5


def _line(e, h):
    """J (centre, -x, +x, -y, +y, -z, +z) of the line: pairs (0, 1), (2, 3) sum to e, couplings h between them."""
    J = [dev(np.zeros(4)) for _ in range(7)]
    J[0][:] = 1.0
    J[2][0] = J[2][2] = -2.0 + e           # a01, a23 (a10 = a32 = 0)
    J[2][1] = J[1][2] = h                  # a12, a21
    return J


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("e,h", [(0.0, 0.5), (2.0 ** -16, 0.5), (2.0 ** -3, 0.5), (0.75, 0.5), (0.5, 0.5)])
def test_two_by_two(prec, e, h):
    from paper_2007_13966_gb300 import ras
    gp = ras.Problem(syn.small_3d(4, 1, 1, seed=1))
    pc = ras.Precond(gp, (1, 1, 1), 0, factor_prec=64, nlevels=2, coarsen=(2, 1, 1), coarse_prec=prec,
                     interp_order=1, mlevel_type=4)
    J = _line(e, h)
    if e == h or (e == 0.0 and prec == 64):
        with pytest.raises(ras.RasError) as err:
            pc.factor(J)
        assert err.value.status == RAS_EZEROPIVOT
        return
    pc.factor(J)
    r = np.array([1.0, 0.5, -0.25, 2.0])
    z = torch.zeros(4, dtype=torch.float64, device="cuda")
    pc.apply(dev(r), z)
    x = np.linalg.solve(np.array([[e, h], [h, e]]), np.array([r[0] + r[1], r[2] + r[3]]))
    # condition number (h + e) / (h - e) <= 5, a few roundings of the elimination
    assert np.abs(host(z) - np.repeat(x, 2)).max() <= (1e-5 if prec == 32 else 1e-13) * np.abs(x).max()
