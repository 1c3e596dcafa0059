"""The FP64 reciprocal (recip64) against IEEE 1 / x, read through the subdomain solves: on a
diagonal operator with r = 1, z is the reciprocal of the diagonal. Within one unit in the
last place for values over FP64's range, of either sign, and on both sides of the limits
(1e-36 and 1e36) between its two forms."""
import numpy as np
import pytest
import torch

from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def _values(n):
    rng = np.random.default_rng(7)
    near = [s * x for c in (1e-36, 1e36) for x in (np.nextafter(c, 0), c, np.nextafter(c, np.inf), c * (1 - 1e-9),
                                                   c * (1 + 1e-9)) for s in (1.0, -1.0)]
    powers = [2.0 ** k for k in range(-130, 131)]
    edges = [m for k in (-100, -3, 0, 1, 60) for m in (np.nextafter(2.0 ** k, 0), np.nextafter(2.0 ** k, np.inf))]
    x = np.array(near + powers + edges)
    wide = 10.0 ** rng.uniform(-300, 300, n // 4) * rng.choice([-1.0, 1.0], n // 4)
    mid = 10.0 ** rng.uniform(-36.5, 36.5, n - x.size - wide.size) * rng.choice([-1.0, 1.0], n - x.size - wide.size)
    return np.concatenate([x, wide, mid])


def test_one_unit_in_the_last_place():
    from paper_2007_13966_gb300 import ras
    res = syn.small_3d(64, 64, 16, seed=1)
    N = res.grid.n
    x = _values(N)
    J = [dev(x)] + [dev(np.zeros(N)) for _ in range(6)]
    pc = ras.Precond(ras.Problem(res), (4, 4, 1), 0, factor_prec=64)
    pc.factor(J)
    z = torch.zeros(N, dtype=torch.float64, device="cuda")
    pc.apply(dev(np.ones(N)), z)
    ref = 1.0 / x
    assert (np.abs(host(z) - ref) <= np.abs(np.spacing(ref))).all()
