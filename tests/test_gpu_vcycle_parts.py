"""The two-level V-cycle (Eq. equ:v-cycle) against its parts, called one by one: the fine
subdomain solves (a one-level handle), the coarse correction (mlevel_type 4) and the
operator. Every sum is one FP64 addition per cell in both, so the accumulating forms inside
the V-cycle (z += P A_c^{-1} R t and the second fine solve's z += M t) give the parts' bits.
And the setting that ras_set_apply_kernel keeps: what it accepts and refuses."""
import pytest
import torch

from oracle import discretization as disc
from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev, j_to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [64, 32, 16])
@pytest.mark.parametrize("dims,parts,overlap", [((32, 32, 16), (2, 2, 1), 2), ((31, 33, 15), (2, 2, 2), 2),
                                                ((40, 25, 1), (3, 2, 1), 1)])
def test_vcycle_equals_its_parts(dims, parts, overlap, prec):
    from paper_2007_13966_gb300 import ras
    res = syn.small_3d(*dims, seed=3)
    p = syn.random_pressure(res, 5)
    _, J = disc.residual(disc.Problem(res), p, 0.98 * p, 0.97 * p, res.dt, 2, want_jac=True)
    gp, Jd = ras.Problem(res), j_to_dev(J)
    two = dict(nlevels=2, coarsen=(4, 4, 4 if dims[2] > 1 else 1), coarse_prec=64 if prec == 64 else 32)
    pcs = [ras.Precond(gp, parts, overlap, factor_prec=prec, **kw)
           for kw in (dict(two, mlevel_type=0), {}, dict(two, mlevel_type=4))]
    for pc in pcs:
        pc.factor(Jd)
    r = dev(syn.random_vector(res.grid.n, 6))
    z, e, c, y = (torch.zeros_like(r) for _ in range(4))
    pcs[0].apply(r, z)
    pcs[1].apply(r, e)
    gp.matvec(Jd, e, y)
    pcs[2].apply(r - y, c)
    e = e + c
    gp.matvec(Jd, e, y)
    pcs[1].apply(r - y, c)
    assert torch.equal(z, e + c)


def test_kernel_setting():
    from paper_2007_13966_gb300 import ras
    gp = ras.Problem(syn.small_3d(4, 40, 40, seed=1))
    ok = ras.Precond(gp, (1, 2, 2), 1, factor_prec=32)
    for k in (1, 0, 1):
        ok.set_apply_kernel(k)
        assert ok.apply_kernel() == k
    ok.set_schedule(2048, 0)
    assert ok.apply_kernel() == 1
    with pytest.raises(ras.RasError):
        ok.set_apply_kernel(2)
    for kw in (dict(factor_prec=64), dict(factor_prec=32, ras_type=0), dict(factor_prec=16, ras_type=2)):
        with pytest.raises(ras.RasError):
            ras.Precond(gp, (1, 2, 2), 1, **kw).set_apply_kernel(1)
    wide = ras.Precond(gp, (1, 1, 1), 0, factor_prec=32)          # 1,600 x-pencils
    with pytest.raises(ras.RasError):
        wide.set_apply_kernel(1)
    assert wide.apply_kernel() == 0
