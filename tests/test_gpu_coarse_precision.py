"""The FP32 coarse correction (Section 3.2, the exact coarse solve with coarse_prec 32)
against the FP64 one of the same handle options: relative error over several reservoirs and
right-hand sides, geometric mean. The bounds are the errors measured with the 64 x 64 pivot
tiles (panels by FP32 multiply-adds) that the present block inverses replaced and must not
exceed: 50 x 50, 20 x 12 x 12 and 16 x 24 x 12 coarse cells (blocks of T = 128, 320 and
384, and so edge tiles of 128 rows and tiles partly beyond the block)."""
import math

import pytest
import torch

from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev

pytestmark = pytest.mark.gpu


def _reservoir(d, seed):
    if d[2] == 1:
        return syn.lognormal_reservoir(*d, 50.0, 50.0, 1.0, sigma=1.0, corr=4.0, seed_k=seed, seed_phi=seed + 1)
    return syn.lognormal_reservoir(*d, 25.0, 25.0, 5.0, sigma=1.0, corr=3.0, seed_k=seed, seed_phi=seed + 1)


@pytest.mark.parametrize("dims,ratio,count,bound", [((100, 100, 1), (2, 2, 1), 10, 1.30e-5),
                                                    ((40, 24, 24), (2, 2, 2), 8, 3.58e-5),
                                                    ((64, 96, 48), (4, 4, 4), 6, 5.14e-5)])
def test_no_further_from_fp64_than_the_tiles_replaced(dims, ratio, count, bound):
    from paper_2007_13966_gb300 import ras
    logs = []
    for s in range(count):
        seed = 100 + 10 * s
        res = _reservoir(dims, seed)
        gp = ras.Problem(res)
        p = dev(syn.random_pressure(res, seed))
        F = torch.zeros_like(p)
        gp.residual_eval(p, 0.99 * p, 0.98 * p, res.dt, 2, F, gp.J)
        vs = [-F] + [dev(syn.random_vector(res.grid.n, seed + 2 + q)) for q in range(3)]
        z = {}
        for prec in (64, 32):
            pc = ras.Precond(gp, tuple(-(-n // 16) for n in dims), 1, factor_prec=64, nlevels=2, coarsen=ratio,
                             coarse_prec=prec, mlevel_type=4)
            pc.factor(gp.J)
            z[prec] = [torch.zeros_like(v) for v in vs]
            for v, zz in zip(vs, z[prec]):
                pc.apply(v, zz)
        logs += [math.log(float((a - b).norm() / b.norm())) for a, b in zip(z[32], z[64])]
    assert math.exp(sum(logs) / len(logs)) < bound
