"""The FP32 coarse correction (Section 3.2, the exact coarse solve with coarse_prec 32)
against the FP64 one of the same handle options: relative error over several reservoirs and
right-hand sides, geometric mean. The bounds are the errors measured with the 64 x 64 pivot
tiles (panels by FP32 multiply-adds) that the present block inverses replaced and must not
exceed: 50 x 50, 20 x 12 x 12 and 16 x 24 x 12 coarse cells (blocks of T = 128, 320 and
384, and so edge tiles of 128 rows and tiles partly beyond the block). The FP64 correction
the same against the oracle's operator, solved with residuals in extended precision, on
16^3 coarse cells (8 blocks of 512)."""
import math

import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as sla
import torch

from oracle import discretization as disc
from oracle import multilevel as ml
from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev, host, j_to_dev

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


def _refined(A, b):
    """A x = b in FP64 with residuals in extended precision."""
    A = sp.csr_matrix(A)
    A.sort_indices()
    lu = sla.splu(sp.csc_matrix(A))
    L = np.longdouble
    x, data = lu.solve(b).astype(L), A.data.astype(L)
    for _ in range(4):
        r = b.astype(L) - np.add.reduceat(data * x[A.indices], A.indptr[:-1])
        x = x + lu.solve(r.astype(np.float64))
    return x.astype(np.float64)


def test_fp64_sums_are_taken_apart():
    """Bound: 1.5 times the 2.03e-13 of the tiles replaced (single reservoirs 1.7e-13 to
    3.0e-13); with every term of an update rounded at the value's own size: 4.1e-13."""
    from paper_2007_13966_gb300 import ras
    dims, ratio, logs = (64, 64, 64), (4, 4, 4), []
    for seed in (5, 15, 25, 35):
        res = _reservoir(dims, seed)
        p = syn.random_pressure(res, seed)
        F, J = disc.residual(disc.Problem(res), p, 0.99 * p, 0.98 * p, res.dt, 2, want_jac=True)
        A, P = disc.jacobian_csr(res.grid, J), ml.interpolation(dims, ratio, 2)
        b = -np.asarray(F).ravel()
        ref = P @ _refined(P.T @ A @ P, P.T @ b)
        pc = ras.Precond(ras.Problem(res), (4, 4, 4), 1, factor_prec=64, nlevels=2, coarsen=ratio, coarse_prec=64,
                         mlevel_type=4)
        pc.factor(j_to_dev(J))
        z = torch.zeros(res.grid.n, dtype=torch.float64, device="cuda")
        pc.apply(dev(b), z)
        logs.append(math.log(np.linalg.norm(host(z) - ref) / np.linalg.norm(ref)))
    assert math.exp(sum(logs) / len(logs)) < 1.5 * 2.03e-13
