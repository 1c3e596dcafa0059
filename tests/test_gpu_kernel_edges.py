"""Kernels at the sizes where their index rules change: the 125-offset Galerkin product with
all offsets' boxes in shared memory and offset by offset (support boxes of 2 to 6 cells
per axis, cut at the boundary), the middle level's sweeps with and without room for guard
cells, the 7-point product on odd sizes and on arrays that are not 16-byte aligned, and
the orthogonalisation around its groups of columns. Tolerances as in the other parity
tests: V-cycle 1e-9 (FP64) and 5e-3 (FP32), product 1e-13, FGMRES histories 1e-9."""
import numpy as np
import pytest
import torch

from oracle import discretization as disc
from oracle import krylov, schwarz
from oracle import multilevel as ml
from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev, host, j_to_dev, rel_err

pytestmark = pytest.mark.gpu


def build(dims, seed=5):
    res = syn.small_3d(*dims, seed=seed)
    p = syn.random_pressure(res, seed)
    _, J = disc.residual(disc.Problem(res), p, 0.98 * p, 0.97 * p, res.dt, 2, want_jac=True)
    return res, J, disc.jacobian_csr(res.grid, J)


THREE = [((24, 20, 16), (2, 2, 2), 1, 1, (2, 2, 2)),
         ((27, 23, 9), (2, 2, 1), 1, 1, (3, 2, 1)),
         ((37, 30, 28), (2, 2, 2), 1, 1, (3, 3, 3)),
         ((160, 160, 3), (2, 2, 3), 0, 20, (2, 2, 1))]   # middle boxes of 60 x 60 x 3: no room for FP64 guard cells


@pytest.mark.parametrize("prec,tol,case", [(64, 1e-9, c) for c in range(4)] + [(32, 5e-3, c) for c in range(3)])
def test_three_level_forms(case, prec, tol):
    from paper_2007_13966_gb300 import ras
    dims, parts, ov, ov_c, ratios = THREE[case]
    res, J, A = build(dims)
    P1 = ml.interpolation(dims, ratios, 2)
    A1 = ml.galerkin(A, P1)
    d1 = ml.coarse_dims(dims, ratios)
    P0 = ml.interpolation(d1, ratios, 2)
    A0 = ml.galerkin(A1, P0)
    T = ml.MultiLevel([A0, A1, A], [None, schwarz.Schwarz(A1, d1, parts, ov_c, prec=prec),
                                    schwarz.Schwarz(A, dims, parts, ov, prec=prec)], [None, P0, P1], ml.DenseCoarse(A0))
    pc = ras.Precond(ras.Problem(res), parts, ov, factor_prec=prec, nlevels=3, coarsen=ratios, mlevel_type=0,
                     coarse_prec=prec, coarse_overlap=ov_c)
    pc.factor(j_to_dev(J))
    r = syn.random_vector(res.grid.n, 1)
    z = torch.full((res.grid.n,), np.nan, dtype=torch.float64, device="cuda")
    pc.apply(dev(r), z)
    assert rel_err(host(z), T(r)) < tol


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 1, 1), (5, 1, 1), (3, 2, 1), (7, 5, 3), (33, 9, 2), (16, 16, 2), (257, 3, 3)])
def test_product_sizes_and_alignment(dims, off):
    from paper_2007_13966_gb300 import ras
    res, J, A = build(dims)
    n = res.grid.n

    def shifted(v):
        t = torch.full((n + 2,), np.nan, dtype=torch.float64, device="cuda")
        t[off:off + n] = dev(v)
        return t, t[off:off + n]

    Js = [shifted(host(t)) for t in j_to_dev(J)]
    x = syn.random_vector(n, 3)
    xt, yt = shifted(x), shifted(np.zeros(n))
    ras.Problem(res).matvec([j[1] for j in Js], xt[1], yt[1])
    assert rel_err(host(yt[1]), A @ x) < 1e-13
    assert bool(torch.isnan(torch.cat([yt[0][:off], yt[0][off + n:]])).all())   # nothing written outside


@pytest.mark.parametrize("restart", [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32])
def test_orthogonalisation_columns(restart):
    from paper_2007_13966_gb300 import ras
    dims = (17, 13, 9)
    res = syn.small_3d(*dims, seed=21)
    g = res.grid
    p0 = np.full(g.n, res.p0)
    F, J = disc.residual(disc.Problem(res), syn.random_pressure(res, 9, 1.0, 3.0), p0, p0, res.dt, 1, want_jac=True)
    A = disc.jacobian_csr(g, J)
    M = schwarz.Schwarz(A, dims, (2, 2, 2), 1)
    hist = []
    krylov.fgmres(lambda v: A @ v, M, -F, rtol=1e-8, atol=0.0, restart=restart, maxit=restart, history=hist)
    gp = ras.Problem(res)
    pc = ras.Precond(gp, (2, 2, 2), 1, factor_prec=64)
    Jd = j_to_dev(J)
    pc.factor(Jd)
    x = torch.zeros(g.n, dtype=torch.float64, device="cuda")
    out = gp.gmres_solve(Jd, pc, dev(-F), x, restart=restart, maxit=restart, rtol=1e-8, atol=0.0)
    h, hist = np.array(out["history"]), np.array(hist)
    assert h.size == hist.size
    assert np.all(np.abs(h - hist) <= 1e-9 * hist + 1e-11 * hist[0])
