"""The persistent batched subdomain solves (FP32 / BF16 factors) take boxes of different
reservoirs in turn in one CTA: each handle has its own shared-memory layout, so the record
ring of one box lies where the last one kept its vector and tables. Three reservoirs with
cubic, small and flat boxes, many more boxes than resident CTAs: each reservoir's FGMRES
iterates are those of a batch of itself alone, bit for bit, in either order (every sum of
the batched solver is taken per reservoir, in a fixed order)."""
import pytest
import torch

from oracle import discretization as disc
from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev, j_to_dev

pytestmark = pytest.mark.gpu

CASES = [((40, 40, 40), (2, 2, 2)), ((64, 64, 40), (10, 11, 8)), ((60, 50, 2), (4, 3, 1))]


@pytest.mark.parametrize("prec", [32, 16])
def test_each_reservoir_as_alone(prec):
    from paper_2007_13966_gb300 import ras
    items = []
    for i, (dims, parts) in enumerate(CASES):
        res = syn.small_3d(*dims, seed=20 + i)
        p = syn.random_pressure(res, 3)
        _, J = disc.residual(disc.Problem(res), p, 0.99 * p, 0.98 * p, res.dt, 2, want_jac=True)
        gp = ras.Problem(res)
        pc = ras.Precond(gp, parts, 1, factor_prec=prec)
        Jd = j_to_dev(J)
        pc.factor(Jd)
        items.append((gp, pc, Jd, dev(syn.random_vector(res.grid.n, 5))))

    def run(sel):
        bs = ras.BatchSolver([it[0] for it in sel], [it[1] for it in sel])
        xs = [torch.zeros_like(it[3]) for it in sel]
        for _ in range(3):
            bs.gmres([it[2] for it in sel], [it[3] for it in sel], xs, restart=5, maxit=5, rtol=1e-300)
        return xs

    alone = [run([it])[0] for it in items]
    assert all(torch.isfinite(x).all() for x in alone)
    for order in ([0, 1, 2], [2, 1, 0]):
        for i, x in zip(order, run([items[i] for i in order])):
            assert torch.equal(x, alone[i]), (order, i)
