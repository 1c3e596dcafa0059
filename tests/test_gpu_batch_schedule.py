"""ras_set_apply_schedule on a handle that is in a batch: the batch takes the new schedule at
its next call (the launch settings, the handles' device tables and the captured cycles are
made again), and its results stay the same bit for bit."""
import pytest
import torch

from oracle import discretization as disc
from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev, j_to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nlevels", [(32, 1), (64, 1), (32, 2)])
def test_schedule_changes_between_calls(prec, nlevels):
    from paper_2007_13966_gb300 import ras
    items = []
    for i, d in enumerate([(40, 40, 20), (24, 20, 28), (30, 18, 18)]):
        res = syn.small_3d(*d, seed=40 + i)
        p = syn.random_pressure(res, 3)
        _, J = disc.residual(disc.Problem(res), p, 0.99 * p, 0.98 * p, res.dt, 2, want_jac=True)
        gp = ras.Problem(res)
        pc = ras.Precond(gp, (3, 3, 2), 1, factor_prec=prec, nlevels=nlevels, coarsen=(4, 4, 4), coarse_prec=prec)
        Jd = j_to_dev(J)
        pc.factor(Jd)
        items.append((gp, pc, Jd, dev(syn.random_vector(res.grid.n, 5))))
    bs = ras.BatchSolver([it[0] for it in items], [it[1] for it in items])

    def run():
        xs = [torch.zeros_like(it[3]) for it in items]
        bs.gmres([it[2] for it in items], [it[3] for it in items], xs, restart=6, maxit=9, rtol=1e-300)
        return xs

    ref = run()
    for which, chunk, threads in [((0,), 2048, 0), ((1, 2), 256, 256), ((0, 1, 2), 1, 0), ((0, 1, 2), 0, 0)]:
        try:
            for i in which:
                items[i][1].set_schedule(chunk, threads)
        except ras.RasError:
            assert prec == 64 and chunk == 2048        # beyond the shared memory of FP64 records
            continue
        for x, y in zip(run(), ref):
            assert torch.equal(x, y), (which, chunk, threads)
