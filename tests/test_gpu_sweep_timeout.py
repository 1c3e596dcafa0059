"""The bounded waits of the FP32 / BF16 subdomain sweeps: with a limit of one poll that the
factor records' copies cannot meet, the linear solve itself reports RAS_ETIMEOUT (single,
batched, one and two levels), a lone ras_apply's wait is reported by the next
factorisation, and with the normal limit the handle's next calls give a fresh handle's
values bit for bit. The limit only shortens the waits: every warp still runs to its end
and the copies that were started land before the block leaves."""
import os

import pytest
import torch

from oracle import discretization as disc
from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev, j_to_dev

pytestmark = pytest.mark.gpu

RAS_ETIMEOUT = -7


@pytest.fixture(scope="module")
def ras():
    from paper_2007_13966_gb300 import ras as R
    return R


@pytest.fixture
def one_poll(monkeypatch):
    class Limit:
        def __enter__(self):
            os.environ["RAS_BARRIER_POLLS"] = "1"

        def __exit__(self, *a):
            del os.environ["RAS_BARRIER_POLLS"]
    return Limit()


def _items(ras, prec, nlevels, dims=((40, 40, 24), (24, 20, 28))):
    out = []
    for i, d in enumerate(dims):
        res = syn.small_3d(*d, seed=40 + i)
        p = syn.random_pressure(res, 3)
        _, J = disc.residual(disc.Problem(res), p, 0.99 * p, 0.98 * p, res.dt, 2, want_jac=True)
        gp = ras.Problem(res)
        make = lambda gp=gp: ras.Precond(gp, (2, 2, 2), 1, factor_prec=prec, nlevels=nlevels, coarsen=(4, 4, 4),
                                         coarse_prec=32)
        out.append((gp, make, j_to_dev(J), dev(syn.random_vector(res.grid.n, 5))))
    return out


def _solve(gp, pc, J, b):
    x = torch.zeros_like(b)
    o = gp.gmres_solve(J, pc, b, x, restart=10, maxit=8, rtol=1e-300)
    assert o["iters"] == 8
    return x


@pytest.mark.parametrize("prec,nlevels", [(32, 1), (16, 1), (32, 2)])
def test_solve_reports_its_own_waits(ras, one_poll, prec, nlevels):
    gp, make, J, b = _items(ras, prec, nlevels)[0]
    pc = make()
    pc.factor(J)
    with one_poll, pytest.raises(ras.RasError) as e:
        _solve(gp, pc, J, b)
    assert e.value.status == RAS_ETIMEOUT
    torch.cuda.synchronize()                       # the context is still usable
    fresh = make()
    fresh.factor(J)
    ref = _solve(gp, fresh, J, b)
    assert torch.isfinite(ref).all()
    assert torch.equal(_solve(gp, pc, J, b), ref)  # nothing left set: no new factorisation needed
    pc.factor(J)
    assert torch.equal(_solve(gp, pc, J, b), ref)


def test_lone_apply_is_reported_once_by_the_next_factorisation(ras, one_poll):
    gp, make, J, b = _items(ras, 32, 1)[0]
    pc = make()
    pc.factor(J)
    z0, z = torch.zeros_like(b), torch.zeros_like(b)
    pc.apply(b, z0)
    with one_poll:
        pc.apply(b, z)
    with pytest.raises(ras.RasError) as e:
        pc.factor(J)
    assert e.value.status == RAS_ETIMEOUT
    pc.factor(J)
    pc.apply(b, z)
    assert torch.equal(z, z0)


@pytest.mark.parametrize("nlevels", [1, 2])
def test_batch_reports_its_waits(ras, one_poll, nlevels):
    items = _items(ras, 32, nlevels)
    pcs = [it[1]() for it in items]
    for it, pc in zip(items, pcs):
        pc.factor(it[2])

    def run(bs):
        xs = [torch.zeros_like(it[3]) for it in items]
        bs.gmres([it[2] for it in items], [it[3] for it in items], xs, restart=10, maxit=8, rtol=1e-300)
        return xs

    bs = ras.BatchSolver([it[0] for it in items], pcs)
    ref = run(bs)
    with one_poll, pytest.raises(ras.RasError) as e:
        run(bs)
    assert e.value.status == RAS_ETIMEOUT
    for x, y in zip(run(bs), ref):
        assert torch.equal(x, y)
