"""Level schedules of the FP32 / BF16 subdomain sweeps on boxes of 18^3 to 24^3 cells, where a
chunk of a few hundred cells is smaller than the widest levels: every candidate of the
autotuner gives the default schedule's values bit for bit (the schedule only says how far
ahead the factor records are staged). tests/test_apply_steps_cpu.py checks the same
schedules' tables on the host."""
import pytest
import torch

from oracle import discretization as disc
from paper_2007_13966_gb300 import autotune
from paper_2007_13966_gb300 import synthetic as syn

from gpu_util import dev, j_to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [32, 16])
@pytest.mark.parametrize("dims,parts,overlap", [((18, 18, 18), (1, 1, 1), 0), ((36, 36, 20), (2, 2, 1), 2),
                                                ((24, 24, 24), (1, 1, 1), 0), ((17, 40, 21), (1, 2, 1), 1)])
def test_small_chunks_give_the_default_values(dims, parts, overlap, prec):
    from paper_2007_13966_gb300 import ras
    res = syn.small_3d(*dims, seed=5)
    p = syn.random_pressure(res, 5)
    _, J = disc.residual(disc.Problem(res), p, 0.98 * p, 0.97 * p, res.dt, 2, want_jac=True)
    pc = ras.Precond(ras.Problem(res), parts, overlap, factor_prec=prec)
    pc.factor(j_to_dev(J))
    r = dev(syn.random_vector(res.grid.n, 2))
    z0, z = torch.zeros_like(r), torch.zeros_like(r)
    pc.apply(r, z0)
    for chunk in autotune.CHUNKS + (1,):
        pc.set_schedule(chunk, 0)
        assert pc.schedule()[0] >= chunk
        z.zero_()
        pc.apply(r, z)
        assert torch.equal(z, z0), chunk
    pc.factor(j_to_dev(J))                      # (no wait ran out)
