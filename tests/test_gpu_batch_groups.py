"""Batches larger than L2, whose instances are stepped group by group (a launch each), against lattices
stepped alone: equal bit for bit.  The instances are uneven, so groups and tiles end inside rows, and
the calls have odd and even step counts (parity and the step counter of the rounding noise cross the
groups)."""
import numpy as np
import pytest

from gpu_cases import maxwell
from paper_2504_15018_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,rounding,mrt,side,count", [(1, 0, False, 512, 12), (1, 0, True, 510, 12),
                                                               (2, 1, False, 512, 18), (0, 0, False, 317, 30)])
def test_groups_match_instances_stepped_alone(precision, rounding, mrt, side, count):
    import paper_2504_15018_gb300 as plb
    insts, fields = [], []
    for k in range(count):
        t = (0.75, 0.8, 0.85)[k % 3]
        rv, rl, _ = maxwell(t)
        dims = (side - 2 * (k % 5), side + k % 3, 1)
        opts = plb.make_opts(precision=precision, fp16_rounding=rounding, wall_y=k % 2, tau_v=1.1, tau_rho_v=rv,
                             tau_rho_l=rl, collision=plb.PLB_MRT if mrt else plb.PLB_BGK, s_e=1.19, s_eps=1.4, s_q=1.2)
        insts.append(plb.make_instance(dims, plb.pr_eos(t), tau=0.8, opts=opts))
        rho = inputs.droplet(dims, (dims[0] / 2, dims[1] / 2), side / 4, rv, rl, 3.0)
        fields.append(inputs.add_noise(rho, inputs.MASTER_SEED + 300 + k, 1e-4))
    b = plb.Batch(plb.PLB_D2Q9, insts)
    for k, rho in enumerate(fields):
        b.init(k, rho, None)
    for n in (3, 2, 3):
        b.step(n)
    b.status()
    for k in (0, count // 3, count // 2, count - 2, count - 1):
        lat = plb.Lattice(0, tuple(insts[k].dims), insts[k].eos, insts[k].tau, insts[k].G, insts[k].eps,
                          opts=insts[k].opts)
        lat.init(fields[k])
        lat.step(8)
        assert np.array_equal(b.populations(k), lat.populations()), k
