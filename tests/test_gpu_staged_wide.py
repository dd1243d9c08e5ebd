"""FP16 D3Q19 lattices large enough for the wide shape of the staged kernel (blocks of several rows or of
narrower segments) to be chosen, against the many-step launch, which has tiles of its own: equal bit for
bit.  Two to ten rows a block with a last group that is not full, one to five segments with a last one
that is not full, 128 and 160 threads, a last chunk of one plane, walls of both kinds inside a block."""
import numpy as np
import pytest

from gpu_cases import case_fields, make_lattice

pytestmark = pytest.mark.gpu

SIZES = [(20, 41, 61), (22, 9, 300), (34, 41, 61), (66, 41, 61), (130, 13, 90), (130, 29, 61), (160, 13, 90),
         (288, 9, 90), (394, 41, 9)]


@pytest.mark.parametrize("rounding,mrt,wall,wall_rho", [(0, False, False, 0.0), (1, True, True, 0.0),
                                                        (0, True, True, 1.0), (1, False, False, 0.0)])
@pytest.mark.parametrize("dims", SIZES)
def test_wide_blocks_equal_tiles(dims, rounding, mrt, wall, wall_rho):
    import paper_2504_15018_gb300 as plb
    rates = dict(s_e=1.19, s_eps=1.4, s_q=1.2, s_pi=1.3, s_m=1.5)
    case = dict(lattice=1, dims=dims, mrt=mrt, rates=rates, wall=wall, wall_rho=wall_rho, precision=2,
                fp16_rounding=rounding, shape="slab", tau=0.9, tau_v=1.1, fext=(1e-6, 0, 0),
                u0=None if wall else (0.02, -0.01, 0.015))
    rho, u0, rv, rl = case_fields(case)
    rows, tiles = make_lattice(case, rv, rl), make_lattice(case, rv, rl)
    rows.init(rho, u0)
    tiles.init(rho, u0)
    for _ in range(6):
        rows.step(1)
    tiles.step(6)
    rows.status()
    assert [plb.plb_launch_counts(x.h)["many_steps"] for x in (rows, tiles)] == [0, 6]
    a, b = rows.get_state()[64:].reshape(19, -1), tiles.get_state()[64:].reshape(19, -1)
    assert np.array_equal(a[:, :2 * rows.n], b[:, :2 * rows.n])
