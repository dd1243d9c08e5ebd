"""FP16 D3Q19 lattices whose rows are no multiple of 64 cell pairs: the in-place kernels, whose blocks then
hold several rows or narrower segments, against the many-step launch, which has tiles of its own and the
same per-cell arithmetic: equal bit for bit.  Rows of 9 pairs (the plain shape) to 200, a last group of
rows and a last segment that are not full, one row, one plane, chunks of planes, both kinds of walls."""
import numpy as np
import pytest

from gpu_cases import case_fields, make_lattice

pytestmark = pytest.mark.gpu

SIZES = [(18, 11, 4), (20, 13, 9), (34, 1, 5), (50, 7, 1), (94, 10, 17), (160, 9, 8), (162, 8, 6), (200, 12, 3),
         (288, 3, 4), (394, 5, 3), (400, 4, 2)]


@pytest.mark.parametrize("mrt,wall,wall_rho", [(False, False, 0.0), (True, True, 0.0), (True, True, 1.0)])
@pytest.mark.parametrize("rounding", [0, 1])
@pytest.mark.parametrize("dims", SIZES)
def test_rows_per_block_equal_tiles(dims, rounding, mrt, wall, wall_rho):
    rates = dict(s_e=1.19, s_eps=1.4, s_q=1.2, s_pi=1.3, s_m=1.5)
    case = dict(lattice=1, dims=dims, mrt=mrt, rates=rates, wall=wall, wall_rho=wall_rho, precision=2,
                fp16_rounding=rounding, shape="slab" if dims[1] >= 12 else "droplet", tau=0.8, tau_v=1.1,
                fext=(1e-6, 0, 0), u0=None if wall else (0.02, -0.01, 0.015))
    rho, u0, rv, rl = case_fields(case)
    rows, tiles = make_lattice(case, rv, rl), make_lattice(case, rv, rl)
    rows.init(rho, u0)
    tiles.init(rho, u0)
    for _ in range(6):
        rows.step(1)
    tiles.step(6)
    rows.status()
    a, b = rows.get_state()[64:].reshape(19, -1), tiles.get_state()[64:].reshape(19, -1)
    assert np.array_equal(a[:, :2 * rows.n], b[:, :2 * rows.n])
