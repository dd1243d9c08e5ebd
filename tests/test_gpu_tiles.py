"""Many steps in one launch (small lattices): plb_step(n) against n calls of plb_step(1), which run
the per-step kernels.  The tiles run the same per-cell arithmetic on the same inputs, so the stored
populations are equal bit for bit; lattices at the edges of the split (one tile, tiles of two rows,
ragged last tiles, one row, two columns, one plane), both cell paths (even and odd nx), every
storage, walls of both kinds and both stepping modes."""
import numpy as np
import pytest

from gpu_cases import case_fields, make_lattice

pytestmark = pytest.mark.gpu

RATES = dict(s_e=1.19, s_eps=1.4, s_q=1.2, s_pi=1.3, s_m=1.5)
SIZES = {
    "d2q9_planar": (0, (8, 256, 1)), "d2q9_one_tile": (0, (6, 5, 1)), "d2q9_two_wide": (0, (2, 17, 1)),
    "d2q9_one_row": (0, (66, 1, 1)), "d2q9_odd": (0, (37, 29, 1)), "d2q9_ragged": (0, (98, 305, 1)),
    "d2q9_remainder_of_one": (0, (33, 40, 1)), "d2q9_largest": (0, (512, 512, 1)),
    "d3q19_even": (1, (34, 18, 12)), "d3q19_odd": (1, (13, 11, 9)), "d3q19_one_plane": (1, (18, 10, 1)),
    "d3q19_two": (1, (2, 2, 2)), "d3q19_largest": (1, (64, 64, 64)),
}


def _stored(lat):
    """The raw populations of the cells (the planes of the store are padded)."""
    raw = lat.get_state()[64:].reshape(lat.Q, -1)
    return raw[:, :lat.n * {0: 8, 1: 4, 2: 2}[int(lat.opts.precision)]]


@pytest.mark.parametrize("mrt,wall,wall_rho", [(False, False, 0.0), (True, True, 0.0), (True, True, 1.0)])
@pytest.mark.parametrize("precision,rounding,streaming", [(0, 0, 0), (1, 0, 0), (1, 0, 1), (2, 0, 0), (2, 1, 1)])
@pytest.mark.parametrize("name", list(SIZES))
def test_many_steps_equal_single_steps(name, precision, rounding, streaming, mrt, wall, wall_rho):
    lattice, dims = SIZES[name]
    if streaming and dims[0] % 2:
        pytest.skip("the single pass needs an even nx")
    case = dict(lattice=lattice, dims=dims, mrt=mrt, rates=RATES, wall=wall, wall_rho=wall_rho, precision=precision,
                fp16_rounding=rounding, streaming=streaming, shape="slab" if dims[1] >= 12 else "droplet",
                tau=0.8, tau_v=1.1, fext=(1e-6, 0, 0), u0=None if wall else (0.02, -0.01, 0.015))
    rho, u0, rv, rl = case_fields(case)
    many, single = make_lattice(case, rv, rl), make_lattice(case, rv, rl)
    many.init(rho, u0)
    single.init(rho, u0)
    for n in (6, 1, 5, 2):                 # even, then from an odd step, then an even number again
        many.step(n)
        for _ in range(n):
            single.step(1)
        many.status()
        assert many.time == single.time
        assert np.array_equal(_stored(many), _stored(single)), n
