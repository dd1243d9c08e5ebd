"""A long plb_step call on a small lattice is several launches of many steps, so that other streams' work
gets its turn, and ends in the populations of the same steps in short calls, bit for bit."""
import numpy as np
import pytest

from gpu_cases import case_fields, make_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,dims,precision,streaming,n", [
    (0, (8, 16, 1), 1, 0, 1205), (0, (8, 16, 1), 1, 1, 1205), (0, (256, 256, 1), 2, 0, 600),
    (1, (24, 20, 16), 0, 0, 604), (1, (48, 32, 32), 1, 1, 777)])
def test_long_calls_are_several_launches(lattice, dims, precision, streaming, n):
    import paper_2504_15018_gb300 as plb
    case = dict(lattice=lattice, dims=dims, precision=precision, streaming=streaming)
    rho, u0, rv, rl = case_fields(case)
    long, short = make_lattice(case, rv, rl), make_lattice(case, rv, rl)
    long.init(rho, u0)
    short.init(rho, u0)
    long.step(n)
    for k in range(0, n, 12):
        short.step(min(12, n - k))
    long.status()
    c = plb.plb_launch_counts(long.h)
    cell_steps = (1 << 21) if precision == 0 else (1 << 24)
    assert c["many_step_launches"] >= max(n / 512, n * long.n / cell_steps), c
    assert c["many_steps"] >= n - 1 and long.time == short.time == n
    assert np.array_equal(long.populations(), short.populations())
