"""The bounded waits of many-step launches: one that runs out ends in PLB_ETIMEOUT, every block returns,
steps after it change nothing until the populations are replaced, and plb_init, plb_set_state and
plb_set_populations each bring the lattice back: it then steps as one that never failed, bit for bit."""
import numpy as np
import pytest

from gpu_cases import case_fields, make_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recover", ["init", "set_state", "set_populations"])
@pytest.mark.parametrize("lattice,dims,precision,streaming", [(0, (256, 96, 1), 1, 0), (0, (98, 60, 1), 1, 1),
                                                              (1, (24, 20, 18), 2, 0), (1, (12, 10, 9), 0, 0)])
def test_a_wait_that_runs_out(lattice, dims, precision, streaming, recover):
    import paper_2504_15018_gb300 as plb
    case = dict(lattice=lattice, dims=dims, precision=precision, streaming=streaming)
    rho, u0, rv, rl = case_fields(case)
    lat, ref = make_lattice(case, rv, rl), make_lattice(case, rv, rl)
    for x in (lat, ref):
        x.init(rho, u0)
        x.step(4)
    state, pops = lat.get_state(), lat.populations()
    plb.plb_withhold_counts(lat.h, 2000)
    lat.step(10)
    with pytest.raises(plb.PlbError) as e:
        lat.status()
    assert e.value.code == plb.PLB_ETIMEOUT
    before = lat.populations()
    lat.step(10)
    with pytest.raises(plb.PlbError) as e:
        lat.status()
    assert e.value.code == plb.PLB_ETIMEOUT
    assert np.array_equal(lat.populations(), before, equal_nan=True)
    if recover == "init":
        lat.init(rho, u0)
        lat.step(4)
    elif recover == "set_state":
        lat.set_state(state)
    else:
        lat.set_populations(pops)
    lat.status()
    lat.step(10)
    ref.step(10)
    lat.status()
    assert plb.plb_launch_counts(lat.h)["many_steps"] >= 24
    assert np.array_equal(lat.populations(), ref.populations())
