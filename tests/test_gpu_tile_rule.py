"""Which small lattices and calls many-step launches take (sizes and steps on both sides of each line), and
that the largest of each kind end in the populations of single steps, bit for bit."""
import numpy as np
import pytest

from gpu_cases import case_fields, make_lattice

pytestmark = pytest.mark.gpu

RATES = dict(s_e=1.19, s_eps=1.4, s_q=1.2, s_pi=1.3, s_m=1.5)


def _lattices(lattice, dims, precision, streaming, count=1, **kw):
    case = dict(lattice=lattice, dims=dims, precision=precision, streaming=streaming, t_ratio=0.85, **kw)
    rho, u0, rv, rl = case_fields(case)
    lats = [make_lattice(case, rv, rl) for _ in range(count)]
    for lat in lats:
        lat.init(rho, u0)
    return lats


LINES = [(0, (512, 512, 1), 1, 0, True), (0, (512, 514, 1), 1, 0, False), (0, (409, 400, 1), 0, 0, True),
         (0, (410, 400, 1), 0, 0, False), (1, (24, 26, 26), 0, 0, True), (1, (26, 26, 26), 0, 0, False),
         (1, (60, 60, 62), 1, 0, True), (1, (62, 60, 62), 1, 0, False), (1, (49, 48, 48), 1, 0, True),
         (1, (51, 48, 48), 1, 0, False), (1, (51, 50, 51), 2, 0, True), (1, (53, 50, 51), 2, 0, False),
         (1, (64, 64, 64), 2, 0, True), (1, (66, 64, 64), 2, 0, False), (1, (64, 64, 64), 1, 1, True)]


@pytest.mark.parametrize("lattice,dims,precision,streaming,tiles", LINES)
def test_sizes(lattice, dims, precision, streaming, tiles):
    import paper_2504_15018_gb300 as plb
    lat, = _lattices(lattice, dims, precision, streaming)
    lat.step(20)
    lat.status()
    assert plb.plb_launch_counts(lat.h)["many_steps"] == (20 if tiles else 0)


@pytest.mark.parametrize("lattice,dims,precision,streaming,least", [
    (0, (256, 256, 1), 1, 0, 2), (0, (258, 256, 1), 1, 0, 4), (0, (416, 512, 1), 2, 0, 4), (0, (418, 512, 1), 1, 0, 6),
    (0, (181, 181, 1), 1, 0, 2), (0, (183, 181, 1), 1, 0, 4), (0, (511, 400, 1), 2, 0, 10), (0, (514, 256, 1), 1, 1, 2),
    (0, (362, 362, 1), 0, 0, 2), (1, (48, 48, 48), 1, 0, 4), (1, (50, 48, 48), 1, 0, 16), (1, (48, 48, 48), 2, 0, 2), (1, (16, 16, 16), 0, 0, 2)])
def test_steps_of_a_call(lattice, dims, precision, streaming, least):
    """From an even step and, in place, from an odd one (which takes one single step first)."""
    import paper_2504_15018_gb300 as plb
    lat, = _lattices(lattice, dims, precision, streaming)
    took = []
    for n in (least - 1, least):
        before = plb.plb_launch_counts(lat.h)["many_steps"]
        lat.step(n)
        took.append(plb.plb_launch_counts(lat.h)["many_steps"] - before)
        if lat.time % 2:
            lat.step(1)
    assert took == [0, least]
    if not streaming:
        lat.step(1)
        before = plb.plb_launch_counts(lat.h)["many_steps"]
        lat.step(least)
        assert plb.plb_launch_counts(lat.h)["many_steps"] == before
        lat.step(1 if lat.time % 2 == 0 else 2)
        lat.step(least + 1)
        assert plb.plb_launch_counts(lat.h)["many_steps"] == before + least
    lat.status()


@pytest.mark.parametrize("mrt", [False, True])
@pytest.mark.parametrize("lattice,dims,precision,streaming", [x[:4] for x in LINES if x[4]])
def test_largest_equal_single_steps(lattice, dims, precision, streaming, mrt):
    kw = dict(wall=True, shape="slab", mrt=True, rates=RATES, fext=(1e-6, 0, 0)) if mrt else dict(u0=(0.02, -0.01, 0.015))
    many, single = _lattices(lattice, dims, precision, streaming, 2, **kw)
    many.step(20)
    for _ in range(20):
        single.step(1)
    many.status()
    assert np.array_equal(many.populations(), single.populations())
