"""The kernels of a single step on small lattices: plb_step(1), which no many-step launch takes over.  The
single pass against many steps in one launch, bit for bit, and after seven steps against the two-pass
kernels as in test_gpu_fused.py (bit for bit; D3Q19 FP32, which collides in another form, within its
bound), on the lattices of that file and on ragged ones of two and three x tiles, FP16 in both roundings."""
import numpy as np
import pytest

from gpu_cases import case_fields, make_lattice
from test_gpu_fused import CASES, RATES, _assert_same

pytestmark = pytest.mark.gpu

WALLS = dict(lattice=1, dims=(70, 20, 9), wall=True, shape="slab", mrt=True, rates=RATES, fext=(2e-6, 0, 0))
ALL = dict(CASES, ragged_fp16s=dict(WALLS, precision=2), ragged_fp16s_sr=dict(WALLS, precision=2, fp16_rounding=1),
           ragged_fp16s_bgk=dict(lattice=1, dims=(134, 19, 13), precision=2, u0=(0.02, -0.01, 0.015)),
           ragged_fp32_bgk=dict(lattice=1, dims=(134, 19, 13), precision=1, u0=(0.02, -0.01, 0.015)),
           ragged_fp16s_d2q9=dict(lattice=0, dims=(130, 37, 1), precision=2, fp16_rounding=1))


@pytest.mark.parametrize("name", list(ALL))
def test_single_pass_matches_the_two_pass_kernels(name):
    import paper_2504_15018_gb300 as plb
    case = ALL[name]
    rho, u0, rv, rl = case_fields(case)
    aa, fu, many = (make_lattice(dict(case, streaming=k), rv, rl) for k in (0, 1, 1))
    for lat in (aa, fu, many):
        lat.init(rho, u0)
    for _ in range(7):
        aa.step(1)
        fu.step(1)
    many.step(7)
    for lat in (aa, fu, many):
        lat.status()
    assert [plb.plb_launch_counts(x.h)["many_steps"] for x in (aa, fu, many)] == [0, 0, 7]
    assert np.array_equal(fu.populations(), many.populations())
    _assert_same(case, aa.populations(), fu.populations(), 7)
