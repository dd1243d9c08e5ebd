"""Density sums of FP32 lattices whose total leaves FP32's range, though no cell does: a thread that visits
two cells of density 2e38 adds them beyond 3.4e38.  Against the host's FP64 sum; a thread's terms are added
in FP64 then, two cells of 19 values, and the passes after it add 50 partials: 90 roundings, 2^-46."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,dims", [(1, (96, 83, 48)), (0, (700, 701, 1))])
@pytest.mark.parametrize("rho", [2e38, 1.0])
def test_sums_beyond_fp32(lattice, dims, rho):
    import paper_2504_15018_gb300 as plb
    lat = plb.Lattice(lattice, dims, plb.pr_eos(0.8), opts=plb.make_opts(precision=plb.PLB_FP32))
    _, w = plb.plb_velocity_set(lattice)
    f = np.repeat((rho * w[:, None]).astype(np.float32).astype(np.float64), lat.n, axis=1)
    lat.set_populations(f)
    total, bound = f.sum(), 2.0 ** -46
    assert abs(lat.reduce(plb.PLB_MEAN_RHO)[0] * lat.n - total) <= bound * total
    lo, hi = (1, 0, 0), dims
    part = total * (dims[0] - 1) / dims[0]
    assert abs(lat.reduce(plb.PLB_MASS, lo, hi)[0] - part) <= bound * part
