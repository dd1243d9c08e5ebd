"""Reductions of FP32 and FP16-shifted lattices (sums in error-free FP32 parts, the speed maximum by
candidates) against the same quantities cell by cell: the stored populations summed on the host with
math.fsum, and one-cell boxes of the library for momentum and speed, whose force term the host lacks.

Bounds.  A thread's sum is exact to FP64 rounding; the block and final passes add at most 8 + 5 + 32 + 5
partials in FP64, so sums of terms x are within 2^-47 of sum |x|.  The speed maximum is the FP64 value
of a cell whose speed is within 2^-40 of the largest.  FP32 moments sum 19 values: 20 x 2^-24."""
import math

import numpy as np
import pytest

from gpu_cases import case_fields, make_lattice

pytestmark = pytest.mark.gpu

SIZES = {"d2q9_odd": (0, (37, 11, 1)), "d2q9_one_row": (0, (66, 1, 1)), "d3q19_odd": (1, (9, 7, 5)),
         "d3q19_even": (1, (10, 6, 6)), "more_cells_than_threads": (1, (96, 83, 48))}


@pytest.mark.parametrize("steps", [4, 5])
@pytest.mark.parametrize("precision,wall,moving", [(1, False, True), (1, True, False), (2, False, True)])
@pytest.mark.parametrize("name", list(SIZES))
def test_reductions_equal_cell_sums(name, precision, wall, moving, steps):
    import paper_2504_15018_gb300 as plb
    lattice, dims = SIZES[name]
    case = dict(lattice=lattice, dims=dims, wall=wall, precision=precision, tau=0.9, fext=(1e-6, 0, 0),
                u0=(0.02, -0.01, 0.015) if moving else None)
    rho0, u0, rv, rl = case_fields(case)
    lat = make_lattice(case, rv, rl)
    lat.init(rho0, u0)
    lat.step(steps)
    f = lat.populations()
    nx, ny, nz = dims
    mean = lat.reduce(plb.PLB_MEAN_RHO)[0]           # (the whole-lattice mass has a kernel of its own)
    assert abs(mean * lat.n - math.fsum(f.ravel())) <= 2.0 ** -47 * np.abs(f).sum()
    lo, hi = (nx // 3, 0, nz // 2), (nx - 1, max(1, ny // 2), nz)
    cube = f.reshape(-1, nz, ny, nx)[:, lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
    assert abs(lat.reduce(plb.PLB_MASS, lo, hi)[0] - math.fsum(cube.ravel())) <= 2.0 ** -47 * np.abs(cube).sum()
    mom, umax = np.array(lat.reduce(plb.PLB_MOMENTUM)[:3]), lat.reduce(plb.PLB_UMAX)[0]
    rho, u, _ = lat.moments()
    speed = np.sqrt((u ** 2).sum(0))
    eps = 20 * 2.0 ** -24
    assert abs(umax - speed.max()) <= 2 * eps * (1 + speed.max())
    if name != "more_cells_than_threads":
        cells = [((x, y, z), (x + 1, y + 1, z + 1)) for z in range(nz) for y in range(ny) for x in range(nx)]
        ms = np.array([lat.reduce(plb.PLB_MOMENTUM, *c)[:3] for c in cells])
        assert np.all(np.abs(ms[:, :lat.D] - (rho * u).T) <= 2 * eps * np.abs(f).sum(0)[:, None])
        for a in range(lat.D):
            assert abs(mom[a] - math.fsum(ms[:, a])) <= 2.0 ** -47 * np.abs(ms[:, a]).sum()
        best = max(lat.reduce(plb.PLB_UMAX, *c)[0] for c in cells)
        assert abs(umax - best) <= 2.0 ** -40 * best
    else:
        assert np.all(np.abs(mom[:lat.D] - (rho * u).sum(1)) <= 2 * eps * np.abs(f).sum())
    lat.status()
