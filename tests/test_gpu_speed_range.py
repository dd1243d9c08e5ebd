"""The largest speed (PLB_UMAX) of FP32 lattices against the speed of single cells in FP64 (PLB_UL1 of a
one-cell box, which sums one FP64 speed): densities and momenta whose squares leave FP32's range, one
such cell in an ordinary field, and, where a thread visits two cells, pairs of cells whose speeds differ by
less than FP32 pairs resolve, cells equal in every bit, and cells at rest.

Bound: both evaluate the same FP64 expression (19 additions, 3 products, a quotient, a root) of the cell of
the largest speed; 2^-48 covers a different order or contraction of them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BOUND = 2.0 ** -48


def _lattice(lattice, dims):
    import paper_2504_15018_gb300 as plb
    return plb.Lattice(lattice, dims, plb.pr_eos(0.8), opts=plb.make_opts(precision=plb.PLB_FP32))


def _cell_speed(lat, s):
    import paper_2504_15018_gb300 as plb
    nx, ny, _ = lat.dims
    c = (s % nx, s // nx % ny, s // (nx * ny))
    return lat.reduce(plb.PLB_UL1, c, tuple(v + 1 for v in c))[0]


def _weights(lattice):
    import paper_2504_15018_gb300 as plb
    return plb.plb_velocity_set(lattice)


FIELDS = {"1e12": 1e12, "1": 1.0, "1e-18": 1e-18, "1e-23": 1e-23, "3e-23": 3e-23, "1e-30": 1e-30, "1e-37": 1e-37}


@pytest.mark.parametrize("one", ["none", "momentum_1e11", "density_1e-30"])
@pytest.mark.parametrize("name", list(FIELDS))
@pytest.mark.parametrize("lattice,dims", [(0, (7, 6, 1)), (1, (5, 4, 3))])
def test_any_density(lattice, dims, name, one):
    import paper_2504_15018_gb300 as plb
    if one == "momentum_1e11" and name == "1e12":
        pytest.skip("nothing out of the ordinary")
    lat = _lattice(lattice, dims)
    c, w = _weights(lattice)
    rng = np.random.RandomState(5)
    u = 0.05 * rng.uniform(-1, 1, (3, lat.n))
    if lattice == 0:
        u[2] = 0
    rho = FIELDS[name] * rng.uniform(0.9, 1.1, lat.n)
    if one == "momentum_1e11":
        rho[lat.n // 2], u[0, lat.n // 2] = 1e12, 0.1
    if one == "density_1e-30":
        rho[lat.n // 2], u[0, lat.n // 2] = 1e-30, 0.3
    f = w[:, None] * rho * (1 + 3 * (c @ u))
    lat.set_populations(f)
    got = lat.reduce(plb.PLB_UMAX)[0]
    want = max(_cell_speed(lat, s) for s in range(lat.n))
    assert want > 0.01
    assert abs(got - want) <= BOUND * want, (got, want)


# more cells than the reduction has threads (1024 blocks of 256): cells s and s + 2^18 are one thread's
DIMS, STRIDE = (96, 83, 48), 1 << 18


@pytest.mark.parametrize("bits", [20, 30, 34, 36, 38, 40, 42, 46])
@pytest.mark.parametrize("second", [False, True])
def test_cells_closer_than_pairs_resolve(bits, second):
    import paper_2504_15018_gb300 as plb
    lat = _lattice(1, DIMS)
    c, w = _weights(1)
    f = np.repeat(w[:, None], lat.n, axis=1)
    s0 = 5000
    cells = [s0, s0 + STRIDE]
    plus = [i for i, v in enumerate(c.tolist()) if v[0] == 1]
    for s in cells:
        f[plus[0], s] += 0.125
    f[plus[1], cells[int(second)]] = 0.0            # make room for a small term beside the other 18
    f[plus[1], cells[1 - int(second)]] = 0.0
    f[plus[1], cells[int(second)]] = 2.0 ** -bits
    lat.set_populations(f)
    got = lat.reduce(plb.PLB_UMAX)[0]
    want = max(_cell_speed(lat, s) for s in cells)
    assert want > 0.05
    assert abs(got - want) <= BOUND * want, (got, want)


@pytest.mark.parametrize("speed", [0.0, 0.07])
def test_uniform_fields(speed):
    import paper_2504_15018_gb300 as plb
    lat = _lattice(1, DIMS)
    u = np.zeros((3, lat.n))
    u[0], u[2] = speed, -0.5 * speed
    lat.init(np.full(lat.n, 7.0), u)
    got, want = lat.reduce(plb.PLB_UMAX)[0], _cell_speed(lat, 12345)
    assert abs(got - want) <= BOUND * want and (want > 0) == (speed > 0), (got, want)
