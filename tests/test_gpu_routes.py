"""Which kernels a call runs, so that tests that compare one path with another do compare two: the steps
that many-step launches take, the groups of a batch, and a batch whose blocks step more instances than
they keep descriptors of."""
import numpy as np
import pytest

from gpu_cases import case_fields, make_lattice, maxwell
from paper_2504_15018_gb300 import inputs
from test_gpu_tiles import SIZES

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,streaming", [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1)])
@pytest.mark.parametrize("name", [n for n in SIZES if not n.endswith("largest")])
def test_steps_taken_by_many_step_launches(name, precision, streaming):
    import paper_2504_15018_gb300 as plb
    lattice, dims = SIZES[name]
    if streaming and dims[0] % 2:
        pytest.skip("the single pass needs an even nx")
    case = dict(lattice=lattice, dims=dims, precision=precision, streaming=streaming, shape="slab")
    rho, _, rv, rl = case_fields(case)
    lat = make_lattice(case, rv, rl)
    lat.init(rho)
    for _ in range(3):
        lat.step(1)
    assert plb.plb_launch_counts(lat.h) == {"many_step_launches": 0, "many_steps": 0}
    lat.step(1)
    lat.step(20)
    assert plb.plb_launch_counts(lat.h)["many_steps"] == 20
    lat.status()


@pytest.mark.parametrize("precision,side,count", [(1, 512, 12), (1, 510, 12), (2, 512, 18), (0, 317, 30)])
def test_large_batches_have_groups(precision, side, count):
    """The batches that test_gpu_batch_groups.py steps; and one that has a single group."""
    import paper_2504_15018_gb300 as plb
    insts = [plb.make_instance((side - 2 * (k % 5), side + k % 3, 1), plb.paper_eos(0.0375, 1.187, 0.044),
                               opts=plb.make_opts(precision=precision)) for k in range(count)]
    assert plb.plb_batch_split(plb.Batch(plb.PLB_D2Q9, insts).b)["groups"] >= 2
    assert plb.plb_batch_split(plb.Batch(plb.PLB_D2Q9, insts[:2]).b)["groups"] == 1


@pytest.mark.parametrize("precision,rounding", [(1, 0), (2, 1), (0, 0)])
def test_blocks_with_many_instances(precision, rounding):
    """More than four instances (one tile each) per block, whose descriptors a block loads four at a time."""
    import torch

    import paper_2504_15018_gb300 as plb
    rv, rl = 0.0375, 1.187
    count = 6 * torch.cuda.get_device_properties(0).multi_processor_count + 5
    insts, fields = [], []
    for k in range(count):
        dims = (8 + k % 3, 6 + k % 4, 1)
        opts = plb.make_opts(precision=precision, fp16_rounding=rounding, wall_y=k % 2)
        insts.append(plb.make_instance(dims, plb.paper_eos(rv, rl, 0.044), tau=0.6 + 0.01 * (k % 7), opts=opts))
        rho = inputs.droplet(dims, (4.0, 3.0), 2.0, rv, rl, 3.0)
        fields.append(inputs.add_noise(rho, inputs.MASTER_SEED + 400 + k, 1e-3))
    b = plb.Batch(plb.PLB_D2Q9, insts)
    b.configure(blocks_per_sm=1)
    assert plb.plb_batch_split(b.b) == {"tiles": count, "groups": 1}
    for k, rho in enumerate(fields):
        b.init(k, rho, None)
    b.step(3)
    b.step(4)
    b.status()
    for k in list(range(14)) + list(range(count - 14, count)) + list(range(20, count, 97)):
        lat = plb.Lattice(0, tuple(insts[k].dims), insts[k].eos, insts[k].tau, insts[k].G, insts[k].eps,
                          opts=insts[k].opts)
        lat.init(fields[k])
        for _ in range(7):
            lat.step(1)
        assert np.array_equal(b.populations(k), lat.populations()), k
