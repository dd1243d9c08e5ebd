"""plb_step_pairs_static solves for the coexistence densities only where its options leave them to
the library: tau(rho) without densities and FP16 storage without rho_ref (solved), and both given
(not solved) step as the same lattice created by plb_create, bit for bit."""
import numpy as np
import pytest

from gpu_cases import maxwell
from paper_2504_15018_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("given", [False, True])
def test_default_and_given_densities(precision, given):
    import torch

    import paper_2504_15018_gb300 as plb
    rv, rl, _ = maxwell(0.8)
    dims, steps = (36, 29, 1), 4
    kw = dict(precision=precision, tau_v=1.2)
    if given:
        kw.update(tau_rho_v=0.9 * rv, tau_rho_l=0.9 * rl, rho_ref=0.5 * rv)
    opts = plb.make_opts(**kw)
    lat = plb.Lattice(plb.PLB_D2Q9, dims, plb.pr_eos(0.8), tau=0.8, opts=opts)
    lat.init(inputs.droplet(dims, (18.0, 14.0), 7.0, rv, rl, 3.0))
    dtype = torch.float32 if precision == 1 else torch.float16
    raw = lambda: torch.from_numpy(lat.get_state()[64:].copy()).view(dtype).reshape(lat.Q, -1)[:, :lat.n]
    pops = raw().cuda().contiguous()
    lat.step(steps)
    plb.plb_step_pairs_static(plb.PLB_D2Q9, dims, plb.pr_eos(0.8), 0.8, -1.0, 2.0, opts, pops.data_ptr(), steps // 2, 0,
                              torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(pops.cpu().numpy(), raw().numpy())
