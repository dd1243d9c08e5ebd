"""The tiling that a batch starts with is one that plb_batch_configure can name and plb_batch_autotune
tries, also where a thread has one cell (FP64, odd widths)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,dims", [(0, (64, 40, 1)), (1, (65, 40, 1)), (1, (64, 40, 1)), (2, (301, 33, 1))])
def test_default_tiling_can_be_restored(precision, dims):
    import paper_2504_15018_gb300 as plb
    insts = [plb.make_instance(dims, plb.paper_eos(0.0375, 1.187, 0.044), opts=plb.make_opts(precision=precision))
             for _ in range(4)]
    b = plb.Batch(plb.PLB_D2Q9, insts)
    default = plb.plb_batch_split(b.b)["tiles"]
    b.configure(tile_cells=4096)
    assert plb.plb_batch_split(b.b)["tiles"] < default
    b.configure(tile_cells=512)
    assert plb.plb_batch_split(b.b)["tiles"] == default
