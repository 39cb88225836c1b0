"""GPU test of CG_OPT_ILP on rank bitmaps: every value that the option takes runs, in their one form."""

import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ilp", [0, 1, 2, 3, 4, 9, 10, 11, 12])
@pytest.mark.parametrize("strategy", ["bitmap", "auto", "hash", "sweep"])
def test_every_value_runs(ilp, strategy):
    import torch
    assert torch.cuda.is_available()
    import paper_2509_19162_gb300 as cg
    cg.build()
    n, gens = 9, w.lrx(9)
    want = cg.growth(n, gens).layers
    with cg.Growth(n, gens, strategy=strategy) as g:
        g.set_ilp(ilp)
        assert g.run().layers == want
        if strategy == "bitmap":
            assert g.stats()["probe_variant"] == 17
