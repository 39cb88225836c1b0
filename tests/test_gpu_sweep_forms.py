"""GPU tests of which form of the sweep runs -- in blocks of states or state by state -- beyond L2
(n = 13, 14), where the limits or the memory cap decide it, and of the state-by-state form at those n
with the automatic order.  Whole numbers: every comparison is exact."""

import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cg():
    import torch
    assert torch.cuda.is_available()
    import paper_2509_19162_gb300 as p
    p.build()
    return p


@pytest.mark.parametrize("n,k,kw,blocks", [
    (13, "pancake", {"max_radius": 4}, False), (13, "pancake", {"max_radius": 5}, True),
    (13, 4, {"stop_above": 1 << 14}, False), (13, 4, {"stop_above": 1 << 18}, True),
    (14, "pancake", {"max_radius": 6}, False), (14, 4, {"stop_above": 1 << 20}, False),
    (14, 4, {"max_radius": 9, "stop_above": 1 << 30}, False), (14, 4, {"stop_above": 1 << 25}, True),
    (12, "pancake", {"max_radius": 3}, True),
])
def test_limited_sweep(cg, n, k, kw, blocks):
    gens = w.pancake(n) if k == "pancake" else w.inverse_closure(w.random_perms(np.random.default_rng(n), n, 2))
    start = np.random.default_rng(n + 1).permutation(n).tolist()
    with cg.Growth(n, gens, strategy="hash", start=start, **kw) as g:
        want, far = g.run(), np.sort(g.last_layer())
    with cg.Growth(n, gens, strategy="sweep", start=start, **kw) as g:
        for _ in range(2):
            got = g.run()
            assert (got.status, got.layers) == (want.status, want.layers)
            assert np.array_equal(np.sort(g.last_layer()), far)
        assert g.stats()["probe_variant"] == (1 if blocks else 2)


def test_small_group_in_a_large_symmetric_group(cg):
    # 10! of 14! elements, whole
    gens = [list(g) + list(range(10, 14)) for g in w.lrx(10)]
    with cg.Growth(14, gens, strategy="sweep") as g:
        assert g.run().layers == cg.growth(10, w.lrx(10)).layers
        assert g.stats()["probe_variant"] == 2


def test_whole_s13_with_three_bits(cg):
    # 2.6 GB hold three bits an element of S_13 (2.4 GB) but not four (3.1 GB): state by state, dense layers
    # in rank order
    want = cg.growth(13, w.lrx(13)).layers
    with cg.Growth(13, w.lrx(13), strategy="sweep", mem_cap=2_600_000_000) as g:
        got = g.run()
        assert got.status == 0 and got.layers == want
        assert g.stats()["probe_variant"] == 2
