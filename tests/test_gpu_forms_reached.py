"""GPU tests of kernel forms at the edge of what reaches them: clusters with more generators than they
keep in shared memory, a key store that ends at the memory cap, arrangement bitmaps of directed sets and
without room for parent-edge tags.  Whole numbers: every comparison is exact."""

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


@pytest.mark.parametrize("n", [8, 9, 10])
def test_cluster_with_many_generators(cg, n):
    # 112, 168 and 240 three-cycles; 64 fit a block's shared memory
    jobs = [(n, w.three_cycles(n), True, -1), (n, w.three_cycles(n), True, 3)]
    with cg.Batch(jobs) as b:
        got = b.run()
        assert b.stats()["strategy_used"] == 4
    for j, r in zip(jobs, got):
        x = cg.growth(*j, strategy="hash")
        assert (r.layers, r.status) == (x.layers, x.status)


@pytest.mark.parametrize("radius", [8, 10, 11, 12])
def test_key_store_at_the_memory_cap(cg, radius):
    # S_13's bitmap takes 0.78 GB of 1.61: what the radius allows, or as far as the states fit
    n, gens = 13, w.inverse_closure(w.random_perms(np.random.default_rng(78), 13, 3))
    whole = cg.growth(n, gens, max_radius=radius, strategy="hash")
    cut = cg.growth(n, gens, max_radius=radius, strategy="bitmap", mem_cap=3 << 29)
    assert whole.status == 1
    assert cut.layers == whole.layers[:len(cut.layers)]
    assert cut.status == (1 if len(cut.layers) == len(whole.layers) else 2)
    fits = whole.total * 8 + 13 * 479001600 // 8 + (2 << 20) <= 3 << 29
    assert (cut.status == 1) == fits


@pytest.mark.parametrize("n,m", [(10, 4), (18, 9), (20, 12), (33, 4), (60, 2), (61, 3), (62, 60), (64, 3)])
@pytest.mark.parametrize("family", ["lx", "consecutive_4cycles", "coxeter"])
def test_binary_cosets_of_directed_sets(cg, n, m, family):
    start = np.random.default_rng(n * 100 + m).permutation([1] * m + [0] * (n - m)).tolist()
    gens = w.FAMILIES[family](n)
    with cg.Growth(n, gens, strategy="hash", start=start) as g:
        want, far, words = g.run(), np.sort(g.last_layer(), axis=0), g.key_words
    with cg.Growth(n, gens, start=start) as g:
        got = g.run()
        assert (got.status, got.layers) == (want.status, want.layers)
        assert np.array_equal(np.sort(g.last_layer(), axis=0), far)
        if words == 1:
            assert g.stats()["strategy_used"] == 3
