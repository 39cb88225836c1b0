"""GPU tests of the rank-bitmap kernels' byte-permute states: every n (their word layouts change at
8 and 12 elements), generators with and without parent edges, more generators than shared memory
holds, and both ways of probing the visited set.  Whole numbers: every comparison is exact."""

import numpy as np
import pytest

import oracle
import workloads as w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cg():
    import torch
    assert torch.cuda.is_available()
    import paper_2509_19162_gb300 as p
    p.build()
    return p


@pytest.mark.parametrize("n", range(2, 10))
@pytest.mark.parametrize("kind", ["random", "random_inv", "pancake"])
def test_bitmap_whole_growth_every_n(cg, n, kind):
    rng = np.random.default_rng(900 + n)
    gens = w.pancake(n) if kind == "pancake" else w.random_perms(rng, n, 2)
    if kind == "random_inv":
        gens = w.inverse_closure(gens)
    want, _ = oracle.growth(n, gens)
    assert cg.growth(n, gens, strategy="bitmap").layers == want
    start = rng.permutation(n).tolist()
    assert cg.growth(n, gens, strategy="bitmap", start=start).layers == want
    # several jobs in one launch: the kernel that learns n per job
    for r in cg.Batch([(n, gens, kind != "random", -1)] * 3, visited="bitmap").run():
        assert r.layers == want


@pytest.mark.parametrize("n,radius", [(10, 9), (11, 8), (12, 7), (13, 6), (14, 6)])
@pytest.mark.parametrize("kind", ["random", "random_inv", "pancake"])
def test_bitmap_against_hash_at_large_n(cg, n, radius, kind):
    rng = np.random.default_rng(950 + n)
    gens = w.pancake(n) if kind == "pancake" else w.random_perms(rng, n, 3)
    if kind == "random_inv":
        gens = w.inverse_closure(gens)
    want = cg.growth(n, gens, max_radius=radius, strategy="hash").layers
    assert cg.growth(n, gens, max_radius=radius, strategy="bitmap").layers == want


@pytest.mark.parametrize("n", [7, 8, 9])
def test_more_generators_than_shared_memory_holds(cg, n):
    # three-cycles: 70, 112 and 168 generators (64 fit), most without a parent-edge tag
    gens = w.three_cycles(n)
    want, _ = oracle.growth(n, gens)
    assert len(gens) > 64
    assert cg.growth(n, gens, strategy="bitmap").layers == want
    assert cg.Batch([(n, gens, True, -1)], visited="bitmap").run()[0].layers == want


@pytest.mark.parametrize("kind,radius", [("random_inv", 11), ("random", 16), ("pancake", 8)])
def test_key_store_grown_between_rounds(cg, kind, radius):
    # S_13's bitmap exceeds L2: one round per launch, the key store (2^24 states at first) grown
    # ahead of the layers that need it; the hash table grows by cutting a layer off and redoing it
    rng = np.random.default_rng(77)
    n = 13
    gens = w.pancake(n) if kind == "pancake" else w.random_perms(rng, n, 3)
    if kind == "random_inv":
        gens = w.inverse_closure(gens)
    with cg.Growth(n, gens, max_radius=radius, strategy="bitmap") as g:
        got = g.run()
        assert g.stats()["state_capacity"] >= got.total > 1 << 24
        assert g.run().layers == got.layers
    assert got.layers == cg.growth(n, gens, max_radius=radius, strategy="hash").layers


def test_key_store_growth_stops_at_the_memory_cap(cg):
    # the bitmap takes 0.78 GB; the cap leaves room for part of the layers only
    n, gens = 13, w.inverse_closure(w.random_perms(np.random.default_rng(78), 13, 3))
    whole = cg.growth(n, gens, max_radius=11, strategy="bitmap")
    cut = cg.growth(n, gens, max_radius=11, strategy="bitmap", mem_cap=3 << 29)
    assert cut.status == 0 or cut.layers == whole.layers[:len(cut.layers)]
    small = cg.growth(n, gens, max_radius=12, strategy="bitmap", mem_cap=3 << 29)
    assert small.status == 2 and small.layers == whole.layers[:len(small.layers)]
