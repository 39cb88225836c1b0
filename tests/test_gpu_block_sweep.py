"""GPU tests of the sweep strategy in blocks of states (n = 10..14): layers and last layer against
the key-list strategies and closed forms, from the identity and from other states, with limits, with
more generators than shared memory holds and for subgroups that fill half of every block.  Whole
numbers: every comparison is exact."""

import math

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


def gens_of(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "random":
        return w.random_perms(rng, n, 2)
    if kind == "random_inv":
        return w.inverse_closure(w.random_perms(rng, n, 2))
    if kind == "even":                  # three-cycles: A_n, half of every block's bits
        return w.cycles_01i_inv(n)
    return w.FAMILIES[kind](n)


@pytest.mark.parametrize("n", [10, 11])
@pytest.mark.parametrize("kind", ["lrx", "lx", "pancake", "random", "random_inv", "even", "star"])
def test_whole_growth_and_antipodes(cg, n, kind):
    gens = gens_of(kind, n, 40 + n)
    start = np.random.default_rng(n).permutation(n).tolist()
    with cg.Growth(n, gens, strategy="hash", start=start) as g:
        want, far = g.run(), np.sort(g.last_layer())
    for s in ("sweep", "auto"):
        with cg.Growth(n, gens, strategy=s, start=start) as g:
            for _ in range(2):          # a handle is run again
                got = g.run()
                assert (got.status, got.layers) == (want.status, want.layers)
                assert np.array_equal(np.sort(g.last_layer()), far)


@pytest.mark.parametrize("n,radius", [(12, 8), (13, 7), (14, 6)])
@pytest.mark.parametrize("kind", ["pancake", "random", "random_inv"])
def test_limited_growth_and_last_layer(cg, n, radius, kind):
    gens = gens_of(kind, n, 60 + n)
    with cg.Growth(n, gens, strategy="hash", max_radius=radius) as g:
        want, far = g.run(), np.sort(g.last_layer())
    with cg.Growth(n, gens, strategy="sweep", max_radius=radius) as g:
        got = g.run()
        assert (got.status, got.layers) == (want.status, want.layers)
        assert np.array_equal(np.sort(g.last_layer()), far)
    stop = want.layers[-2]
    r = cg.growth(n, gens, strategy="sweep", stop_above=stop - 1)
    assert r.status == 3 and r.layers == want.layers[:len(r.layers)] and r.layers[-1] >= stop


def test_mahonian_and_memory(cg):
    row = [1]
    for j in range(2, 13):              # inversions of S_12
        new = [0] * (len(row) + j - 1)
        for i, x in enumerate(row):
            for t in range(j):
                new[i + t] += x
        row = new
    assert cg.growth(12, w.coxeter(12)).layers == row
    # 1/4 GiB holds the three-bit sweep but not the blocks' four bits; the layers are the same
    assert cg.growth(12, w.coxeter(12), mem_cap=1 << 28).layers == row
    assert cg.growth(12, w.coxeter(12), strategy="sweep", mem_cap=1 << 28).layers == row


def test_more_generators_than_shared_memory_holds(cg):
    gens = w.three_cycles(10)           # 240
    got = cg.growth(10, gens, strategy="sweep")
    assert got.layers == cg.growth(10, gens, strategy="hash").layers
    assert sum(got.layers) == math.factorial(10) // 2


@pytest.mark.parametrize("n,kind,radius", [(11, "pancake", 9), (12, "coxeter", 24), (12, "lrx", 38),
                                           (12, "random_inv", 16), (12, "random", 27), (13, "pancake", 10)])
def test_radius_limited_growth_goes_on_in_blocks(cg, n, kind, radius):
    # the key list hands over to the blocks when the last layer is predicted to be dense
    gens = gens_of(kind, n, 80 + n)
    start = np.random.default_rng(n).permutation(n).tolist()
    with cg.Growth(n, gens, strategy="bitmap", max_radius=radius, start=start) as g:
        want, far = g.run(), np.sort(g.last_layer())
    with cg.Growth(n, gens, max_radius=radius, start=start) as g:
        for _ in range(2):
            got = g.run()
            assert g.stats()["strategy_used"] == 4 and g.stats()["launches"] > 3
            assert (got.status, got.layers) == (want.status, want.layers)
            assert np.array_equal(np.sort(g.last_layer()), far)


@pytest.mark.parametrize("n,kind,radius", [(11, "pancake", 5), (12, "lrx", 29), (13, "random_inv", 15), (12, "star", 6)])
def test_radius_limited_growth_that_stays_sparse(cg, n, kind, radius):
    gens = gens_of(kind, n, 80 + n)
    with cg.Growth(n, gens, strategy="hash", max_radius=radius) as g:
        want, far = g.run(), np.sort(g.last_layer())
    with cg.Growth(n, gens, max_radius=radius) as g:
        got = g.run()
        assert g.stats()["strategy_used"] == 3
        assert (got.status, got.layers) == (want.status, want.layers)
        assert np.array_equal(np.sort(g.last_layer()), far)


@pytest.mark.parametrize("kind,radius", [("pancake", 12), ("coxeter", 34), ("coxeter", 64)])
def test_served_job_over_its_share_keeps_its_layers(cg, kind, radius):
    # a served job that would store more states than its share holds stops there, in blocks as on the list
    n, share = 12, 1 << 30
    gens = w.FAMILIES[kind](n)
    want = cg.growth(n, gens, strategy="bitmap", max_radius=radius, mem_cap=share)
    from paper_2509_19162_gb300.serve import Server
    with Server(job_mem_cap=share) as s:
        i = s.submit(n, gens, max_radius=radius)
        while i not in s.finished():
            s.step()
        got = s.result(i)
    assert (got.status, got.layers) == (want.status, want.layers)


@pytest.mark.parametrize("n", range(2, 10))
@pytest.mark.parametrize("kind", ["random", "random_inv", "coxeter", "lx"])
def test_shared_memory_growth_every_small_n(cg, n, kind):
    gens = gens_of(kind, n, 20 + n) if n > 2 or kind in ("random", "random_inv") else [[1, 0]]
    start = np.random.default_rng(n).permutation(n).tolist()
    for lim in ({}, {"max_radius": 3}, {"stop_above": 4}):
        with cg.Growth(n, gens, strategy="hash", start=start, **lim) as g:
            want, far = g.run(), np.sort(g.last_layer())
        with cg.Growth(n, gens, start=start, **lim) as g:
            for _ in range(2):
                got = g.run()
                assert (got.status, got.layers) == (want.status, want.layers)
                assert np.array_equal(np.sort(g.last_layer()), far)


@pytest.mark.parametrize("cap", [1 << 20, 24 << 20, 0])
def test_batch_of_clusters(cg, cap):
    # n = 2..12 in one batch: a block each up to 8, a cluster each for 9 and 10, the rest as key lists;
    # with too little memory for clusters everything is a key list
    jobs = []
    for n in range(2, 13):
        for kind in ("random", "random_inv", "coxeter", "lx"):
            gens = gens_of(kind, n, 300 + n) if n > 2 or kind in ("random", "random_inv") else [[1, 0]]
            inv = kind in ("random_inv", "coxeter") or n == 2
            jobs.append((n, gens, inv, -1 if n <= 10 else 7))
            jobs.append((n, gens, inv, 5))
    with cg.Batch(jobs, mem_cap=cap) as b:
        first, again = b.run(), b.run()
    assert [(r.layers, r.status) for r in first] == [(r.layers, r.status) for r in again]
    for (n, gens, inv, rad), r in zip(jobs, first):
        want = cg.growth(n, gens, inv, rad, strategy="hash")
        if cap and r.status == 2:       # cut off by the batch's memory: exact so far
            assert r.layers == want.layers[:len(r.layers)]
        else:
            assert (r.layers, r.status) == (want.layers, want.status)


def test_batch_with_more_generators_than_shared_memory_holds(cg):
    gens = w.three_cycles(8)            # 112
    for r in cg.Batch([(8, gens, True, -1), (9, w.three_cycles(9), True, -1)]).run():
        assert r.status == 0
    assert cg.Batch([(8, gens, True, -1)]).run()[0].layers == cg.growth(8, gens, strategy="hash").layers
