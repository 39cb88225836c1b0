"""GPU tests of launches that grow several jobs of n = 11 and more together: jobs whose generators just
fit a warp's shared memory beside others that leave it to staged states, rank bitmaps beside hash
tables, layers that are mostly new and layers that are mostly found.  Whole numbers: every comparison
is exact."""

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


def pairs(n, k, seed):
    """k generators closed under inverses, none its own."""
    gens, rng = [], np.random.default_rng(seed)
    while len(gens) < k:
        p = rng.permutation(n).tolist()
        q = w.inverse(p)
        if p != q and p not in gens:
            gens += [p, list(q)]
    return gens


@pytest.mark.parametrize("ks", [(4, 46, 10), (48, 4, 2), (9, 11, 46, 48, 1)])
def test_rooms_of_jobs_side_by_side(cg, ks):
    # 46 generators' selectors fit a warp's room, as do 10 generators of a hash-table job
    jobs = []
    for i, k in enumerate(ks):
        if k % 2 == 0:
            jobs.append((11, pairs(11, k, i), True, -1 if k > 9 else 14))
        gens = w.random_perms(np.random.default_rng(100 + k), 13, k)
        jobs.append((13, gens, False, 7 if k < 5 else 5 if k < 12 else 3))
        jobs.append((12, w.lrx(12), True, 24))
    want = [cg.growth(n, g, inv, rad, strategy="sweep" if n == 11 else "hash") for n, g, inv, rad in jobs]
    with cg.Batch(jobs) as b:
        for _ in range(2):
            for r, x in zip(b.run(), want):
                assert (r.layers, r.status) == (x.layers, x.status)


@pytest.mark.parametrize("n,k,radius", [(11, 4, 14), (11, 4, -1), (11, 10, -1), (12, 10, 8), (12, 2, 20), (11, 3, -1)])
def test_reading_first_or_not(cg, n, k, radius):
    # several S_11 and S_12 under the same rule in one batch and in one server, against one at a time
    from paper_2509_19162_gb300.serve import Server
    sets = [pairs(n, k, 10 * n + j) if k % 2 == 0 else w.random_perms(np.random.default_rng(j), n, k) for j in range(3)]
    closed = k % 2 == 0
    want = [cg.growth(n, g, closed, radius, strategy="sweep").layers for g in sets]
    with cg.Batch([(n, g, closed, radius) for g in sets]) as b:
        assert [r.layers for r in b.run()] == want
    with Server() as s:
        ids = [s.submit(n, g, closed, max_radius=radius) for g in sets]
        done = set()
        while len(done) < len(ids):
            s.step()
            done |= set(s.finished())
        assert [s.result(i).layers for i in ids] == want


def product(n, parts, seed):
    """Adjacent transpositions of S_a x S_b x .. on consecutive elements, renamed at random."""
    gens, o = [], 0
    for m in parts:
        gens += [w.families.transposition(n, o + i, o + i + 1) for i in range(m - 1)]
        o += m
    s = np.random.default_rng(seed).permutation(n).tolist()
    si = w.inverse(s)
    return [[si[g[s[i]]] for i in range(n)] for g in gens]


@pytest.mark.parametrize("count", [2, 30, 170])
@pytest.mark.parametrize("n", [9, 10])
def test_thin_growths_few_and_many(cg, n, count):
    # groups that fill little of S_n and growths cut off early, in clusters when they are few and as lists
    # when they are many, beside others that fill it
    kinds = [lambda j: (n, product(n, (n - 3, 2), j), True, -1), lambda j: (n, product(n, (n - 4, 3), j), True, 6),
             lambda j: (n, w.inverse_closure(w.random_perms(np.random.default_rng(j), n, 3)), True, 3),
             lambda j: (n, [list(g) + list(range(n - 2, n)) for g in w.lx(n - 2)], False, -1)]
    jobs = [kinds[j % 4](j) for j in range(count)]
    jobs[count // 2:count // 2] = [(n, w.lrx(n), True, -1), (8, product(8, (5, 2), 1), True, -1)]
    want = {}
    with cg.Batch(jobs) as b:
        for _ in range(2):
            for i, r in enumerate(b.run()):
                j = jobs[i]
                key = i if j[3] == 3 else str(sorted(map(tuple, j[1]))) + str(j[3])
                if key not in want:
                    want[key] = cg.growth(*j, strategy="hash")
                assert (r.layers, r.status) == (want[key].layers, want[key].status)


@pytest.mark.parametrize("sets", [("lrx",), ("lrx",) * 4, ("lrx",) * 5, ("lx", "coxeter"), ("coxeter", "lx", "lrx"),
                                  ("pancake", "coxeter")])
def test_a_handful_of_whole_s10(cg, sets):
    # few generators in all: lists on the whole grid; more: clusters; beside small jobs or one of n = 9 too
    def whole(n, f):
        return (n, w.FAMILIES[f](n), f != "lx", -1)
    for rest in ([], [whole(7, "coxeter")] * 3, [whole(9, "lrx")]):
        jobs = [whole(10, f) for f in sets] + rest
        with cg.Batch(jobs) as b:
            for _ in range(2):
                for j, r in zip(jobs, b.run()):
                    x = cg.growth(*j, strategy="hash")
                    assert (r.layers, r.status) == (x.layers, x.status)
