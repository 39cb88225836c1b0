"""GPU tests of two-word cosets on both sides of the orbit size from which AUTO ranks arrangements."""

import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts,family,used", [
    ((65, 1), "lrx", 1), ((127, 1), "coxeter", 1), ((70, 1), "lx", 1),      # a state a position: hash table
    ((31, 2), "lrx", None),                                                # 33 elements of one bit: one word
    ((22, 1, 9), "lrx", None), ((30, 1, 1, 1), "lrx", 3), ((64, 2), "lx", 3), ((38, 1, 1), "coxeter", 3),
])
def test_orbits_small_and_large_enough_to_rank(counts, family, used):
    import torch
    assert torch.cuda.is_available()
    import paper_2509_19162_gb300 as cg
    cg.build()
    start = [v for v, c in enumerate(counts) for _ in range(c)]
    n, gens = len(start), w.FAMILIES[family](len(start))
    start = np.random.default_rng(n).permutation(start).tolist()
    kw = {"max_radius": 30} if len(counts) == 3 and counts[2] > 5 else {}
    out = []
    for strategy in ("hash", "auto"):
        with cg.Growth(n, gens, strategy=strategy, start=start, **kw) as g:
            for _ in range(2):
                r = g.run()
                out.append((r.status, r.layers, np.sort(g.last_layer(), axis=0).tolist()))
            if strategy == "auto" and used:
                assert g.stats()["strategy_used"] == used
    assert all(o == out[0] for o in out)
