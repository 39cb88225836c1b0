"""GPU tests of the sorted step where layers are thin beside the number of generators: a state's
generators spread over several threads of the histogram, a tile of candidates that spans many
generators.  Whole numbers: every comparison is exact."""

import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,family,radius", [
    (6, "all_transpositions", -1),      # 15 generators, tags: layers of at most 274 states
    (7, "all_transpositions", -1),      # 21 generators
    (8, "three_cycles", -1),            # 112 generators: 37 to 4725 states a layer, tiles across 110
    (9, "reversals", 4),                # 36 generators
    (10, "three_cycles", 2),            # 240 generators, the second step's 57,600 candidates
    (11, "coxeter", 12),                # 10 generators, layers on both sides of a tile's 4096 keys
])
def test_thin_layers_with_many_generators(n, family, radius):
    import torch
    assert torch.cuda.is_available()
    import paper_2509_19162_gb300 as cg
    cg.build()
    out = []
    for strategy in ("sort", "hash"):
        with cg.Growth(n, w.FAMILIES[family](n), strategy=strategy, max_radius=radius, keep_last=True) as g:
            r = g.run()
            out.append((r.status, r.layers, np.sort(np.asarray(g.last_layer(), dtype=np.uint64))))
    assert out[0][:2] == out[1][:2]
    assert np.array_equal(out[0][2], out[1][2])


@pytest.mark.parametrize("n,family,kw", [
    (5, "star", {}), (7, "lrx", {}), (8, "lrx", {}),                        # one block to the end, or at the end
    (8, "lrx", {"max_radius": 3}), (8, "lrx", {"max_radius": 10}),          # stopped in one block, after larger steps
    (8, "coxeter", {"stop_above": 20}), (9, "coxeter", {"stop_above": 3000}),
])
def test_last_layer_has_plain_keys(n, family, kw):
    # states carry the generator that leads back above their keys while the growth goes on
    import paper_2509_19162_gb300 as cg
    out = []
    for strategy in ("sort", "hash"):
        with cg.Growth(n, w.FAMILIES[family](n), strategy=strategy, keep_last=True, **kw) as g:
            for _ in range(2):
                r = g.run()
                out.append((r.status, r.layers, np.sort(np.asarray(g.last_layer(), dtype=np.uint64)).tolist()))
            if strategy == "sort" and n < 8:
                assert g.stats()["launches"] == 1       # nothing beside the one block
    assert all(o == out[0] for o in out)
