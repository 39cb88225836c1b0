"""bench.py names the kernels that grew a batch from the library's stats."""

import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402
import workloads as w  # noqa: E402


@pytest.mark.parametrize("stats,kernel,has,lacks", [
    ({"strategy_used": 4, "probe_variant": 1, "launches": 2}, None, ["cluster_grow"], ["hash_grow"]),
    ({"strategy_used": 3, "probe_variant": 17, "launches": 2}, "hash_grow_kernel<1, 2, 1, 0>", ["hash_grow"], ["cluster"]),
    ({"strategy_used": 1, "probe_variant": 12, "launches": 2}, "hash_grow_kernel<4, 1, 1, 0>", ["hash_grow"], ["cluster"]),
    ({"strategy_used": 3, "probe_variant": 17, "launches": 4}, None, ["cluster_grow", "hash_grow"], []),
])
def test_labels(stats, kernel, has, lacks):
    name, text = bench.batch_kernels(stats)
    assert name == kernel
    assert all(h in text for h in has) and not any(x in text for x in lacks)


@pytest.mark.gpu
def test_stats_say_which_kernels_ran():
    import torch
    assert torch.cuda.is_available()
    import paper_2509_19162_gb300 as cg
    cg.build()
    small, large, listed = (7, w.coxeter(7), True, -1), (9, w.lrx(9), True, -1), (11, w.lrx(11), True, 20)
    for jobs, visited, strategy, launches in (([small], "auto", 4, 1), ([small, large], "auto", 4, 2),
                                              ([listed], "auto", 3, 2), ([small, large, listed], "auto", 3, 4),
                                              ([small, large], "hash", 1, 2)):
        with cg.Batch(jobs, visited=visited) as b:
            for _ in range(2):
                b.run()
                st = b.stats()
                assert (st["strategy_used"], st["launches"]) == (strategy, launches)
            name, text = bench.batch_kernels(st)
            assert ("cluster" in text) == (visited == "auto" and len(jobs) + (jobs[0] is small) > 1)
            assert (name is None) == ("cluster" in text)


def test_block_bytes_by_hand():
    # S_4 in 6 blocks of 4 states, a 4-byte word each: layers 1, 3, 5, 6, 5, 3, 1 under adjacent transpositions
    layers = [1, 3, 5, 6, 5, 3, 1]
    grid = sum(4 * (a + b + 3 * c) + 2 for a, b, c in zip(layers, [0] + layers, layers[1:] + [0]))
    assert bench.block_bytes(4, layers, False) == grid
    assert bench.block_bytes(4, layers, True) == sum(4 * (2 * 6 + 3 * c) for c in layers[1:] + [0])
    # a layer takes a word a block at most: whole S_12 pancake, 12!/64 words of 8 bytes
    big = bench.block_bytes(12, [1, 10 ** 9], False)
    assert big == 8 * (1 + 3 * 7484400) + 8 * (7484400 + 1) + 4 * ((7484400 + 31) // 32)
