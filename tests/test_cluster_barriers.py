"""Thread-block clusters: a block may reach into another block's shared memory only after a barrier of
the cluster has shown that the other block runs.  Nothing on a GPU shows a missing first barrier
reliably, and the access is undefined without it, so the order is read from the kernels' source."""

import os
import re

import numpy as np
import pytest

import workloads as w

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_19162_gb300", "csrc")


def _bodies(text):
    """(name, body without comments) of every function definition that ends at a line "}"."""
    text = re.sub(r"//[^\n]*|__launch_bounds__\([^)]*\)", "", text)
    for m in re.finditer(r"^(?:__global__|__device__)[^;{]*?(\w+)\([^;{]*\)\s*\{\n(.*?)^\}", text, re.S | re.M):
        yield m.group(1), m.group(2)


def test_cluster_barrier_before_the_first_remote_access():
    found = {}
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name)) as f:
                found.update({n: b for n, b in _bodies(f.read()) if "map_shared_rank" in b})
    assert {"cluster_grow", "cluster_grow_kernel"} <= set(found)
    for name, body in found.items():
        # a lambda that only names the remote word is not an access; its first use is
        first = body.index("*word(") if "auto word =" in body else body.index("map_shared_rank")
        assert re.search(r"cl\.sync\(\)|growth_sync<", body[:first]), f"{name}: remote access before a barrier"


@pytest.mark.gpu
@pytest.mark.parametrize("n", [9, 10])
def test_first_pass_of_many_clusters(n):
    # more growths than clusters run at once, launched again and again: the first pass of every launch
    # hands out jobs while its blocks are still starting
    import torch
    assert torch.cuda.is_available()
    import paper_2509_19162_gb300 as p
    p.build()
    rng = np.random.default_rng(n)
    jobs = [(n, w.inverse_closure(w.random_perms(rng, n, 2)), True, 6) for _ in range(96)]
    want = [p.growth(*j, strategy="hash").layers for j in jobs]
    with p.Batch(jobs) as b:
        for _ in range(20):
            assert [r.layers for r in b.run()] == want
