"""Performance cases of the growth library: what users have it do, through its public entry points.

A case is one growth (``Growth(...).run()``, the whole call from the generators to the closed
handle, with the antipodes read back where a permutation group is grown whole), one run of a
prepared batch, or one stream of jobs taken through a prepared server.  Inputs come from a seed: the
central state a graph is grown from is a random arrangement, and random generator sets are drawn
from it.

Kinds of case
  "perm"     whole growth of a permutation Cayley graph of a named family from a random permutation;
             ``strategy`` and ``mem_cap`` as in ``Growth`` ("auto" and 0: the library's choice).
  "random"   growth of S_n under k random permutations and their inverses, stopped after the first
             layer larger than ``stop_above``.
  "coset"    growth of the orbit of a vector with repeated values (a Schreier coset graph), from a
             random arrangement of ``counts`` ("15,15": fifteen zeros, fifteen ones).
  "batch"    ``jobs`` independent random groups (half with their inverses) run together.
  "serve"    ``jobs`` jobs of mixed families and sizes submitted to a server and stepped to the end.
"""

import math

import numpy as np

from paper_2509_19162_gb300 import Batch, Growth
from paper_2509_19162_gb300.serve import Server


# ---- generator sets ---------------------------------------------------------------------------

def _swap(n, i, j):
    p = list(range(n))
    p[i], p[j] = p[j], p[i]
    return p


def _coxeter(n):
    return [_swap(n, i, i + 1) for i in range(n - 1)]


def _cyclic_coxeter(n):
    return _coxeter(n) + [_swap(n, 0, n - 1)]


def _star(n):
    return [_swap(n, 0, i) for i in range(1, n)]


def _all_transpositions(n):
    return [_swap(n, i, j) for i in range(n) for j in range(i + 1, n)]


def _pancake(n):
    return [[j - 1 - i if i < j else i for i in range(n)] for j in range(2, n + 1)]


def _lx(n):
    return [[(i + 1) % n for i in range(n)], _swap(n, 0, 1)]


def _lrx(n):
    left, x = _lx(n)
    return [left, _inverse(left), x]


def _four_cycles(n):
    gens = []
    for i in range(n - 3):
        p = list(range(n))
        p[i], p[i + 1], p[i + 2], p[i + 3] = i + 1, i + 2, i + 3, i
        gens.append(p)
    return gens


FAMILIES = {"coxeter": _coxeter, "cyclic_coxeter": _cyclic_coxeter, "star": _star,
            "all_transpositions": _all_transpositions, "pancake": _pancake, "lx": _lx, "lrx": _lrx,
            "four_cycles": _four_cycles}


def _inverse(p):
    inv = [0] * len(p)
    for i, v in enumerate(p):
        inv[v] = i
    return inv


def _random_gens(rng, n, k, inverses):
    gens = []
    while len(gens) < k:
        p = rng.permutation(n).tolist()
        if p != list(range(n)) and p not in gens:
            gens.append(p)
    if inverses:
        gens += [q for q in map(_inverse, list(gens)) if q not in gens]
    return gens


# ---- the cases ----------------------------------------------------------------------------------

def listed():
    return [
        # The smallest real call: a textbook graph of 40,320 states in 29 layers, latency bound.
        {"name": "s8_coxeter", "kind": "perm", "family": "coxeter", "n": 8, "strategy": "auto", "mem_cap": 0},
        # A directed graph (L and X without R): 3.6 M states in many thin layers, full visited set.
        {"name": "s10_lx_directed", "kind": "perm", "family": "lx", "n": 10, "strategy": "auto", "mem_cap": 0},
        # The ordinary research call and the framework's headline: S_11 under L, R, X.
        {"name": "s11_lrx", "kind": "perm", "family": "lrx", "n": 11, "strategy": "auto", "mem_cap": 0},
        # A large whole group with many generators whose visited set still fits L2.
        {"name": "s12_pancake", "kind": "perm", "family": "pancake", "n": 12, "strategy": "auto", "mem_cap": 0},
        # The largest: 6.2 G states, 50 GB of layers, a visited set far beyond L2.
        {"name": "s13_pancake", "kind": "perm", "family": "pancake", "n": 13, "strategy": "auto", "mem_cap": 0},
        # Random generators without locality, a truncated growth of a group too large to finish.
        {"name": "s14_random", "kind": "random", "n": 14, "k": 3, "stop_above": 1 << 27},
        # A memory cap (a shared GPU) that the stored layers exceed: bitmaps instead of state lists.
        {"name": "s12_coxeter_1gib", "kind": "perm", "family": "coxeter", "n": 12, "strategy": "auto",
         "mem_cap": 1 << 30},
        # The sorted two-layer step, which undirected growths beyond memory use.
        {"name": "s11_lrx_sorted", "kind": "perm", "family": "lrx", "n": 11, "strategy": "sort", "mem_cap": 0},
        # The binary Schreier graph of the paper's tables: 155 M states, one bit an element.
        {"name": "bin30_lrx", "kind": "coset", "family": "lrx", "counts": "15,15"},
        # A long vector of four values: keys of two words.
        {"name": "coset40_lrx", "kind": "coset", "family": "lrx", "counts": "35,2,2,1"},
        # Screening of many small random groups, n in 6..10.
        {"name": "batch1024", "kind": "batch", "jobs": 1024, "n_min": 6, "n_max": 10},
        # A job service under mixed load, n in 8..12.
        {"name": "serve40", "kind": "serve", "jobs": 40, "n_min": 8, "n_max": 12},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["perm", "perm", "perm", "random", "coset", "coset", "batch", "serve"])
    if kind == "perm":
        how = rng.choice(["auto", "auto", "capped", "sort"])
        if how == "sort":
            return {"kind": kind, "family": rng.choice(["lrx", "coxeter", "pancake", "star"]), "n": rng.randint(7, 11),
                    "strategy": "sort", "mem_cap": 0}
        family = rng.choice(["coxeter", "cyclic_coxeter", "star", "pancake", "lx", "lrx", "all_transpositions"])
        n = rng.randint(6, 10 if family in ("all_transpositions", "lx") else 12)
        if how == "capped" and n >= 9:      # between the bitmaps' bytes and the stored layers'
            return {"kind": kind, "family": family, "n": n, "strategy": "auto",
                    "mem_cap": int(math.factorial(n) * rng.uniform(0.9, 4.0))}
        return {"kind": kind, "family": family, "n": n, "strategy": "auto", "mem_cap": 0}
    if kind == "random":
        return {"kind": kind, "n": rng.randint(12, 16), "k": rng.randint(2, 4), "stop_above": _log(rng, 1 << 14, 1 << 27)}
    if kind == "coset":
        how = rng.choice(["binary", "values", "two_words"])
        if how == "binary":
            n = rng.randint(18, 30)
            return {"kind": kind, "family": rng.choice(["lrx", "pancake", "coxeter", "four_cycles"]),
                    "counts": "%d,%d" % (n // 2, n - n // 2)}
        if how == "values":
            a, b, c = rng.randint(5, 9), rng.randint(3, 6), rng.randint(2, 4)
            return {"kind": kind, "family": rng.choice(["lrx", "coxeter"]), "counts": "%d,%d,%d" % (a, b, c)}
        if rng.random() < 0.5:
            return {"kind": kind, "family": rng.choice(["lrx", "pancake"]), "counts": "%d,2,2,1" % rng.randint(29, 37)}
        return {"kind": kind, "family": rng.choice(["lrx", "four_cycles"]), "counts": "%d,%d" % (rng.randint(62, 75), 4)}
    if kind == "batch":
        return {"kind": kind, "jobs": _log(rng, 24, 1536), "n_min": rng.randint(4, 6), "n_max": rng.randint(8, 10)}
    return {"kind": kind, "jobs": rng.randint(8, 56), "n_min": rng.randint(6, 8), "n_max": rng.randint(10, 12)}


# ---- what a user's program has in hand ------------------------------------------------------------

def _serve_jobs(case, rng):
    """(n, generators, radius cap) of each job: families and sizes in turn, random generators and
    caps from the seed."""
    names = ("coxeter", "all_transpositions", "lrx", "pancake", "random")
    span = case["n_max"] - case["n_min"] + 1
    jobs = []
    for i in range(case["jobs"]):
        name, n = names[i % 5], case["n_min"] + (i // 5 + i) % span
        if name == "random":
            gens = _random_gens(rng, n, 2 + i // 5 % 3, True)
        else:
            gens = FAMILIES[name](n)
        top = {"coxeter": n * (n - 1) // 2, "lrx": n * (n - 1) // 2, "all_transpositions": n - 1,
               "pancake": math.ceil(1.2 * n) + 2, "random": n * n // 2 + 4 * n}[name]
        jobs.append((n, gens, max(6, top) - int(rng.integers(0, max(2, top // 4)))))
    return jobs


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "perm":
        n = case["n"]
        return {"kind": kind, "n": n, "gens": FAMILIES[case["family"]](n), "start": rng.permutation(n).tolist(),
                "strategy": case["strategy"], "mem_cap": case["mem_cap"], "stop_above": 0, "antipodes": True}
    if kind == "random":
        return {"kind": kind, "n": case["n"], "gens": _random_gens(rng, case["n"], case["k"], True), "start": None,
                "strategy": "auto", "mem_cap": 0, "stop_above": case["stop_above"], "antipodes": False}
    if kind == "coset":
        counts = [int(c) for c in case["counts"].split(",")]
        start = rng.permutation(np.repeat(np.arange(len(counts)), counts)).tolist()
        return {"kind": kind, "n": len(start), "gens": FAMILIES[case["family"]](len(start)), "start": start,
                "strategy": "auto", "mem_cap": 0, "stop_above": 0, "antipodes": False}
    if kind == "batch":
        jobs = []
        for j in range(case["jobs"]):
            n, k = int(rng.integers(case["n_min"], case["n_max"] + 1)), int(rng.integers(2, 6))
            gens = _random_gens(rng, n, k, j % 2 == 0)
            jobs.append((n, gens, all(_inverse(g) in gens for g in gens), -1))
        return {"kind": kind, "batch": Batch(jobs)}
    return {"kind": kind, "jobs": _serve_jobs(case, rng), "server": Server()}


# ---- one pass -------------------------------------------------------------------------------------

LAYERS = 1024       # more than any growth of these ranges has


def _table(results):
    """Layer sizes of many growths, a row each (zeros after the last layer), and their statuses."""
    sizes = np.zeros((len(results), LAYERS), dtype=np.int64)
    for row, r in zip(sizes, results):
        row[:len(r.layers)] = r.layers
    return {"sizes": sizes, "status": np.array([r.status for r in results], dtype=np.int64)}


def run(state):
    if state["kind"] == "batch":
        return _table(state["batch"].run())
    if state["kind"] == "serve":
        server = state["server"]
        ids = [server.submit(n, gens, max_radius=cap) for n, gens, cap in state["jobs"]]
        done = {}
        while len(done) < len(ids):
            server.step()
            for i in server.finished():
                done[i] = server.result(i)
        return _table([done[i] for i in ids])
    with Growth(state["n"], state["gens"], mem_cap=state["mem_cap"], strategy=state["strategy"],
                stop_above=state["stop_above"], keep_last=state["antipodes"], start=state["start"]) as g:
        out = _table([g.run()])
        if state["antipodes"]:      # the states farthest from the start; they come in no particular order
            out["antipodes"] = np.sort(g.last_layer()).view(np.int64)
    return out


# ---- what a pass cannot do without -----------------------------------------------------------------

def _growth_work(states, expanded, k, n, visited_bytes):
    """Every state is written once and read once as a frontier key (8 bytes), every visited bit set;
    every edge out of an expanded state moves n elements (counted as operations)."""
    return {"bytes": 8.0 * states + 8.0 * expanded + visited_bytes, "flops": 1.0 * k * expanded * n}


def _add(a, b):
    return {"bytes": a["bytes"] + b["bytes"], "flops": a["flops"] + b["flops"]}


def work(case):
    kind = case["kind"]
    if kind == "perm":
        n = case["n"]
        order, k = math.factorial(n), len(FAMILIES[case["family"]](n))
        return _growth_work(order, order, k, n, order / 8)
    if kind == "random":
        k, order = 2 * case["k"], math.factorial(case["n"])
        layer, states, expanded = k, 1 + k, 1
        while layer <= case["stop_above"] and states < order // 4:
            expanded, layer = states, layer * (k - 1)
            states += layer
        return _growth_work(states, expanded, k, case["n"], states / 8)
    if kind == "coset":
        counts = [int(c) for c in case["counts"].split(",")]
        n, orbit = sum(counts), math.factorial(sum(counts))
        for c in counts:
            orbit //= math.factorial(c)
        bits = n * max(1, math.ceil(math.log2(len(counts))))
        out = _growth_work(orbit, orbit, len(FAMILIES[case["family"]](n)), n, orbit / 8)
        out["bytes"] *= 1 if bits <= 64 else 2
        return out
    out = {"bytes": 0.0, "flops": 0.0}
    if kind == "batch":         # n uniform, k uniform in 2..5, half of the sets doubled by inverses
        span = case["n_max"] - case["n_min"] + 1
        for n in range(case["n_min"], case["n_max"] + 1):
            order = math.factorial(n)
            one = _growth_work(order, order, 3.5 * 1.5, n, order / 8)
            share = case["jobs"] / span
            out = _add(out, {"bytes": one["bytes"] * share, "flops": one["flops"] * share})
        return out
    for n, gens, _ in _serve_jobs(case, np.random.default_rng(0)):
        order = math.factorial(n)
        out = _add(out, _growth_work(order, order, len(gens), n, order / 8))
    return out
