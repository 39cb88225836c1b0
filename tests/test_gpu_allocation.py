"""GPU tests of what a growth does with device memory: every allocation of every path failing once,
after which the same handle grows the graph as if nothing had been, and everything given back at the
end."""

import ctypes

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


class Device:
    """An allocator for the library: counts allocations, can fail one or all above a size, and knows
    what is held."""

    def __init__(self):
        import torch
        from paper_2509_19162_gb300 import _cg
        self.fail_at, self.limit = -1, None
        self.calls, self.live, self.held, self.peak = 0, {}, 0, 0

        def alloc(nbytes, stream, ctx):
            i, self.calls = self.calls, self.calls + 1
            if i == self.fail_at or (self.limit is not None and nbytes > self.limit):
                return None
            p = int(torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0))
            self.live[p] = int(nbytes)
            self.held += int(nbytes)
            self.peak = max(self.peak, self.held)
            return p

        def free(p, stream, ctx):
            if p:
                self.held -= self.live.pop(int(p))
                torch.cuda.caching_allocator_delete(int(p))

        self._cg, self._refs = _cg, (_cg.ALLOC_FN(alloc), _cg.FREE_FN(free))

    def __enter__(self):
        self._cg.check(self._cg.cg_set_allocator(self._refs[0], self._refs[1], None), "cg_set_allocator")
        return self

    def __exit__(self, *exc):
        self._cg.check(self._cg.cg_set_allocator(self._cg.ALLOC_FN(), self._cg.FREE_FN(), None), "cg_set_allocator")


PATHS = {
    "one block": (7, w.coxeter(7), {}),
    "one cluster": (9, w.lrx(9), {}),
    "rank bitmap": (10, w.lrx(10), {}),
    "hash table": (9, w.lx(9), {"strategy": "hash"}),
    "blocks": (11, w.coxeter(11), {}),
    "blocks after a list": (11, w.pancake(11), {"max_radius": 9}),
    "sweep": (9, w.lrx(9), {"strategy": "sweep"}),
    "sort": (9, w.lrx(9), {"strategy": "sort"}),
    "sort, many candidates": (10, w.coxeter(10), {"strategy": "sort"}),
    "list, then sort": (10, w.coxeter(10), {"mem_cap": 12 << 20}),
    "arrangement bitmap": (20, w.lrx(20), {"start": [1] * 10 + [0] * 10}),
    "two words, arrangements": (70, w.lrx(70), {"start": [1] * 3 + [0] * 67}),
    "two words, table": (18, w.lrx(18), {"max_radius": 9}),
}


@pytest.mark.parametrize("path", PATHS)
def test_a_run_after_a_failed_allocation(cg, path):
    # (a path took a buffer that a failed run had left for one that was ready: null tables, no maps)
    from paper_2509_19162_gb300._cg import CgError
    n, gens, kw = PATHS[path]
    with Device() as dev:
        with cg.Growth(n, gens, **kw) as g:
            want = g.run()
            far = np.sort(g.last_layer(), axis=0)
        total = dev.calls
        assert total > 0 and dev.held == 0
        for i in range(total):
            with cg.Growth(n, gens, **kw) as g:
                dev.fail_at = dev.calls + i
                try:
                    cut = g.run()
                    assert cut.status in (want.status, 2) and cut.layers == want.layers[:len(cut.layers)]
                except CgError as e:
                    assert e.code == -3
                    assert dev.held == 0            # a failed run holds nothing
                    with pytest.raises(CgError):
                        g.last_layer()
                dev.fail_at = -1
                again = g.run()
                assert (again.status, again.layers) == (want.status, want.layers)
                assert np.array_equal(np.sort(g.last_layer(), axis=0), far)
            assert dev.held == 0


@pytest.mark.parametrize("strategy", ["auto", "sweep"])
def test_sweep_without_room_for_a_fourth_bit(cg, strategy):
    # S_12 in blocks takes 240 MB, state by state 183 MB: a device with 200 MB to give still grows it
    n, gens = 12, w.pancake(12)
    want = cg.growth(n, gens, strategy="bitmap")
    with Device() as dev:
        dev.limit = 200 << 20
        with cg.Growth(n, gens, strategy=strategy) as g:
            for _ in range(2):
                got = g.run()
                assert (got.status, got.layers) == (want.status, want.layers)
            assert len(g.last_layer()) == want.layers[-1]
        assert dev.peak <= dev.limit and dev.held == 0


def test_large_binary_coset_without_room_for_every_state(cg):
    # 2.3 G arrangements of 34 bits: their keys take 18.7 GB, the first radii next to nothing
    n, start = 34, [1] * 17 + [0] * 17
    want = cg.growth(n, w.lrx(n), max_radius=12, strategy="hash", start=start)
    with Device() as dev:
        dev.limit = 4 << 30
        with cg.Growth(n, w.lrx(n), max_radius=12, start=start) as g:
            for _ in range(2):
                got = g.run()
                assert (got.status, got.layers) == (want.status, want.layers)
        assert dev.held == 0


def test_one_handle_stays_within_its_memory_cap(cg):
    # S_12: blocks 240 MB, state by state 183 MB, a list what it is given; never two of them at once
    from paper_2509_19162_gb300 import _cg
    n, gens, cap = 12, w.pancake(12), 300 << 20
    whole = cg.growth(n, gens, strategy="bitmap").layers
    with Device() as dev:
        with cg.Growth(n, gens, strategy="sweep", mem_cap=cap) as g:
            for order in ("auto", "rank", "auto"):
                g.set_sweep_order(order)
                assert g.run().layers == whole
                assert dev.peak <= cap
        with cg.Growth(n, gens, mem_cap=cap) as g:
            for stop in (0, 1000, 0):
                assert _cg.cg_growth_set_option(g._h, _cg.CG_OPT_STOP_ABOVE, stop) == 0
                got = g.run().layers
                assert got == whole[:len(got)] and (len(got) == len(whole) if not stop else got[-1] > stop)
                assert dev.peak <= cap
        assert dev.held == 0


def test_a_server_step_after_a_failed_allocation(cg):
    from paper_2509_19162_gb300._cg import CgError
    from paper_2509_19162_gb300.serve import Server
    want = cg.growth(8, w.lrx(8)).layers
    with Device() as dev:
        for i in range(6):              # the server's own five buffers, the job's
            with Server() as s:
                job = s.submit(8, w.lrx(8))
                dev.fail_at = dev.calls + i
                with pytest.raises(CgError) as e:
                    s.step()
                assert e.value.code == -3
                dev.fail_at = -1
                while job not in s.finished():
                    s.step()
                assert s.result(job).layers == want
            assert dev.held == 0


def test_a_solo_job_after_a_failed_allocation(cg):
    # a job that the server grows alone stays queued when its growth fails
    from paper_2509_19162_gb300._cg import CgError
    from paper_2509_19162_gb300.serve import Server
    n, radius, share = 12, 20, 1 << 30
    want = cg.growth(n, w.pancake(n), max_radius=radius, strategy="bitmap", mem_cap=share)   # as far as its share goes
    with Device() as dev:
        with Server(job_mem_cap=share) as s:
            job = s.submit(n, w.pancake(n), max_radius=radius)
            dev.fail_at = dev.calls + 5         # behind the server's own five buffers
            with pytest.raises(CgError) as e:
                s.step()
            assert e.value.code == -3 and s.load()[0] == 1
            dev.fail_at = -1
            while job not in s.finished():
                s.step()
            assert s.result(job).layers == want.layers
        assert dev.held == 0
