"""The waits of the general backward kernel (csrc/rib_bwd_sm100.cu) in a model of its warps with random delays (tests/test_frame_barriers.py:
a wait answers by parity, so its phase must be the one that is complete).  Copies in and out end at times of their own.  Every role of
several warps is two processes here.  Rank 16: P^T and dS^T lie over the scores of one of three buffers.  Rank 32: dP^T has two buffers of
its own, dK~ reads dS from shared memory.  dV rows leave through V's slot, dK rows through a tile of their own; they are drained by the warps that
drain dQ~ or by others (`apart`).  No GPU needed."""
import heapq

import pytest

from test_frame_barriers import Model

WARPS = (0, 1)           # of a role of several warps


class Backward(Model):
    """`items` key blocks of `tiles` query tiles each; unit u = 2 * tile + half, its scores in buffer u mod 3.  `fault`: a rule left out."""

    def __init__(self, items, tiles, seed, rank, apart, fault=None):
        super().__init__([tiles] * items, seed, True)
        self.count, self.tiles, self.rank, self.apart, self.total, self.fault = items, tiles, rank, apart, items * tiles, fault
        for name in ("dq", "drain", "v", "load", "store"):
            self.scale[name] = self.rng.choice((0.1, 1.0, 5.0))
        both = len(WARPS)
        self.counts = {"pready": both, "dpfree": both, "dqfree": both, "accfree": both, "dsfree": 2 if rank == 32 else 1,
                       "kvempty": 1 if fault == "slot" else 1 + both}

    def on(self, name, unit):
        return ((name, unit & 1), unit >> 1) if self.fault == name else ((name, unit & 3), unit >> 2)

    def arrive(self, bar, count=1):
        super().arrive(bar, self.counts.get(bar if isinstance(bar, str) else bar[0], 1))

    def all_done(self, *what):
        return all((*what, w) in self.finished for w in WARPS)

    def units(self, item):
        return range(2 * self.tiles * item, 2 * self.tiles * (item + 1))

    def copy(self, name, what, bar):
        """A bulk copy that was asked for."""
        self.issued.add(what)

        def complete():
            self.finished.add(what)
            self.arrive(bar)
        self.later(self.delay(name), complete)

    def producer(self):
        for item in range(self.count):
            if item >= 2:
                yield "wait", ("kvempty", item & 1), (item >> 1) - 1
                assert all(("s", u) in self.finished for u in self.units(item - 2)), "V under dP^T"
                assert all(("dq", u >> 1) in self.finished for u in self.units(item - 2)), "K~ under dQ~"
                assert self.all_done("out", item - 2), "V under the rows of dV"
            self.copy("load", ("kv", item), ("kvfull", item & 1))
            for g in range(item * self.tiles, (item + 1) * self.tiles):
                if g >= 4:
                    yield "wait", ("qempty", g & 3), (g >> 2) - 1
                    for u in (2 * g - 8, 2 * g - 7):
                        assert ("dv", u) in self.finished and ("dk", u) in self.finished and self.all_done("p", u), "query rows in use"
                self.copy("load", ("q", g), ("qfull", g & 3))

    def scores(self):
        for u in range(2 * self.total):
            h, g, item = u & 1, u >> 1, u // (2 * self.tiles)
            if u % (2 * self.tiles) == 0:
                yield "wait", ("kvfull", item & 1), item >> 1
            if h == 0:
                yield "wait", ("qfull", g & 3), g >> 2
            yield ("wait", *self.on("pfree", u - 3))
            assert ("kv", item) in self.finished and ("q", g) in self.finished
            assert u < 3 or ("dv", u - 3) in self.finished and (self.rank == 32 or ("dk", u - 3) in self.finished)
            if self.rank == 32:
                yield "wait", ("dpfree", h), g - 1
                assert u < 2 or self.all_done("read", u - 2)
            yield "delay", self.delay("s")
            assert ("kv", item + 2) not in self.issued and ("q", g + 4) not in self.issued
            self.contract("s", ("s", u), [self.on("sfull", u)[0]])

    def gradients(self):
        for u in range(2 * self.total):
            item, last = u // (2 * self.tiles), (u + 1) % (2 * self.tiles) == 0
            yield ("wait", *self.on("pready", u))
            assert self.all_done("p", u)
            if u % (2 * self.tiles) == 0 and item:
                yield "wait", "accfree", item - 1
                assert self.all_done("acc", item - 1)
            yield "delay", self.delay("v")
            self.contract("v", ("dv", u), [self.on("pfree", u)[0]] if self.rank == 32 else [])
            bars = [self.on("pfree", u)[0]] if self.rank == 16 else [("dsfree", (u >> 1) & 1)] if u & 1 else []
            self.contract("v", ("dk", u), bars + ([("qempty", (u >> 1) & 3)] if u & 1 else []) + (["accfull"] if last else []))

    def query_gradients(self):
        for g in range(self.total):
            for u in (2 * g, 2 * g + 1):
                yield ("wait", *self.on("pready", u))
                assert self.all_done("p", u)
            if g:
                yield "wait", "dqfree", g - 1
                assert self.all_done("drained", g - 1)
            yield "delay", self.delay("dq")
            item, last = g // self.tiles, (g + 1) % self.tiles == 0
            self.contract("dq", ("dq", g), [("dsfree", g & 1), "dqfull"] + ([("kvempty", item & 1)] if last else []))

    def arithmetic(self, h, warp):
        for g in range(self.total):
            u = 2 * g + h
            yield ("wait", *self.on("sfull", u))
            yield "wait", ("qfull", g & 3), g >> 2
            assert ("s", u) in self.finished and ("q", g) in self.finished
            yield "delay", self.delay("soft")
            yield "wait", ("dsfree", g & 1), (g >> 1) - 1
            assert g < 2 or ("dq", g - 2) in self.finished and (self.rank == 16 or ("dk", u - 4 + 1 - h) in self.finished)
            self.finished.add(("read", u, warp))
            if self.rank == 32:
                self.arrive(("dpfree", h))
            yield "delay", self.delay("soft")
            assert ("q", g + 4) not in self.issued
            self.finished.add(("p", u, warp))
            self.arrive(self.on("pready", u)[0])

    def drain_item(self, item, warp):
        yield "wait", "accfull", item
        u = 2 * self.tiles * (item + 1)
        assert ("dk", u - 1) in self.finished and ("dv", u) not in self.issued
        assert all(("s", v) in self.finished for v in self.units(item)) and ("kv", item + 2) not in self.issued, "dV rows over V"
        assert item == 0 or ("out", item - 1, warp) in self.finished, "dK rows over those of the item before"
        yield "delay", self.delay("drain")
        assert ("kv", item + 2) not in self.issued
        self.finished.add(("acc", item, warp))
        self.arrive("accfree")
        self.copy("store", ("out", item, warp), ("group", warp))

    def release_slot(self, item, warp):
        yield "wait", ("group", warp), item
        assert ("kv", item + 2) not in self.issued, "the slot went before its rows had been read"
        if self.fault != "slot":
            self.arrive(("kvempty", item & 1))

    def drain_items(self, warp):
        for item in range(self.count):
            yield from self.drain_item(item, warp)
            yield from self.release_slot(item, warp)

    def drain(self, warp):
        for g in range(self.total):
            last = (g + 1) % self.tiles == 0
            if last and not self.apart:
                yield from self.drain_item(g // self.tiles, warp)
            yield "wait", "dqfull", g
            assert ("dq", g) in self.finished and ("dq", g + 1) not in self.issued
            yield "delay", self.delay("drain")
            self.finished.add(("drained", g, warp))
            self.arrive("dqfree")
            if last and not self.apart:
                yield from self.release_slot(g // self.tiles, warp)

    def run(self):
        self.pipe = {}
        processes = [self.producer(), self.scores(), self.gradients(), self.query_gradients()]
        for w in WARPS:
            processes += [self.arithmetic(0, w), self.arithmetic(1, w), self.drain(w)] + ([self.drain_items(w)] if self.apart else [])
        for process in processes:
            self.later(self.delay("soft"), lambda process=process: self.step(process))
        while self.queue:
            self.now, _, what = heapq.heappop(self.queue)
            what()
        assert sum(f[0] == "drained" for f in self.finished) == len(WARPS) * self.total, "the warps wait for one another"
        assert sum(f[0] == "out" for f in self.finished) == len(WARPS) * self.count


SHAPES = [(1, 8), (3, 8), (5, 1), (2, 18), (6, 2)]
FORMS = [(16, True), (16, False), (32, False)]


@pytest.mark.parametrize("rank,apart", FORMS)
@pytest.mark.parametrize("items,tiles", SHAPES)
def test_every_wait_sees_its_own_phase(items, tiles, rank, apart):
    for seed in range(200):
        Backward(items, tiles, seed, rank, apart).run()


@pytest.mark.parametrize("fault", ["slot", "pready"])
@pytest.mark.parametrize("rank,apart", FORMS)
def test_the_model_finds_a_rule_that_is_left_out(rank, apart, fault):
    """slot: V's slot is given back by the last dQ~ alone.  pready: P^T and dS^T announced per half of a tile, of which dQ~'s issuer may miss a phase."""
    found = 0
    for items, tiles in SHAPES:
        for seed in range(100):
            try:
                Backward(items, tiles, seed, rank, apart, fault).run()
            except AssertionError:
                found += 1
    assert found
