"""The waits of the general backward kernel (csrc/rib_bwd_sm100.cu) in a model of its warps with random delays (tests/test_frame_barriers.py:
a wait answers by parity, so its phase must be the one that is complete).  Rank 16: P^T and dS^T lie over the scores of one of three
buffers.  Rank 32: dP^T has two buffers of its own, dK~ reads dS from shared memory.  dV and dK~ are drained by the warps that drain dQ~
or by others (`apart`).  No GPU needed."""
import heapq

import pytest

from test_frame_barriers import Model


class Backward(Model):
    """`items` key blocks of `tiles` query tiles each; unit u = 2 * tile + half, its scores in buffer u mod 3."""

    def __init__(self, items, tiles, seed, rank, apart):
        super().__init__([tiles] * items, seed, True)
        self.tiles, self.rank, self.apart, self.total = tiles, rank, apart, items * tiles
        for name in ("dq", "drain", "v"):
            self.scale[name] = self.rng.choice((0.1, 1.0, 5.0))

    @staticmethod
    def on(name, unit):
        return (name, unit & 3), unit >> 2

    def scores(self):
        for u in range(2 * self.total):
            h, g = u & 1, u >> 1
            yield ("wait", *self.on("pfree", u - 3))
            assert u < 3 or ("dv", u - 3) in self.finished and (self.rank == 32 or ("dk", u - 3) in self.finished)
            if self.rank == 32:
                yield "wait", ("dpfree", h), g - 1
                assert u < 2 or ("read", u - 2) in self.finished
            yield "delay", self.delay("s")
            self.contract("s", ("s", u), [self.on("sfull", u)[0]])

    def gradients(self):
        for u in range(2 * self.total):
            item, last = u // (2 * self.tiles), (u + 1) % (2 * self.tiles) == 0
            yield ("wait", *self.on("pready", u))
            assert ("p", u) in self.finished
            if u % (2 * self.tiles) == 0 and item:
                yield "wait", "accfree", item - 1
                assert ("acc", item - 1) in self.finished
            yield "delay", self.delay("v")
            self.contract("v", ("dv", u), [self.on("pfree", u)[0]] if self.rank == 32 else [])
            bars = [self.on("pfree", u)[0]] if self.rank == 16 else [("dsfree", (u >> 1) & 1)] if u & 1 else []
            self.contract("v", ("dk", u), bars + (["accfull"] if last else []))

    def query_gradients(self):
        for g in range(self.total):
            for u in (2 * g, 2 * g + 1):
                yield ("wait", *self.on("pready", u))
                assert ("p", u) in self.finished
            if g:
                yield "wait", "dqfree", g - 1
                assert ("drained", g - 1) in self.finished
            yield "delay", self.delay("dq")
            self.contract("dq", ("dq", g), [("dsfree", g & 1), "dqfull"])

    def arithmetic(self, h):
        for g in range(self.total):
            u = 2 * g + h
            yield ("wait", *self.on("sfull", u))
            assert ("s", u) in self.finished
            yield "delay", self.delay("soft")
            yield "wait", ("dsfree", g & 1), (g >> 1) - 1
            assert g < 2 or ("dq", g - 2) in self.finished and (self.rank == 16 or ("dk", u - 4 + 1 - h) in self.finished)
            self.finished.add(("read", u))
            if self.rank == 32:
                self.arrive(("dpfree", h))
            yield "delay", self.delay("soft")
            self.finished.add(("p", u))
            self.arrive(self.on("pready", u)[0])

    def drain_item(self, item):
        yield "wait", "accfull", item
        u = 2 * self.tiles * (item + 1)
        assert ("dk", u - 1) in self.finished and ("dv", u) not in self.issued
        yield "delay", self.delay("drain")
        self.finished.add(("acc", item))
        self.arrive("accfree")

    def drain_items(self):
        for item in range(self.total // self.tiles):
            yield from self.drain_item(item)

    def drain(self):
        for g in range(self.total):
            if (g + 1) % self.tiles == 0 and not self.apart:
                yield from self.drain_item(g // self.tiles)
            yield "wait", "dqfull", g
            assert ("dq", g) in self.finished and ("dq", g + 1) not in self.issued
            yield "delay", self.delay("drain")
            self.finished.add(("drained", g))
            self.arrive("dqfree")

    def arrive(self, bar, count=1):
        super().arrive(bar, 2 if self.rank == 32 and bar[0] == "dsfree" else count)

    def run(self):
        self.pipe = {}
        processes = [self.scores(), self.gradients(), self.query_gradients(), self.arithmetic(0), self.arithmetic(1), self.drain()]
        for process in processes + ([self.drain_items()] if self.apart else []):
            self.later(self.delay("soft"), lambda process=process: self.step(process))
        while self.queue:
            self.now, _, what = heapq.heappop(self.queue)
            what()
        assert sum(f[0] == "drained" for f in self.finished) == self.total, "the warps wait for one another"


@pytest.mark.parametrize("rank,apart", [(16, True), (16, False), (32, False)])
@pytest.mark.parametrize("items,tiles", [(1, 8), (3, 8), (5, 1), (2, 18)])
def test_every_wait_sees_its_own_phase(items, tiles, rank, apart):
    for seed in range(200):
        Backward(items, tiles, seed, rank, apart).run()
