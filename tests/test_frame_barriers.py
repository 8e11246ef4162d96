"""The waits of the frame kernel (csrc/rib_fwd_frame_sm100.cu) on its score and PV contractions, in a model of its warps with random
delays.  A parity wait cannot tell a phase from the one two before or after it, so each must be on a barrier of which the phase before is
known to be complete and the next cannot be yet; a commit tells when contractions are complete, and how long its arrival takes is open:
two commits behind the same contractions may arrive in either order.  No GPU needed."""
import heapq
import random

import pytest

BUFFERS = 3


class WrongPhase(AssertionError):
    pass


class Model:
    """One CTA.  Unit u = 2 * block + tile; its scores, and P over them, are in buffer u mod 3.  `split`: scores and completed PV are
    announced per tile and parity of the block, as P is; else scores per buffer, completed PV per tile and, for the next scores, per buffer."""

    def __init__(self, items, seed, split):
        self.items, self.rng, self.split = items, random.Random(seed), split
        self.now, self.queue, self.order = 0.0, [], 0
        self.done, self.waiting, self.arrivals = {}, {}, {}
        self.issued, self.finished = set(), set()          # (kind, unit)
        self.scale = {name: self.rng.choice((0.1, 1.0, 5.0)) for name in ("s", "pv0", "pv1", "soft", "lag", "mma")}

    def later(self, delay, what):
        self.order += 1
        heapq.heappush(self.queue, (self.now + delay, self.order, what))

    def delay(self, name):
        return self.scale[name] * self.rng.expovariate(1.0)

    def arrive(self, bar, count=1):
        self.arrivals[bar] = self.arrivals.get(bar, 0) + 1
        if self.arrivals[bar] % count == 0:
            self.done[bar] = self.done.get(bar, 0) + 1
            for process, phase in self.waiting.pop(bar, []):
                self.wait(process, bar, phase)

    def wait(self, process, bar, phase):
        """Answers by the parity of the phase, and checks that it is that phase which is complete, and none behind it."""
        done = self.done.get(bar, 0)
        if (done - 1) & 1 != phase & 1:
            self.waiting.setdefault(bar, []).append((process, phase))
        elif done != phase + 1:
            raise WrongPhase(f"{bar}: asked for phase {phase}, {done} complete")
        else:
            self.later(0.0, lambda: self.step(process))

    def step(self, process):
        try:
            what = next(process)
        except StopIteration:
            return
        if what[0] == "delay":
            self.later(what[1], lambda: self.step(process))
        else:
            self.wait(process, *what[1:])

    def contract(self, warp, what, bars):
        """Contractions of a warp finish in order; every commit behind them arrives at a time of its own."""
        self.issued.add(what)
        self.pipe[warp] = finish = max(self.pipe.get(warp, 0.0), self.now) + self.delay("mma")

        def complete():
            self.finished.add(what)
            for bar in bars:
                self.later(self.delay("lag"), lambda bar=bar: self.arrive(bar))
        self.later(finish - self.now, complete)

    def pv_phase(self, tile, block):                    # barrier and phase of a completed PV
        return (("pv", tile, block & 1), block >> 1) if self.split else (("pv", tile), block)

    def score_phase(self, tile, block):
        u = 2 * block + tile
        return (("s", tile, block & 1), block >> 1) if self.split else (("s", u % BUFFERS), u // BUFFERS)

    def blocks(self):
        return [(block, j, n) for block, (j, n) in enumerate((j, n) for n in self.items for j in range(n))]

    def scores(self):
        for block, _, _ in self.blocks():
            for tile in range(2):
                u = 2 * block + tile
                if self.split:
                    yield ("wait", *self.pv_phase(1 - tile, (u - 3) >> 1))
                else:
                    yield "wait", ("pfree", u % BUFFERS), u // BUFFERS - 1
                assert u < BUFFERS or ("pv", u - BUFFERS) in self.finished, "scores over a P that PV still reads"
                yield "delay", self.delay("s")
                self.contract("s", ("s", u), [self.score_phase(tile, block)[0]])

    def pv(self, tile):
        for block, _, _ in self.blocks():
            u = 2 * block + tile
            yield "wait", ("pready", tile, block & 1), block >> 1
            assert all(("p", u, half) in self.finished for half in range(2))
            yield "delay", self.delay(f"pv{tile}")
            self.contract(f"pv{tile}", ("pv", u), ([] if self.split else [("pfree", u % BUFFERS)]) + [self.pv_phase(tile, block)[0]])

    def softmax(self, tile, half):
        for block, j, n in self.blocks():
            u = 2 * block + tile
            yield ("wait", *self.score_phase(tile, block))
            assert ("s", u) in self.finished
            yield "delay", self.delay("soft")
            if j and self.rng.random() < 0.3:           # the maximum grew: the output so far is scaled
                yield ("wait", *self.pv_phase(tile, block - 1))
                assert ("pv", u - 2) in self.finished and ("pv", u) not in self.issued
            if not self.split and j == n - 1 and block:
                yield ("wait", *self.pv_phase(tile, block - 1))
            self.finished.add(("p", u, half))
            self.arrive(("pready", tile, block & 1), 2)
            if j == n - 1:                              # the output is read
                yield ("wait", *self.pv_phase(tile, block))
                assert ("pv", u) in self.finished and ("pv", u + 2) not in self.issued
                yield "delay", self.delay("soft")
                assert ("pv", u + 2) not in self.issued

    def run(self):
        self.pipe = {}
        processes = [self.scores(), self.pv(0), self.pv(1)] + [self.softmax(t, h) for t in range(2) for h in range(2)]
        for process in processes:
            self.later(self.delay("soft"), lambda process=process: self.step(process))
        while self.queue:
            self.now, _, what = heapq.heappop(self.queue)
            what()
        assert len([f for f in self.finished if f[0] == "pv"]) == 2 * sum(self.items), "the warps wait for one another"


SHAPES = [[1], [1, 1, 1, 1, 1], [2, 1, 3, 1], [8, 8], [3, 5, 2, 7, 1, 4]]


@pytest.mark.parametrize("items", SHAPES, ids=str)
def test_every_wait_sees_its_own_phase(items):
    for seed in range(400):
        Model(items, seed, split=True).run()


def test_the_model_finds_a_wait_that_may_see_another_phase():
    """Completed PV announced per tile, by a commit other than the one that the next scores wait for."""
    found = 0
    for items in SHAPES:
        for seed in range(400):
            try:
                Model(items, seed, split=False).run()
            except (AssertionError, WrongPhase):
                found += 1
    assert found
