"""The waits of the backward kernel for windows of 16 x 16 (csrc/rib_window16_sm100.cu) in a model of its warps with random delays
(tests/test_frame_barriers.py: a wait answers by parity, so its phase must be the one that is complete).  Copies in and out end at times of their
own; every role of several warps is two processes.  Unit u = 4 * window + 2 * key block + query tile.  No GPU needed."""
import heapq

import pytest

from test_frame_barriers import Model

WARPS = (0, 1)           # of a role of several warps


class Backward(Model):
    """A CTA with `windows` windows.  `fault`: a rule left out."""

    def __init__(self, windows, seed, fault=None):
        super().__init__([], seed, True)
        self.windows, self.units, self.fault = windows, 4 * windows, fault
        for name in ("grad", "drain", "load", "scalars"):
            self.scale[name] = self.rng.choice((0.1, 1.0, 5.0))
        self.scale["store"] = self.rng.choice((0.1, 1.0, 30.0))
        self.counts = dict.fromkeys(("sfree", "pready", "sready", "ldfree", "ld", "kvfree", "qfree", "vote"), len(WARPS))

    def arrive(self, bar, count=1):
        super().arrive(bar, self.counts.get(bar if isinstance(bar, str) else bar[0], 1))

    def all_done(self, *what):
        return all((*what, w) in self.finished for w in WARPS)

    def copy(self, name, what, bar):
        self.issued.add(what)

        def complete():
            self.finished.add(what)
            self.arrive(bar)
        self.later(self.delay(name), complete)

    def producer(self):
        for t in range(self.windows):
            if t >= 2:
                yield "wait", ("empty", t & 1), (t >> 1) - 1
                old = range(4 * (t - 2), 4 * (t - 1))
                assert all((kind, u) in self.finished for u in old for kind in ("s", "dv", "dk")) and self.all_done("ld", t - 2), "rows in use"
                assert ("out", t - 2, 0) in self.finished and ("out", t - 2, 1) in self.finished, "rows of gradients on their way out"
            self.copy("load", ("window", t), ("full", t & 1))

    def scores(self):
        for u in range(self.units):
            if u % 4 == 0:
                yield "wait", ("full", u >> 2 & 1), u >> 3
            if u:
                yield "wait", "sfree", u - 1
                assert self.all_done("read", u - 1)
            assert ("window", u >> 2) in self.finished
            yield "delay", self.delay("s")
            self.contract("s", ("s", u), ["sfull"])

    def gradients(self):
        for u in range(self.units):
            yield "wait", "pready", u
            assert self.all_done("p", u)
            if u % 2 == 0:
                yield "wait", "kvfree", u >> 1
                assert u == 0 or self.all_done("kv", (u >> 1) - 1), "dV, dK~ of the block before have not been read"
            yield "delay", self.delay("grad")
            self.contract("grad", ("dv", u), ["pdone"])
            yield "wait", "sready", u
            assert self.all_done("ds", u)
            if u % 4 == 0:
                yield "wait", "qfree", u >> 2
                assert u == 0 or self.all_done("q", (u >> 2) - 1), "dQ~ of the window before has not been read"
            yield "delay", self.delay("grad")
            self.contract("grad", ("dk", u), ["sdone"] + (["acc"] if u % 2 else []))

    def arithmetic(self, warp):
        for u in range(self.units):
            t = u >> 2
            if u % 4 == 0:
                yield "wait", ("ld", t & 1), t >> 1
                assert self.all_done("ld", t)
            yield "wait", "sfull", u
            assert ("s", u) in self.finished and ("s", u + 1) not in self.issued
            yield "delay", self.delay("soft")
            assert not any(("ld", t + 2, w) in self.finished for w in WARPS), "scalars overwritten"
            self.finished.add(("read", u, warp))
            self.arrive("sfree")
            if u % 4 == 0:
                self.arrive("ldfree")
            yield "delay", self.delay("soft")
            if u:
                yield "wait", "pdone", u - 1
                assert ("dv", u - 1) in self.finished
            self.finished.add(("p", u, warp))
            self.arrive("pready")
            if u:
                yield "wait", "sdone", u - 1
                assert ("dk", u - 1) in self.finished
            self.finished.add(("ds", u, warp))
            self.arrive("sready")

    def scalars(self, warp):
        for t in range(self.windows):
            if self.fault != "scalars":              # (the window's arrival alone would do: its stage is refilled after window t - 2)
                if t >= 1:
                    yield "wait", "ldfree", t - 1
                yield "delay", self.delay("scalars")
                yield "wait", ("full", t & 1), t >> 1
                assert ("window", t) in self.finished and ("window", t + 2) not in self.issued, "dO of another window"
            yield "delay", self.delay("scalars")
            assert t < 2 or self.all_done("read", 4 * (t - 2) + 3), "scalars of a window that is still worked on"
            assert ("window", t + 2) not in self.issued
            self.finished.add(("ld", t, warp))
            self.arrive(("ld", t & 1))

    def drain(self, warp):
        self.arrive("kvfree")
        self.arrive("qfree")
        for t in range(self.windows):
            for J in range(2):
                u = 4 * t + 2 * J + 1
                yield "wait", "acc", 2 * t + J
                assert ("dk", u) in self.finished and ("dv", u) in self.finished and ("dv", u + 1) not in self.issued
                yield "delay", self.delay("drain")
                # rows of dK go over those of K, whose scores and dQ~ are done; rows of dQ over those of Q
                assert all(("s", v) in self.finished and ("dk", v) in self.finished for v in range(u - 1 if J == 0 else u - 3, u + 1))
                assert ("window", t + 2) not in self.issued
                self.finished.add(("kv", 2 * t + J, warp))
                self.arrive("kvfree")
                yield "delay", self.delay("drain")
                if J == 1:
                    self.finished.add(("q", t, warp))
                    self.arrive("qfree")
                self.finished.add(("staged", t, J, warp))
                if self.fault != "vote":
                    self.arrive("vote")
                    yield "wait", "vote", 2 * t + J
                if warp == 0:                        # its thread stores the rows of all
                    assert self.all_done("staged", t, J) and ("window", t + 2) not in self.issued, "rows that are not there yet"
                    self.copy("store", ("out", t, J), "group")
                    if J == 1:
                        yield "group", 2 * t + 2
                        self.arrive(("empty", t & 1))

    def wait_group(self, process, stores):
        """Stores end in any order: asked for again until all are read."""
        if self.done.get("group", 0) >= stores:
            self.later(0.0, lambda: self.step(process))
        else:
            self.later(0.1, lambda: self.wait_group(process, stores))

    def step(self, process):
        try:
            what = next(process)
        except StopIteration:
            return
        if what[0] == "group":
            self.wait_group(process, what[1])
        elif what[0] == "delay":
            self.later(what[1], lambda: self.step(process))
        else:
            self.wait(process, *what[1:])

    def run(self):
        self.pipe = {}
        processes = [self.producer(), self.scores(), self.gradients()]
        for w in WARPS:
            processes += [self.arithmetic(w), self.scalars(w), self.drain(w)]
        for process in processes:
            self.later(self.delay("soft"), lambda process=process: self.step(process))
        while self.queue:
            self.now, _, what = heapq.heappop(self.queue)
            what()
        assert sum(f[0] == "out" for f in self.finished) == 2 * self.windows, "the warps wait for one another"


@pytest.mark.parametrize("windows", [1, 2, 3, 8, 25])
def test_every_wait_sees_its_own_phase(windows):
    for seed in range(200):
        Backward(windows, seed).run()


@pytest.mark.parametrize("fault", ["vote", "scalars"])
def test_the_model_finds_a_rule_that_is_left_out(fault):
    """vote: rows stored without the barrier of the warps that stage them.  scalars: their columns refilled without a look at the windows
    under way (dO from global memory, say)."""
    found = 0
    for windows in (3, 8):
        for seed in range(200):
            try:
                Backward(windows, seed, fault).run()
            except AssertionError:
                found += 1
    assert found
