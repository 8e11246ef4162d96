"""The waits of the general forward kernel (csrc/rib_fwd_sm100.cu) in the model of tests/test_frame_barriers.py: the same buffers and
barriers, but an item's output is read inside the next item's first block, before P of that block is handed over.  No GPU needed."""
import pytest

from test_frame_barriers import SHAPES, Model


class Deferred(Model):
    def softmax(self, tile, half):
        block = 0
        for block, j, n in self.blocks():
            u = 2 * block + tile
            yield ("wait", *self.score_phase(tile, block))
            assert ("s", u) in self.finished
            yield "delay", self.delay("soft")
            if j == 0 and block:
                yield ("wait", *self.pv_phase(tile, block - 1))
                assert ("pv", u - 2) in self.finished and ("pv", u) not in self.issued
            self.finished.add(("p", u, half))
            self.arrive(("pready", tile, block & 1), 2)
        yield ("wait", *self.pv_phase(tile, block))
        assert ("pv", 2 * block + tile) in self.finished


@pytest.mark.parametrize("items", SHAPES, ids=str)
def test_every_wait_sees_its_own_phase(items):
    for seed in range(400):
        Deferred(items, seed, split=True).run()
