"""The feature generator at the edges of its blocks (16 tokens) and of its 4-column pieces, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import rib_generator_oracle as gen
from paper_2603_06738_b200 import binding

pytestmark = pytest.mark.gpu


# window, L, dh, r: one token short of a block, exactly one, several with a remainder; widths that are no multiple of 4
@pytest.mark.parametrize("window,L,dh,r", [(3, 2, 5, 7), (4, 1, 4, 4), (5, 6, 33, 18), (9, 16, 63, 1), (64, 12, 48, 18)])
def test_generator_edges(window, L, dh, r):
    rng = np.random.default_rng(window + L)
    ws = [np.float32(rng.normal(0, 0.3, s)) for s in ((2 + 4 * L, dh), (dh,), (dh, r), (dh, r))]
    grads = [np.float32(rng.normal(size=(window * window, r))) for _ in range(2)]
    gw, gg = [torch.from_numpy(w).cuda() for w in ws], [torch.from_numpy(g).cuda() for g in grads]
    ref = gen.forward(*ws, window, L)[:2] + gen.backward(*ws, *grads, window, L)
    for _ in range(3):                              # the gradients start from zero on every call
        got = binding.rib_generate_features(*gw, window) + binding.rib_generate_features_bwd(*gw, *gg, window)
    for i, (g, want) in enumerate(zip(got, ref)):
        g = g.double().cpu().numpy()
        # features are rounded to bf16 (2^-9 of a value); gradients are fp32 sums of up to 4096 terms
        assert np.linalg.norm(g - want) <= (3e-3 if i < 2 else 2e-6) * np.linalg.norm(want), i
