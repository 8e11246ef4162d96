"""The gate's backward at the edges of its tiles: 16 x 16 pixels in the depth-wise part, 128 consecutive pixels in the point-wise part, whose
filter takes runs of 8 or 16 pixels where the width of the map is a multiple of that, else pairs."""
import numpy as np
import pytest
import torch

from oracle import cla_oracle as cla
from paper_2603_06738_b200 import binding, synthetic

from parity_util import compare, to_f64

pytestmark = pytest.mark.gpu


def inputs(B, H, W, D):
    x = synthetic.bf16_tensor(320 + H, "x", (B, H, W, D), 1.0)
    dgate = synthetic.bf16_tensor(321 + W, "gate", (B, H, W, D), 1.0)
    rng = np.random.default_rng(322)
    ws = [np.float32(rng.normal(0, s, shape)) for s, shape in ((0.35, (D, 3, 3)), (0.2, D), (1.5 / np.sqrt(D), (D, D)), (0.3, D))]
    return x, ws, dgate


@pytest.mark.parametrize("B,H,W,D", [(2, 15, 17, 64), (1, 17, 15, 128), (1, 16, 33, 192), (2, 33, 16, 64), (1, 1, 49, 64), (1, 49, 1, 64),
                                     (3, 31, 31, 128)])
def test_edges_of_tiles(B, H, W, D):
    x, ws, dgate = inputs(B, H, W, D)
    binding.rib_set_path(binding.RIB_PATH_GENERIC)          # the point-wise part in fp32, so that what is left is this part's own error
    try:
        got = binding.rib_cla_gate_bwd(x.cuda(), *[torch.from_numpy(w).cuda() for w in ws], dgate.cuda())
    finally:
        binding.rib_set_path(binding.RIB_PATH_NONE)
    torch.cuda.synchronize()
    assert binding.rib_query_status() == 0
    ref = cla.gate_bwd(to_f64(x), *ws, to_f64(dgate))
    # dx: one rounding to bf16 (half a step, 2^-9 of the value) beside fp32 arithmetic; sums of fp32 products over at most 2883 pixels
    compare("dx", to_f64(got[0]), ref[0], max_abs=2.0 ** -8 * max(1.0, np.abs(ref[0]).max()), rel_l2=2.0 ** -8)
    for name, g, r in zip(("dw_dw", "db_dw"), got[1:3], ref[1:3]):
        compare(name, to_f64(g), r, max_abs=1e-3 * max(1.0, np.abs(r).max()), rel_l2=1e-4)


@pytest.mark.parametrize("B,H,W,D", [(1, 1, 8, 64), (1, 3, 16, 192), (3, 7, 24, 128), (2, 5, 48, 192), (1, 9, 24, 192), (2, 11, 16, 64), (5, 33, 32, 192)])
def test_runs_of_pixels(B, H, W, D):
    x, ws, dgate = inputs(B, H, W, D)
    got = binding.rib_cla_gate_bwd(x.cuda(), *[torch.from_numpy(w).cuda() for w in ws], dgate.cuda())
    assert binding.rib_last_path() == binding.RIB_PATH_SM100
    torch.cuda.synchronize()
    assert binding.rib_query_status() == 0
    ref = cla.gate_bwd(to_f64(x), *ws, to_f64(dgate))
    # Y, dZ and the point-wise matrix enter the MMAs as bf16: the bounds of test_gate_backward_matches_the_oracle
    for name, g, r in zip(("dx", "dw_dw", "db_dw", "dw_pw", "db_pw"), got, ref):
        compare(name, to_f64(g), r, max_abs=1e-2 * max(1.0, np.abs(r).max()), rel_l2=5e-3)
