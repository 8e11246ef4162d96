"""The general forward kernel's three score buffers rotate over blocks, items and passes: windows of 1 to 18 key blocks, several items
per CTA, both softmax forms, and a second pass that begins wherever the first one left the buffers."""
import numpy as np
import pytest
import torch

from oracle import rib_padded_oracle as pad
from paper_2603_06738_b200 import binding, synthetic
from paper_2603_06738_b200.synthetic import Workload

from parity_util import compare, make, oracle_fwd, run_fwd, to_f64

pytestmark = pytest.mark.gpu

CASES = [
    Workload("b_w16", 1, 128, 128, 5, 32, 16, 16, 8, seed=301),              # 2 blocks, 320 items: 2 or 3 per CTA
    Workload("b_w32_r32", 2, 96, 96, 3, 32, 32, 32, 0, seed=302),            # 8 blocks
    Workload("b_w48", 1, 96, 96, 2, 16, 8, 48, 24, seed=303),                # 18 blocks
    Workload("b_40x104_w32", 3, 40, 104, 3, 32, 16, 32, 0, seed=304),        # 1 (half of it without keys), 2, 4 and 8 blocks
    Workload("b_24x56_w48", 2, 24, 56, 3, 24, 24, 48, 0, seed=305),          # 2 and 9 blocks
]


@pytest.mark.parametrize("form", ["fast", "exact", "redone"])
@pytest.mark.parametrize("wl", CASES, ids=lambda w: w.name)
def test_every_element(wl, form):
    cpu, gpu = make(wl, with_dout=False)
    if form == "redone":                      # keys of every third window row and column 200 nat from the rest: some items are redone
        cpu["k"][:, ::3 * wl.window // 2, ::3 * wl.window // 2] *= 220.0
        gpu = {k: v.cuda() for k, v in cpu.items()}
    binding.rib_set_path(binding.RIB_PATH_SM100_EXACT if form == "exact" else binding.RIB_PATH_NONE)
    try:
        if wl.H % wl.window or wl.W % wl.window:
            out, lse = binding.rib_window_attn_fwd_padded(gpu["q"], gpu["k"], gpu["v"], gpu["pq"], gpu["pk"], wl.window, wl.shift)
            ref_out, ref_lse = pad.fwd(*(to_f64(cpu[k]) for k in ("q", "k", "v", "pq", "pk")), wl.window, wl.shift)
        else:
            out, lse = run_fwd(gpu, wl)
            ref_out, ref_lse = oracle_fwd(cpu, wl)
        assert binding.rib_last_path() == binding.RIB_PATH_SM100
    finally:
        binding.rib_set_path(binding.RIB_PATH_NONE)
    torch.cuda.synchronize()
    assert binding.rib_query_status() == 0
    # (bounds of redone items as in test_scores_beyond_the_fast_softmax_range_are_redone_exactly)
    far = form == "redone"
    if far:
        assert np.abs(ref_lse).max() > 100
    compare("out", to_f64(out), ref_out, max_abs=2e-2 if far else 1e-2)
    compare("lse", to_f64(lse), ref_lse, max_abs=2e-2 * max(1.0, np.abs(ref_lse).max() / 100) if far else 1e-2)


@pytest.mark.parametrize("d", [16, 32])
def test_an_output_that_is_aligned_to_16_bytes_only(d):
    """Rows of out leave as 32-byte sectors where they are such; elsewhere the same bits, and nothing beyond them."""
    wl = Workload("b_align", 1, 64, 64, 2, d, 16, 32, 8, seed=306)
    _, gpu = make(wl, with_dout=False)
    args = [gpu[k] for k in ("q", "k", "v", "pq", "pk")]
    expected, _ = binding.rib_window_attn_fwd(*args, wl.window, wl.shift)
    n = expected.numel()
    memory = torch.full((n + 64,), 3.0, dtype=torch.bfloat16, device="cuda")
    out = memory[8:8 + n].view(expected.shape)
    assert out.data_ptr() % 32 == 16
    binding.rib_window_attn_fwd(*args, wl.window, wl.shift, out=out)
    torch.cuda.synchronize()
    assert torch.equal(out, expected)
    assert (memory[:8] == 3.0).all() and (memory[8 + n:] == 3.0).all()
