"""Windows of 8 x 8 tokens (rib_window8_sm100.cu): more tiles than stages and CTAs, one tile, head-wise tables, every width class, many
heads; every element against the C oracle."""
import pytest
import torch

from oracle import rib_oracle
from paper_2603_06738_b200 import binding, synthetic
from paper_2603_06738_b200.synthetic import Workload

from parity_util import compare, to_f64

pytestmark = pytest.mark.gpu

# name, B, H, W, heads, d, r, window, shift
CASES = [
    Workload("w8_one_window_pair_row", 1, 16, 16, 1, 32, 16, 8, 0, seed=401),
    Workload("w8_many_tiles_one_head", 3, 160, 160, 1, 32, 16, 8, 0, seed=402),            # 600 tiles on one head: several per CTA
    Workload("w8_six_heads", 4, 96, 96, 6, 32, 16, 8, 0, seed=403),                        # rings wrap round
    Workload("w8_headwise_d16_r24", 2, 64, 48, 12, 16, 24, 8, 0, seed=404, headwise=True),
    Workload("w8_d24_r8", 1, 32, 112, 4, 24, 8, 8, 0, seed=405),
    Workload("w8_d8_r32", 2, 48, 16, 5, 8, 32, 8, 0, seed=406),
    Workload("w8_d30_r18", 1, 48, 48, 6, 30, 18, 8, 0, seed=407),                          # zero-padded copies
    Workload("w8_more_heads_than_sms", 1, 16, 32, 160, 8, 8, 8, 0, seed=408),
]


@pytest.mark.parametrize("spread", [1.0, 10.0], ids=["", "large_logits"])
@pytest.mark.parametrize("wl", CASES, ids=lambda w: w.name)
def test_windows_of_8(wl, spread):
    cpu = synthetic.make_inputs(wl, with_dout=True)
    cpu["q"] = (cpu["q"].float() * spread).to(torch.bfloat16)
    gpu = {k: v.cuda() for k, v in cpu.items()}
    args = [gpu[k] for k in ("q", "k", "v", "pq", "pk")]
    fwd, bwd = ((binding.rib_window_attn_fwd_headwise, binding.rib_window_attn_bwd_headwise) if wl.headwise
                else (binding.rib_window_attn_fwd, binding.rib_window_attn_bwd))
    out, lse = fwd(*args, wl.window, wl.shift)
    grads = bwd(*args, out, lse, gpu["dout"], wl.window, wl.shift)
    torch.cuda.synchronize()
    assert binding.rib_query_status() == 0 and binding.rib_last_path() == binding.RIB_PATH_SM100
    f64 = [to_f64(cpu[k]) for k in ("q", "k", "v", "pq", "pk")]
    ref_out, ref_lse = rib_oracle.fwd(*f64, wl.window, wl.shift)
    ref = rib_oracle.bwd(*f64, to_f64(cpu["dout"]), wl.window, wl.shift)
    # rows average over 64 keys only: values of a few units, whose bf16 steps grow with them (2^-8 of a value), and gradients
    # that are sums of 64 products with dS rounded to bf16 (2^-9 each)
    scale = lambda a: 1e-2 * max(1.0, float(abs(a).max()))
    compare("out", to_f64(out), ref_out, max_abs=scale(ref_out))
    compare("lse", to_f64(lse), ref_lse)
    for name, got, want in zip(("dq", "dk", "dv", "dpq", "dpk"), grads, ref):
        compare(name, to_f64(got), want, max_abs=scale(want), rel_l2=5e-3 if spread == 1.0 else 1e-2)
    none = fwd(*args, wl.window, wl.shift, want_lse=False)
    assert none[1] is None and torch.equal(none[0], out)
