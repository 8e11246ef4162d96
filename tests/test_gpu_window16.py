"""Windows of 16 x 16 tokens (rib_window16_sm100.cu): several windows per CTA, one window, shifts, masks, windows that reach beyond
the map, every width class; every element against the numpy oracles."""
import pytest
import torch

from oracle import rib_masked_oracle, rib_padded_oracle
from paper_2603_06738_b200 import binding, synthetic
from paper_2603_06738_b200.synthetic import Workload

from parity_util import compare, to_f64

pytestmark = pytest.mark.gpu

# name, B, H, W, heads, d, r, window, shift
CASES = [
    Workload("w16_one_window", 1, 16, 16, 1, 32, 16, 16, 0, seed=501),
    Workload("w16_many_windows_s8", 1, 256, 192, 1, 32, 16, 16, 8, seed=502),               # 192 windows of one head: two per CTA
    Workload("w16_rings_wrap", 2, 64, 64, 37, 8, 8, 16, 0, seed=503),                       # 32 windows on 4 CTAs per head
    Workload("w16_headwise_d16_r24_s8", 1, 48, 32, 12, 16, 24, 16, 8, seed=504, headwise=True),
    Workload("w16_rank32", 1, 64, 96, 6, 32, 32, 16, 0, seed=505),
    Workload("w16_partial", 2, 40, 56, 3, 24, 16, 16, 0, seed=506),
    Workload("w16_partial_s8", 1, 24, 72, 6, 32, 32, 16, 8, seed=507),
    Workload("w16_patch", 1, 8, 8, 2, 32, 16, 16, 8, seed=508),                             # one patch in the middle of the extension
    Workload("w16_d24_r8_s8", 2, 32, 48, 4, 24, 8, 16, 8, seed=513),
    Workload("w16_d24_r24_s8", 1, 48, 32, 3, 24, 24, 16, 8, seed=514),
    Workload("w16_d30_r18", 1, 48, 32, 6, 30, 18, 16, 8, seed=509),                         # zero-padded copies
]


def check(wl, spread, oracle, fwd, bwd):
    cpu = synthetic.make_inputs(wl, with_dout=True)
    cpu["q"] = (cpu["q"].float() * spread).to(torch.bfloat16)
    gpu = {k: v.cuda() for k, v in cpu.items()}
    args = [gpu[k] for k in ("q", "k", "v", "pq", "pk")]
    out, lse = fwd(*args, wl.window, wl.shift)
    grads = bwd(*args, out, lse, gpu["dout"], wl.window, wl.shift)
    torch.cuda.synchronize()
    assert binding.rib_query_status() == 0 and binding.rib_last_path() == binding.RIB_PATH_SM100
    f64 = [to_f64(cpu[k]) for k in ("q", "k", "v", "pq", "pk")]
    ref_out, ref_lse = oracle.fwd(*f64, wl.window, wl.shift)
    ref = oracle.bwd(*f64, to_f64(cpu["dout"]), wl.window, wl.shift)
    # bf16 steps grow with the values (2^-8 of a value); dS is rounded to bf16 (2^-9) before sums of up to 256 products
    scale = lambda a: 1e-2 * max(1.0, float(abs(a).max()))
    compare("out", to_f64(out), ref_out, max_abs=scale(ref_out))
    compare("lse", to_f64(lse), ref_lse)
    for name, got, want in zip(("dq", "dk", "dv", "dpq", "dpk"), grads, ref):
        compare(name, to_f64(got), want, max_abs=scale(want), rel_l2=5e-3 if spread == 1.0 else 1e-2)


@pytest.mark.parametrize("spread", [1.0, 10.0], ids=["", "large_logits"])
@pytest.mark.parametrize("wl", CASES, ids=lambda w: w.name)
def test_windows_of_16(wl, spread):
    check(wl, spread, rib_padded_oracle, binding.rib_window_attn_fwd_padded, binding.rib_window_attn_bwd_padded)


@pytest.mark.parametrize("wl", [w for w in CASES if w.H % 16 == 0 and w.W % 16 == 0], ids=lambda w: w.name)
def test_masked_windows_of_16(wl):
    check(wl, 1.0, rib_masked_oracle, binding.rib_window_attn_fwd_masked, binding.rib_window_attn_bwd_masked)


@pytest.mark.parametrize("wl", [
    Workload("w16_exact_masked", 1, 48, 32, 3, 32, 32, 16, 8, seed=510),
    Workload("w16_exact_masked_headwise", 2, 32, 32, 2, 8, 32, 16, 8, seed=511, headwise=True),
    Workload("w16_exact_partial", 1, 24, 72, 6, 32, 32, 16, 8, seed=512),
], ids=lambda w: w.name)
def test_the_exact_form_is_taken_where_it_is_asked_for(wl):
    """rib_set_path(RIB_PATH_SM100_EXACT): lse from fp32 sums of unrounded exponentials, also for masks and windows beyond the map."""
    cpu = synthetic.make_inputs(wl, with_dout=False)
    args = [cpu[k].cuda() for k in ("q", "k", "v", "pq", "pk")]
    masked = wl.H % 16 == 0 and wl.W % 16 == 0
    fwd, oracle = (binding.rib_window_attn_fwd_masked, rib_masked_oracle) if masked else (binding.rib_window_attn_fwd_padded, rib_padded_oracle)
    binding.rib_set_path(binding.RIB_PATH_SM100_EXACT)
    try:
        out, lse = fwd(*args, wl.window, wl.shift)
        assert binding.rib_last_path() == binding.RIB_PATH_SM100
    finally:
        binding.rib_set_path(binding.RIB_PATH_NONE)
    torch.cuda.synchronize()
    ref_out, ref_lse = oracle.fwd(*(to_f64(cpu[k]) for k in ("q", "k", "v", "pq", "pk")), wl.window, wl.shift)
    compare("out", to_f64(out), ref_out)
    # sqrt(d / r) is a power of two here, so the scaled query rows are exact: what is left are fp32 logits and sums (2^-24 each);
    # probabilities rounded to bf16 (2^-9 each over up to 256 keys) would leave some 1e-5 of lse
    compare("lse", to_f64(lse), ref_lse, rel_l2=2e-6)
