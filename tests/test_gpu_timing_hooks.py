"""The timing interface names the kernel that ran and brackets every launch of the attention and generator calls."""
import pytest
import torch

from paper_2603_06738_b200 import binding, synthetic
from paper_2603_06738_b200.synthetic import Workload

pytestmark = pytest.mark.gpu

GENERAL = ["rib_bwd_prepare_kernel", "rib_bwd_sm100_kernel", "rib_bwd_finish_kernel"]
WIN16 = ["rib_window16_clear_kernel", "rib_window16_clear_kernel", "rib_window16_bwd_kernel"]

# H, W, window, shift, the forward kernel, the backward kernels
CASES = [
    (32, 32, 32, 0, "rib_fwd_sm100_kernel", GENERAL),
    (32, 48, 8, 0, "rib_window8_fwd_kernel", ["rib_window8_clear_kernel", "rib_window8_bwd_kernel"]),
    (32, 48, 16, 8, "rib_fwd_sm100_kernel", WIN16),
    (40, 24, 16, 0, "rib_window16_fwd_kernel", WIN16),
    (41, 23, 16, 0, "rib_fwd_frame_sm100_kernel", ["rowdot_kernel", "generic_bwd_dq_kernel", "generic_bwd_dkv_kernel"]),
]


def bracketed(call):
    binding.rib_profile_begin(16)
    before = binding.rib_kernel_launches()
    result = call()
    launched = binding.rib_kernel_launches() - before
    entries = binding.rib_profile_end(16)
    assert len(entries) == launched and all(0.0 < ms < 1000.0 for _, ms in entries)
    return result, [binding.KERNEL_NAMES[k] for k, _ in entries]


@pytest.mark.parametrize("H,W,window,shift,forward,backward", CASES)
def test_every_launch_is_bracketed_under_its_own_name(H, W, window, shift, forward, backward):
    cpu = synthetic.make_inputs(Workload("hooks", 1, H, W, 2, 32, 16, window, shift, seed=701), with_dout=True)
    gpu = {k: v.cuda() for k, v in cpu.items()}
    args = [gpu[k] for k in ("q", "k", "v", "pq", "pk")]
    (out, lse), names = bracketed(lambda: binding.rib_window_attn_fwd_padded(*args, window, shift))
    assert names == [forward]
    _, names = bracketed(lambda: binding.rib_window_attn_bwd_padded(*args, out, lse, gpu["dout"], window, shift))
    assert names == backward


def test_the_generator_backward_is_two_launches():
    ws = [torch.randn(s, device="cuda") for s in ((42, 32), (32,), (32, 16), (32, 16))]
    grads = [torch.randn(256, 16, device="cuda") for _ in range(2)]
    _, names = bracketed(lambda: binding.rib_generate_features_bwd(*ws, *grads, 16))
    assert names == ["rib_generator_clear_kernel", "rib_generator_bwd_kernel"]


@pytest.mark.parametrize("H,W,r,masked,kernel", [
    (128, 128, 16, False, "rib_fwd_sm100_kernel"),                  # whole windows
    (128, 128, 16, True, "rib_window16_fwd_kernel"),
    (120, 136, 16, False, "rib_window16_fwd_kernel"),               # 8 x 9 windows, 8 heads: 576 pairs
    (120, 152, 16, False, "rib_fwd_sm100_kernel"),                  # 8 x 10: 640
    (120, 152, 32, False, "rib_window16_fwd_kernel"),
])
def test_the_forward_kernel_of_windows_of_16(H, W, r, masked, kernel):
    cpu = synthetic.make_inputs(Workload("rule", 1, H, W, 8, 32, r, 16, 8, seed=702), with_dout=False)
    args = [cpu[k].cuda() for k in ("q", "k", "v", "pq", "pk")]
    fwd = binding.rib_window_attn_fwd_masked if masked else binding.rib_window_attn_fwd_padded
    (out, lse), names = bracketed(lambda: fwd(*args, 16, 8))
    assert names == [kernel]
    binding.rib_set_path(binding.RIB_PATH_SM100_EXACT)              # the other kernel agrees: two bf16 roundings of values up to 4
    try:
        other, other_lse = fwd(*args, 16, 8)
    finally:
        binding.rib_set_path(binding.RIB_PATH_NONE)
    assert (out.float() - other.float()).abs().max() <= 2.0 ** -6 and (lse - other_lse).abs().max() <= 2e-3
