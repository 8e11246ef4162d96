"""GPU parity for frames with a side that is no multiple of 8 (rib_fwd_frame_sm100_kernel), every element, against the numpy
oracle; the any-shape kernel, which keeps everything in fp32, is the measure of its precision."""
import numpy as np
import pytest
import torch

from oracle import rib_padded_oracle as pad
from paper_2603_06738_b200 import binding, synthetic
from paper_2603_06738_b200.synthetic import Workload

from parity_util import compare, to_f64

pytestmark = pytest.mark.gpu

# name, B, H, W, heads, d, r, window, shift
CASES = [
    Workload("f_1x1_w16", 1, 1, 1, 1, 32, 16, 16, 0, seed=201),                   # a single token
    Workload("f_7x5_w16", 2, 7, 5, 2, 32, 16, 16, 0, seed=202),                   # less than a patch
    Workload("f_9x17_w16", 2, 9, 17, 3, 32, 16, 16, 0, seed=203),                 # patches of one row and one column
    Workload("f_31x15_w16", 1, 31, 15, 2, 32, 16, 16, 0, seed=204),               # the last patch row holds 7 of 8
    Workload("f_20x28_w16_s8", 2, 20, 28, 2, 32, 16, 16, 8, seed=205),            # the extension wraps into the window's middle
    Workload("f_5x60_w32_s24", 1, 5, 60, 2, 32, 16, 32, 24, seed=206),            # fewer rows than the shift
    Workload("f_45x83_w32", 1, 45, 83, 3, 32, 16, 32, 0, seed=207),
    Workload("f_40x84_w32_s16_r32", 2, 40, 84, 2, 32, 32, 32, 16, seed=208),      # one side a multiple of 8
    Workload("f_50x70_w48_s8_d16_r24", 1, 50, 70, 3, 16, 24, 48, 8, seed=209),
    Workload("f_66x67_w64_d24_r8", 1, 66, 67, 2, 24, 8, 64, 0, seed=210),
    Workload("f_37x21_w32_headwise", 1, 37, 21, 3, 32, 16, 32, 8, seed=211, headwise=True),
    Workload("f_43x29_w16_d30_r18", 2, 43, 29, 3, 30, 18, 16, 0, seed=212),       # 60-byte rows: zero-padded copies
    Workload("f_27x99_w96_d8_r8", 1, 27, 99, 2, 8, 8, 96, 0, seed=213),
]


def run(wl, gpu, path):
    binding.rib_set_path(path)
    try:
        out, lse = binding.rib_window_attn_fwd_padded(gpu["q"], gpu["k"], gpu["v"], gpu["pq"], gpu["pk"], wl.window, wl.shift)
        used = binding.rib_last_path()
    finally:
        binding.rib_set_path(binding.RIB_PATH_NONE)
    torch.cuda.synchronize()
    assert binding.rib_query_status() == 0
    return to_f64(out), to_f64(lse), used


@pytest.mark.parametrize("spread", [1.0, 12.0], ids=["", "large_logits"])
@pytest.mark.parametrize("wl", CASES, ids=lambda w: w.name)
def test_frames_are_as_precise_as_the_any_shape_kernel(wl, spread):
    cpu = synthetic.make_inputs(wl, with_dout=False)
    cpu["q"] = (cpu["q"].float() * spread).to(torch.bfloat16)          # large logits: the running maximum moves, probabilities underflow
    gpu = {k: v.cuda() for k, v in cpu.items()}
    ref_out, ref_lse = pad.fwd(*(to_f64(cpu[k]) for k in ("q", "k", "v", "pq", "pk")), wl.window, wl.shift)
    out, lse, used = run(wl, gpu, binding.RIB_PATH_NONE)
    assert used == binding.RIB_PATH_SM100
    wide_out, wide_lse, used = run(wl, gpu, binding.RIB_PATH_GENERIC)
    assert used == binding.RIB_PATH_GENERIC
    # half a unit in the last place of bf16 is at most 2^-8 of the value; large logits pick single values out, up to 4.5 in size
    compare("out", out, ref_out, max_abs=max(1e-2, 1.02 * 2.0 ** -8 * float(np.abs(ref_out).max())))
    off = lambda a, b: float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30))
    # out is rounded to bf16 on both sides (1.7e-3 of its size); what is left of the fp32 arithmetic decides a few roundings
    assert off(out, ref_out) <= 1.02 * off(wide_out, ref_out) + 1e-6
    # lse: 48 to 64 fp32 products per logit and fp32 sums, logits of up to 12 * 6 in size: 2^-24 * sqrt(64) * a few
    assert off(lse, ref_lse) <= 2e-6, (off(lse, ref_lse), off(wide_lse, ref_lse))


def test_a_frame_beside_others_reads_and_writes_nothing_beyond_itself():
    """The batch items around a frame hold NaN: patches that straddle its border must not pick them up."""
    wl = Workload("f_20x28_nan", 3, 20, 28, 2, 32, 16, 16, 0, seed=214)
    cpu = synthetic.make_inputs(wl, with_dout=False)
    for k in ("q", "k", "v"):
        cpu[k][0] = float("nan")
        cpu[k][2] = float("nan")
    gpu = {k: v.cuda() for k, v in cpu.items()}
    out, lse, _ = run(wl, gpu, binding.RIB_PATH_NONE)
    middle = {k: cpu[k][1:2] for k in ("q", "k", "v")}
    ref_out, ref_lse = pad.fwd(*(to_f64(middle[k]) for k in ("q", "k", "v")), to_f64(cpu["pq"]), to_f64(cpu["pk"]), wl.window, 0)
    compare("out", out[1:2], ref_out)
    compare("lse", lse[1:2], ref_lse)
    assert np.isnan(out[0]).all() and np.isnan(out[2]).all()


# several items per CTA (148 SMs at most): query buffers, accumulators, score buffers and barrier phases cross from item to item
MANY = [
    Workload("f_125x203_w16", 2, 125, 203, 6, 32, 16, 16, 0, seed=215),                # 1248 items of one or two blocks
    Workload("f_77x107_w32_r32", 4, 77, 107, 6, 32, 32, 32, 0, seed=216),              # items of 1 to 8 blocks, odd patch counts, rank 32
    Workload("f_83x61_w32_s8", 6, 83, 61, 6, 32, 16, 32, 8, seed=217),
]


@pytest.mark.parametrize("wl", MANY, ids=lambda w: w.name)
def test_frames_with_many_items_per_cta(wl):
    cpu = synthetic.make_inputs(wl, with_dout=False)
    gpu = {k: v.cuda() for k, v in cpu.items()}
    ref_out, ref_lse = pad.fwd(*(to_f64(cpu[k]) for k in ("q", "k", "v", "pq", "pk")), wl.window, wl.shift)
    out, lse, used = run(wl, gpu, binding.RIB_PATH_NONE)
    assert used == binding.RIB_PATH_SM100
    compare("out", out, ref_out)
    assert np.linalg.norm(lse - ref_lse) <= 2e-6 * np.linalg.norm(ref_lse)
    for _ in range(3):                                   # no sum's order depends on timing
        again, lse_again, _ = run(wl, gpu, binding.RIB_PATH_NONE)
        assert np.array_equal(out, again) and np.array_equal(lse, lse_again)


@pytest.mark.parametrize("what", ["v", "k", "pk", "pq", "pq_all"])
@pytest.mark.parametrize("shape", [(20, 28, 32, 16, 16), (45, 27, 32, 32, 32), (20, 28, 30, 18, 16)], ids=lambda s: "x".join(map(str, s)))
def test_infinities_come_out_as_from_the_any_shape_kernel(shape, what):
    """One infinite (or -inf) entry: NaN, inf and -inf at the same places as from the fp32 kernel, finite values beside them."""
    H, W, d, r, window = shape
    wl = Workload("f_inf", 2, H, W, 2, d, r, window, 0, seed=218)
    cpu = synthetic.make_inputs(wl, with_dout=False)
    inf = float("inf")
    if what in ("v", "k"):
        for y, x, c, value in ((0, 1, 3, inf), (H - 1, W - 1, 5, -inf)):      # the last patch as well: it may fill half a key block
            cpu[what][1, y, x, 1, c] = value
    elif what == "pk":
        cpu["pk"][window + 1, 2], cpu["pk"][3, 4] = inf, -inf
    else:
        cpu["pq"][window + 2, 3] = -inf
        if what == "pq_all":                                                  # every logit of that row is -inf
            cpu["pk"][:, 3] = cpu["pk"][:, 3].abs() + 0.5
    gpu = {k: v.cuda() for k, v in cpu.items()}
    out, lse, used = run(wl, gpu, binding.RIB_PATH_NONE)
    wide_out, wide_lse, _ = run(wl, gpu, binding.RIB_PATH_GENERIC)
    assert used == binding.RIB_PATH_SM100 and not (np.isfinite(wide_out).all() and np.isfinite(wide_lse).all())
    for got, want in ((out, wide_out), (lse, wide_lse)):
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert np.array_equal(np.isposinf(got), np.isposinf(want)) and np.array_equal(np.isneginf(got), np.isneginf(want))
        fine = np.isfinite(want)                 # the roundings to bf16 that the order of an fp32 sum decides: one step of values up to 2
        compare("finite values", got[fine], want[fine], max_abs=2.0 ** -7, rel_l2=3e-4)


@pytest.mark.parametrize("wl", [CASES[6], CASES[8], MANY[0], MANY[2]], ids=lambda w: w.name)
def test_lse_of_frames_is_no_further_off_than_from_the_any_shape_kernel(wl):
    cpu = synthetic.make_inputs(wl, with_dout=False)
    gpu = {k: v.cuda() for k, v in cpu.items()}
    _, ref = pad.fwd(*(to_f64(cpu[k]) for k in ("q", "k", "v", "pq", "pk")), wl.window, wl.shift)
    off = [np.linalg.norm(run(wl, gpu, path)[1] - ref) / np.linalg.norm(ref) for path in (binding.RIB_PATH_NONE, binding.RIB_PATH_GENERIC)]
    print(f"lse: relative error {off[0]:.3e}, any-shape kernel {off[1]:.3e}")
    assert off[0] <= off[1], off
