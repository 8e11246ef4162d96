"""Rows that TMA cannot address (even head widths and ranks that are no multiples of 8), windows of the general kernels: every
remainder of a 16-byte piece that the row copies, the preparation and the finishing kernel meet, against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import rib_padded_oracle as padded
from paper_2603_06738_b200 import binding
from paper_2603_06738_b200.synthetic import Workload

from parity_util import compare, make, oracle_bwd, oracle_fwd, run_bwd, run_fwd, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,r,headwise", [(2, 18, False), (4, 8, True), (6, 30, False), (10, 2, False), (12, 16, True), (18, 32, False),
                                          (26, 20, True), (28, 22, False), (30, 18, False), (32, 18, False)])
def test_every_remainder_of_a_row(d, r, headwise):
    wl = Workload(f"narrow_d{d}_r{r}", 1, 32, 96, 3, d, r, 32, 8, seed=500 + d, headwise=headwise)
    cpu, gpu = make(wl, with_dout=True)
    out, lse = run_fwd(gpu, wl)
    assert binding.rib_last_path() == binding.RIB_PATH_SM100
    grads = run_bwd(gpu, wl, out, lse)
    assert binding.rib_last_path() == binding.RIB_PATH_SM100
    ref_out, ref_lse = oracle_fwd(cpu, wl)
    compare("out", to_f64(out), ref_out)
    compare("lse", to_f64(lse), ref_lse)
    for name, got, ref in zip(("dq", "dk", "dv", "dpq", "dpk"), grads, oracle_bwd(cpu, wl)):
        # a bf16 result of size x is spaced 2^-7 x apart: the absolute bound follows the largest entry, the relative one is the usual
        compare(name, to_f64(got), ref, max_abs=1e-2 * max(1.0, float(np.abs(ref).max())))


GUARD = 256                # elements behind each result that nothing may write


def guarded(shape, dtype):
    """A tensor of NaN of the given shape (one row of it per leading index) and the memory behind it, NaN as well."""
    flat = torch.full((int(np.prod(shape)) + GUARD,), float("nan"), dtype=dtype, device="cuda")
    return flat[:-GUARD].view(shape), flat[-GUARD:]


def tables_apart(t, heads, stride):
    """The head-wise tables `t` with their beginnings `stride` elements apart, NaN between them."""
    apart = torch.full((heads, stride), float("nan"), dtype=t.dtype, device="cuda")
    apart[:, :t[0].numel()] = t.reshape(heads, -1)
    return apart


def both_passes(wl, gpu, gap):
    """Both passes through the C entry points of maps that the windows may reach beyond, head-wise tables `gap` elements further apart
    than they are long.  Returns out, lse, dq, dk, dv, dpq, dpk, after looking at what lies behind and between the results."""
    lib, n, r = binding.library(), wl.n, wl.r
    stride = (n * r + gap) if wl.headwise else 0
    pq, pk = (tables_apart(gpu[k], wl.heads, stride) if wl.headwise else gpu[k] for k in ("pq", "pk"))
    image, dims = (wl.B, wl.H, wl.W, wl.heads, wl.d), (wl.B, wl.H, wl.W, wl.heads, wl.d, r, wl.window, wl.shift)
    res = [guarded(image, torch.bfloat16) for _ in range(4)]                       # out, dq, dk, dv
    lse = guarded((wl.B, wl.heads, wl.H, wl.W), torch.float32)
    tables = [guarded((wl.heads, stride) if wl.headwise else (n, r), torch.float32) for _ in range(2)]
    ptr, stream = lambda t: t.data_ptr(), torch.cuda.current_stream().cuda_stream
    inputs = [ptr(gpu["q"]), ptr(gpu["k"]), ptr(gpu["v"]), ptr(pq), ptr(pk), stride]
    assert lib.rib_window_attn_fwd_padded(*inputs, *dims, ptr(res[0][0]), ptr(lse[0]), stream) == 0
    assert binding.rib_last_path() == binding.RIB_PATH_SM100
    ws = torch.empty(lib.rib_window_attn_bwd_padded_workspace(stride, *dims[:-1]), dtype=torch.uint8, device="cuda")
    assert lib.rib_window_attn_bwd_padded(*inputs, ptr(res[0][0]), ptr(lse[0]), ptr(gpu["dout"]), *dims, *(ptr(t) for t, _ in res[1:]),
                                          *(ptr(t) for t, _ in tables), ptr(ws), ws.numel(), stream) == 0
    assert binding.rib_last_path() == binding.RIB_PATH_SM100
    torch.cuda.synchronize()
    assert binding.rib_query_status() == 0
    for _, behind in (*res, lse, *tables):
        assert bool(torch.isnan(behind).all())
    sums = [t for t, _ in tables]
    if wl.headwise:
        assert all(bool(torch.isnan(t[:, n * r:]).all()) for t in sums)
        sums = [t[:, :n * r].reshape(wl.heads, n, r) for t in sums]
    return [to_f64(t) for t in (res[0][0], lse[0], *(t for t, _ in res[1:]), *sums)]


@pytest.mark.parametrize("H,W,heads,d,r,window,shift,headwise", [
    (72, 88, 3, 30, 18, 32, 16, False),        # windows reach beyond the map: positions that are no tokens, out and dq in the caller's rows
    (72, 88, 3, 10, 20, 32, 16, True),
    (40, 56, 3, 26, 16, 48, 24, False),        # one window; the rank is a multiple of 8, the head is not
    (72, 40, 2, 24, 18, 32, 8, True),          # the head is a multiple of 8, the rank is not
    (88, 40, 2, 2, 2, 32, 0, False),
])
def test_rows_on_maps_that_windows_reach_beyond(H, W, heads, d, r, window, shift, headwise):
    wl = Workload(f"narrow_{H}x{W}_d{d}_r{r}", 1, H, W, heads, d, r, window, shift, seed=600 + d, headwise=headwise)
    cpu, gpu = make(wl, with_dout=True)
    got = both_passes(wl, gpu, gap=0)
    ins = [to_f64(cpu[k]) for k in ("q", "k", "v", "pq", "pk", "dout")]
    ref = [*padded.fwd(*ins[:5], window, shift), *padded.bwd(*ins, window, shift)]
    for name, a, b in zip(("out", "lse", "dq", "dk", "dv", "dpq", "dpk"), got, ref):
        compare(name, a, b, max_abs=1e-2 * max(1.0, float(np.abs(b).max())))          # (as above)


@pytest.mark.parametrize("H,W", [(64, 96), (72, 88)])
@pytest.mark.parametrize("d,r", [(30, 18), (12, 16), (32, 22)])
def test_head_wise_tables_further_apart_than_they_are_long(H, W, d, r):
    """The tables are copied one by one then; what lies between them is neither read nor written, and the results are those of tables
    without gaps: forward bit for bit, sums of the backward up to the order of their additions."""
    wl = Workload(f"narrow_gaps_d{d}_r{r}", 1, H, W, 3, d, r, 32, 8, seed=700 + d, headwise=True)
    cpu, gpu = make(wl, with_dout=True)
    apart, packed = both_passes(wl, gpu, gap=64), both_passes(wl, gpu, gap=0)
    for name, a, b in zip(("out", "lse", "dk", "dv"), (apart[i] for i in (0, 1, 3, 4)), (packed[i] for i in (0, 1, 3, 4))):
        assert np.array_equal(a, b), name
    for name, a, b in zip(("dq", "dpq", "dpk"), (apart[i] for i in (2, 5, 6)), (packed[i] for i in (2, 5, 6))):
        # fp32 sums of at most 8 key blocks and 9 windows, each to 2^-24 of its terms; dq is rounded to bf16 behind that, where a
        # last place is 2^-8 of the value: few roundings differ
        compare(name, a, b, max_abs=2.0 ** -7 * float(np.abs(b).max()), rel_l2=1e-3 if name == "dq" else 1e-5)
