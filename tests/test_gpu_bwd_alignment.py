"""Rows of dq and dv leave as 32-byte sectors where they are such: gradients that begin 16 bytes beside a sector have the same values,
and nothing around them is written."""
import pytest
import torch

from paper_2603_06738_b200 import binding
from paper_2603_06738_b200.synthetic import Workload

from parity_util import make, run_fwd

pytestmark = pytest.mark.gpu

CASES = [
    Workload("a_w32_d32", 1, 64, 64, 3, 32, 16, 32, 8, seed=311),
    Workload("a_w32_d16_r24", 1, 64, 64, 2, 16, 24, 32, 0, seed=312),
    Workload("a_w16_d32", 1, 64, 64, 3, 32, 16, 16, 8, seed=313),
    Workload("a_w16_d16_r24", 1, 64, 64, 2, 16, 24, 16, 0, seed=314),
    Workload("a_w16_d24", 1, 64, 64, 2, 24, 8, 16, 0, seed=315),             # rows of 48 bytes: never sectors
]


@pytest.mark.parametrize("wl", CASES, ids=lambda w: w.name)
def test_gradients_that_are_aligned_to_16_bytes_only(wl):
    _, gpu = make(wl)
    q, k, v, pq, pk, dout = (gpu[name] for name in ("q", "k", "v", "pq", "pk", "dout"))
    out, lse = run_fwd(gpu, wl)
    expected = binding.rib_window_attn_bwd(q, k, v, pq, pk, out, lse, dout, wl.window, wl.shift)[:3]
    size = q.numel()
    memory = [torch.full((size + 64,), 3.0, dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    grads = [m[8:8 + size].view(q.shape) for m in memory]
    assert all(g.data_ptr() % 32 == 16 for g in grads)
    dpq, dpk = (torch.empty(pq.shape, dtype=torch.float32, device="cuda") for _ in range(2))
    need = binding.rib_window_attn_bwd_workspace(wl.B, wl.H, wl.W, wl.heads, wl.d, wl.r, wl.window)
    workspace = torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")
    pointers = [t.data_ptr() for t in (q, k, v, pq, pk, out, lse, dout)]
    rc = binding.library().rib_window_attn_bwd(*pointers, wl.B, wl.H, wl.W, wl.heads, wl.d, wl.r, wl.window, wl.shift,
                                               *(t.data_ptr() for t in (*grads, dpq, dpk)), workspace.data_ptr(), workspace.numel(),
                                               torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    torch.cuda.synchronize()
    assert binding.rib_query_status() == 0 and binding.rib_last_path() == binding.RIB_PATH_SM100
    for name, got, want, m in zip(("dq", "dk", "dv"), grads, expected, memory):
        assert (m[:8] == 3.0).all() and (m[8 + size:] == 3.0).all(), name
        if name == "dq":
            # fp32 sums over key blocks in any order: at most 8 terms below 8 in size, 2 * 7 * 2^-24 * 64 < 1e-4 apart, and a bf16 step
            assert ((got.float() - want.float()).abs() <= want.float().abs() * 2.0 ** -7 + 1e-4).all()
        else:
            assert torch.equal(got, want), name
