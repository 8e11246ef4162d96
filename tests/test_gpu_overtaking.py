"""Backward passes whose main kernel overtakes the kernel that clears its gradients (windows of 8 and 16 tokens, feature generator):
old values in the results, gaps between head-wise tables, a side stream with late inputs, CUDA graphs."""
import numpy as np
import pytest
import torch

from oracle import rib_generator_oracle as gen
from oracle import rib_oracle
from paper_2603_06738_b200 import binding, synthetic
from paper_2603_06738_b200.synthetic import Workload

from parity_util import compare, to_f64

pytestmark = pytest.mark.gpu

LATE = 20_000_000          # GPU clock cycles (about 10 ms) by which a side stream's inputs are late


def attention(wl):
    """(run, check): run() enqueues the backward pass into buffers that stay; head-wise tables lie 64 elements apart."""
    cpu = synthetic.make_inputs(wl, with_dout=True)
    gpu = {k: v.cuda() for k, v in cpu.items()}
    gap, per_table = 64, wl.n * wl.r
    stride = per_table + gap if wl.headwise else 0
    tables = wl.heads if wl.headwise else 1

    def spread(t):
        wide = torch.full((tables, per_table + gap), 7.0, dtype=t.dtype, device="cuda")
        wide[:, :per_table] = t.reshape(tables, per_table)
        return wide
    pq, pk = spread(gpu["pq"]), spread(gpu["pk"])
    fwd = binding.rib_window_attn_fwd_headwise if wl.headwise else binding.rib_window_attn_fwd
    out, lse = fwd(*(gpu[k] for k in ("q", "k", "v", "pq", "pk")), wl.window, wl.shift)
    dout = torch.zeros_like(gpu["dout"])
    grads = [torch.empty_like(gpu["q"]) for _ in range(3)]
    dpq, dpk = (torch.empty((tables, per_table + gap), dtype=torch.float32, device="cuda") for _ in range(2))
    shape = (wl.B, wl.H, wl.W, wl.heads, wl.d, wl.r, wl.window)
    workspace = torch.empty(binding.rib_window_attn_bwd_headwise_workspace(stride, *shape), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()

    def soil():
        for t in (*grads, dpq, dpk):
            t.fill_(float("nan"))

    def run():
        dout.copy_(gpu["dout"])
        rc = binding.library().rib_window_attn_bwd_headwise(
            *(t.data_ptr() for t in (gpu["q"], gpu["k"], gpu["v"], pq, pk)), stride, out.data_ptr(), lse.data_ptr(), dout.data_ptr(), *shape, wl.shift,
            *(t.data_ptr() for t in (*grads, dpq, dpk)), workspace.data_ptr(), workspace.numel(), torch.cuda.current_stream().cuda_stream)
        assert rc == 0 and binding.rib_last_path() == binding.RIB_PATH_SM100

    ref = rib_oracle.bwd(*(to_f64(cpu[k]) for k in ("q", "k", "v", "pq", "pk", "dout")), wl.window, wl.shift)

    def check():
        assert torch.isnan(dpq[:, per_table:]).all() and torch.isnan(dpk[:, per_table:]).all()       # between the tables: not touched
        for name, got, want in zip(("dq", "dk", "dv", "dpq", "dpk"), (*grads, dpq[:, :per_table], dpk[:, :per_table]), ref):
            compare(name, to_f64(got).reshape(want.shape), want, max_abs=1e-2 * max(1.0, float(np.abs(want).max())))
    return soil, run, check


def generator(window, L, dh, r):
    rng = np.random.default_rng(7)
    ws = [np.float32(rng.normal(0, 0.3, s)) for s in ((2 + 4 * L, dh), (dh,), (dh, r), (dh, r))]
    gs = [np.float32(rng.normal(size=(window * window, r))) for _ in range(2)]
    gw, late = [torch.from_numpy(w).cuda() for w in ws], [torch.from_numpy(g).cuda() for g in gs]
    given = [torch.zeros_like(g) for g in late]
    results = [torch.empty_like(w) for w in gw]
    torch.cuda.synchronize()

    def soil():
        for t in results:
            t.fill_(float("nan"))

    def run():
        for g, l in zip(given, late):
            g.copy_(l)
        rc = binding.library().rib_generate_features_bwd(*(t.data_ptr() for t in (*gw, *given)), window, L, dh, r, *(t.data_ptr() for t in results),
                                                         torch.cuda.current_stream().cuda_stream)
        assert rc == 0
    ref = gen.backward(*ws, *gs, window, L)

    def check():
        for i, (got, want) in enumerate(zip(results, ref)):
            assert np.linalg.norm(to_f64(got) - want) <= 2e-6 * np.linalg.norm(want), i          # fp32 sums of up to 1024 terms
    return soil, run, check


CASES = {
    "w8": lambda: attention(Workload("o_w8", 2, 48, 64, 3, 32, 16, 8, 0, seed=601)),
    "w8_headwise": lambda: attention(Workload("o_w8_headwise", 1, 32, 48, 5, 16, 24, 8, 0, seed=602, headwise=True)),
    "w16": lambda: attention(Workload("o_w16", 2, 64, 48, 3, 32, 16, 16, 8, seed=603)),
    "w16_headwise": lambda: attention(Workload("o_w16_headwise", 1, 32, 48, 5, 16, 24, 16, 0, seed=604, headwise=True)),
    "generator": lambda: generator(32, 10, 32, 16),
    "generator_odd": lambda: generator(9, 3, 33, 18),
}


@pytest.mark.parametrize("name", CASES)
def test_a_side_stream_with_late_inputs_and_old_results(name):
    soil, run, check = CASES[name]()
    side = torch.cuda.Stream()
    soil()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        for _ in range(2):                       # the second call finds the first one's sums
            torch.cuda._sleep(LATE)
            run()
    side.synchronize()
    assert binding.rib_query_status(side) == 0
    check()


@pytest.mark.parametrize("name", CASES)
def test_under_capture(name):
    soil, run, check = CASES[name]()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        run()
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    soil()
    torch.cuda.synchronize()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert binding.rib_query_status() == 0
    check()
