"""Rows that TMA cannot address (even head widths and ranks that are no multiples of 8), windows of the general kernels: every
remainder of a 16-byte piece that the row copies, the preparation and the finishing kernel meet, against the CPU oracle."""
import numpy as np
import pytest

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
