"""Split sequences of two key halves whose summary pass has more work units (sequence, segment, key half)
than the GPU has SMs, so that a CTA walks several: 50 sequences of six chunks with Dk = 128 give 200 on 152
SMs.  Outputs and final state against the fp64 oracle at the mixer's bar, mild and strong decays."""
import numpy as np
import pytest
import torch

import oracle
from gla_testutil import assert_within_bar, inputs_f64, to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, H, grid_h, grid_w, Dk, Dv, dtype, order, tau, z_mean, segments, chunks per segment) on 152 SMs
CASES = [
    (2, 25, 18, 20, 128, 64, "f16", wl.ROW_FWD, 16.0, 0.0, 3, 2),
    (1, 50, 18, 20, 72, 64, "bf16", wl.COL_REV, 1.0, -1.0, 3, 2),
    (5, 10, 21, 20, 128, 40, "bf16", wl.ROW_REV, 1.0, -5.0, 3, 3),   # exact chunks, the last segment one
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-{c[2]}x{c[3]}-d{c[4]}_{c[5]}-{c[6]}-o{c[7]}" for c in CASES])
def test_summary_ctas_walk_several_units(case):
    B, H, gh, gw, Dk, Dv, dtype, order, tau, zm, nseg, length = case
    gla.load()
    assert gla.split_plan(B, H, gh, gw, Dk, Dv, 152) == (nseg, length)
    assert 2 * B * H * (nseg - 1) > 152
    inp = wl.make_inputs(B, H, gh, gw, Dk, Dv, dtype, seed=9600 + CASES.index(case), tau=tau, z_mean=zm)
    f = inputs_f64(inp, dtype)
    t = {n: to_torch(inp[n], dtype) for n in ("q", "k", "v", "g")}
    ref_o, ref_s = oracle.recurrence(f["q"], f["k"], f["v"], f["g"], gh, gw, order)
    out = torch.full_like(t["v"], float("nan"))
    out, fs = gla.forward(t["q"], t["k"], t["v"], t["g"], gh, gw, order, out=out)
    torch.cuda.synchronize()
    assert gla.sync_status() == 0
    assert gla.last_schedule()[0] == "tc_split"
    assert_within_bar(out.float().cpu().numpy().astype(np.float64), ref_o, dtype, "out")
    assert_within_bar(fs.cpu().numpy().astype(np.float64), ref_s, dtype, "final_state")
