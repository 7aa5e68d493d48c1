"""The start state of a split sequence's segments, folded from the earlier segments' summaries, at
the edges of the fold: one summary, a ring of exactly and just over four, one batch of decay products
(32) and one more, segments of two chunks (no third chunk to hold back) and longer ones, two value
slices, padded key channels, strong decay, and the fused output gate.  Against the fp64 oracle at the
mixer's bar, outputs and final state."""
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
    (4, 19, 8, 48, 64, 64, "f16", wl.ROW_FWD, 16.0, 0.0, 2, 3),     # one summary, three chunks
    (1, 2, 24, 24, 64, 64, "bf16", wl.COL_REV, 16.0, 0.0, 5, 2),    # four summaries
    (1, 6, 44, 44, 64, 64, "f16", wl.ROW_REV, 1.0, -1.0, 16, 2),    # strong decay, last segment one chunk
    (1, 2, 65, 64, 32, 128, "bf16", wl.ROW_FWD, 16.0, 0.0, 33, 2),  # 32 summaries: one batch; two slices
    (1, 4, 80, 80, 32, 64, "f16", wl.COL_FWD, 16.0, 0.0, 34, 3),    # 33: a second batch
    (1, 2, 128, 128, 64, 64, "bf16", wl.ROW_REV, 16.0, 0.0, 64, 4), # 63, held-back chunks
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-{c[2]}x{c[3]}-d{c[4]}_{c[5]}-{c[6]}-o{c[7]}" for c in CASES])
def test_start_states(case):
    B, H, gh, gw, Dk, Dv, dtype, order, tau, zm, nseg, length = case
    gla.load()
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert gla.split_plan(B, H, gh, gw, Dk, Dv, 152) == (nseg, length)
    inp = wl.make_inputs(B, H, gh, gw, Dk, Dv, dtype, seed=9800 + CASES.index(case), tau=tau, z_mean=zm)
    f = inputs_f64(inp, dtype)
    t = {n: to_torch(inp[n], dtype) for n in ("q", "k", "v", "g")}
    ref_o, ref_s = oracle.recurrence(f["q"], f["k"], f["v"], f["g"], gh, gw, order)
    rng = np.random.Generator(np.random.PCG64(9850))
    r = wl.round_to_storage(rng.standard_normal((B, gh * gw, H, Dv)) * 1.5, dtype)
    w = (1.0 + 0.2 * rng.standard_normal(Dv)).astype(np.float32)
    for gated in (False, True):
        out = torch.full_like(t["v"], float("nan"))
        if gated:
            out, fs = gla.forward_gated(t["q"], t["k"], t["v"], t["g"], to_torch(r, dtype), torch.from_numpy(w).cuda(),
                                        1e-5, gh, gw, order, out=out)
            ref = oracle.gated_output(ref_o, wl.storage_to_f64(r, dtype), w.astype(np.float64), 1e-5)
        else:
            out, fs = gla.forward(t["q"], t["k"], t["v"], t["g"], gh, gw, order, out=out)
            ref = ref_o
        torch.cuda.synchronize()
        assert gla.sync_status() == 0
        assert gla.last_schedule()[0] == "tc_split"
        got = out.float().cpu().numpy().astype(np.float64)
        if gated and Dv > 64:  # a second kernel gates the rounded outputs: twice the bar
            e = np.linalg.norm(got - ref) / np.linalg.norm(ref)
            assert np.isfinite(got).all() and e <= 4e-3
        else:
            assert_within_bar(got, ref, dtype, f"gated {gated}")
        assert_within_bar(fs.cpu().numpy().astype(np.float64), ref_s, dtype, "final_state")
