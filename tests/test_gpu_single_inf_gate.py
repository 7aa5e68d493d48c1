"""A single log gate of -inf (gamma = 0) among mild ones: in the first half of a chunk, past its middle
and at its last position.  Past the middle the mid-chunk prefix of its channel is 0 x -inf = NaN and only
the score mode's maximum can tell; a chunk that misses it writes NaN outputs and a NaN state.  Outputs
and final state against the fp64 oracle at the mixer's bar: every order, one and two key halves, padded
key channels, whole, split and balanced launches."""
import numpy as np
import pytest
import torch

import oracle
from gla_testutil import assert_within_bar, inputs_f64, to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, H, grid_h, grid_w, Dk, Dv, dtype, schedule on 152 SMs)
CASES = [
    (1, 2, 16, 20, 64, 64, "f16", "tc"),
    (1, 2, 16, 20, 32, 64, "bf16", "tc"),          # the channel 32 away is padding
    (1, 2, 16, 20, 128, 64, "bf16", "tc"),
    (1, 2, 24, 24, 64, 64, "bf16", "tc_split"),
    (1, 1, 32, 24, 128, 128, "f16", "tc_split"),
    (16, 12, 16, 12, 64, 64, "f16", "tc_balanced"),
]


@pytest.mark.parametrize("pos", [20, 40, 63])
@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-{c[2]}x{c[3]}-d{c[4]}_{c[5]}-{c[6]}-{c[7]}" for c in CASES])
def test_one_zero_decay(case, pos):
    B, H, gh, gw, Dk, Dv, dtype, sched = case
    gla.load()
    inp = wl.make_inputs(B, H, gh, gw, Dk, Dv, dtype, seed=9900 + CASES.index(case), tau=16.0)
    g0 = wl.storage_to_f64(inp["g"], dtype)
    t = {n: to_torch(inp[n], dtype) for n in ("q", "k", "v")}
    for order in wl.ALL_ORDERS:
        g = g0.copy()
        token = oracle.scan_tokens(order, gh, gw)[64 + pos]   # the second chunk
        g.reshape(B, gh * gw, H, Dk)[:, token, :, Dk - 3] = -np.inf
        gs = wl.round_to_storage(g, dtype)
        f = inputs_f64(dict(inp, g=gs), dtype)
        ref_o, ref_s = oracle.recurrence(f["q"], f["k"], f["v"], f["g"], gh, gw, order)
        out, fs = gla.forward(t["q"], t["k"], t["v"], to_torch(gs, dtype), gh, gw, order, schedule="tc")
        torch.cuda.synchronize()
        assert gla.sync_status() == 0
        if torch.cuda.get_device_properties(0).multi_processor_count == 152:
            assert gla.last_schedule()[0] == sched
        assert_within_bar(out.float().cpu().numpy().astype(np.float64), ref_o, dtype, f"out order {order}")
        assert_within_bar(fs.cpu().numpy().astype(np.float64), ref_s, dtype, f"state order {order}")
