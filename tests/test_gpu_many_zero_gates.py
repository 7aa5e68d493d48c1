"""Many log gates of -inf (gamma = 0) among mild ones, several per channel and chunk: the decays of the keys
after a channel's last zero gate must keep their precision although the chunk's prefix has passed many of
them.  Outputs and final state against the fp64 oracle at the mixer's bar; every order, one and two key
halves, few and padded key channels, whole and split launches."""
import numpy as np
import pytest
import torch

import oracle
from gla_testutil import assert_within_bar, inputs_f64, to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, H, grid_h, grid_w, Dk, Dv, dtype)
CASES = [
    (2, 3, 16, 20, 64, 64, "f16"),
    (4, 2, 9, 11, 8, 64, "bf16"),
    (1, 2, 16, 20, 128, 64, "bf16"),
    (1, 2, 32, 24, 64, 64, "f16"),     # split
    (1, 1, 40, 24, 128, 128, "f16"),   # split, two key halves
]


@pytest.mark.parametrize("share", [0.05, 0.2, 0.6])
@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-{c[2]}x{c[3]}-d{c[4]}_{c[5]}-{c[6]}" for c in CASES])
def test_many_zero_decays(case, share):
    B, H, gh, gw, Dk, Dv, dtype = case
    gla.load()
    inp = wl.make_inputs(B, H, gh, gw, Dk, Dv, dtype, seed=9950 + CASES.index(case), tau=16.0)
    g = wl.storage_to_f64(inp["g"], dtype)
    rng = np.random.Generator(np.random.PCG64(83))
    g[rng.random(g.shape) < share] = -np.inf
    inp["g"] = wl.round_to_storage(g, dtype)
    f = inputs_f64(inp, dtype)
    t = {n: to_torch(inp[n], dtype) for n in ("q", "k", "v", "g")}
    for order in wl.ALL_ORDERS:
        ref_o, ref_s = oracle.recurrence(f["q"], f["k"], f["v"], f["g"], gh, gw, order)
        out, fs = gla.forward(t["q"], t["k"], t["v"], t["g"], gh, gw, order, schedule="tc")
        torch.cuda.synchronize()
        assert gla.sync_status() == 0
        assert_within_bar(out.float().cpu().numpy().astype(np.float64), ref_o, dtype, f"out order {order}")
        assert_within_bar(fs.cpu().numpy().astype(np.float64), ref_s, dtype, f"state order {order}")
