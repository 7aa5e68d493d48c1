"""The CUDA-core recurrence cut into segments across a thread-block cluster: every cluster size the
launch rule picks, one, two and four groups per CTA, ragged and empty last segments, CTAs with idle
groups, two column blocks, widths that are no multiple of four, all orders, against the fp64 oracle at
the mixer's bars."""
import numpy as np
import pytest
import torch

import oracle
from gla_testutil import assert_within_bar, inputs_f64, to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, H, grid_h, grid_w, Dk, Dv, dtype, tau, z_mean, share of gamma = 0 gates); the cluster on 152 SMs
CASES = [
    (1, 2, 33, 31, 64, 64, "f32", 16.0, 0.0, 0.0),     # 16 CTAs, 32 segments, the last one ragged
    (1, 3, 29, 25, 40, 72, "f32", 1.0, -1.0, 0.02),    # 16, two column blocks, an empty last segment
    (1, 1, 20, 27, 33, 50, "f16", 16.0, 0.0, 0.0),     # 16, scalar loads and stores
    (2, 6, 13, 20, 20, 24, "f32", 1.0, -1.0, 0.0),     # 4 of four groups, a whole CTA empty
    (3, 11, 19, 23, 64, 61, "f32", 16.0, 0.0, 0.02),   # 8, scalar
    (5, 9, 11, 12, 128, 128, "f32", 16.0, 0.0, 0.0),   # 2 of one group, two column blocks
    (5, 18, 11, 12, 96, 64, "bf16", 1.0, -1.0, 0.0),   # 3 of one group
    (11, 13, 9, 10, 64, 64, "f32", 16.0, 0.0, 0.0),    # 2
    (19, 9, 6, 7, 64, 64, "f32", 1.0, -1.0, 0.0),      # whole sequences, one group idle
    (1, 1, 5, 5, 32, 8, "f32", 16.0, 0.0, 0.0),        # whole, three groups idle
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-{c[2]}x{c[3]}-d{c[4]}_{c[5]}-{c[6]}" for c in CASES])
def test_segments(case):
    B, H, gh, gw, Dk, Dv, dtype, tau, zm, zero = case
    gla.load()
    inp = wl.make_inputs(B, H, gh, gw, Dk, Dv, dtype, seed=9100 + CASES.index(case), tau=tau, z_mean=zm)
    if zero > 0:
        rng = np.random.Generator(np.random.PCG64(78))
        g = wl.storage_to_f64(inp["g"], dtype)
        g[rng.random(g.shape) < zero] = -np.inf
        inp["g"] = wl.round_to_storage(g, dtype)
    f = inputs_f64(inp, dtype)
    t = {n: to_torch(inp[n], dtype) for n in ("q", "k", "v", "g")}
    for order in wl.ALL_ORDERS:
        ref_o, ref_s = oracle.recurrence(f["q"], f["k"], f["v"], f["g"], gh, gw, order)
        out, fs = gla.forward(t["q"], t["k"], t["v"], t["g"], gh, gw, order, schedule="simt")
        torch.cuda.synchronize()
        assert gla.sync_status() == 0
        assert_within_bar(out.float().cpu().numpy().astype(np.float64), ref_o, dtype, f"out order {order}")
        assert_within_bar(fs.cpu().numpy().astype(np.float64), ref_s, dtype, f"state order {order}")
