"""Chunks whose decays are too strong for the split score operands (CUDA-core scores from blocks of 16
and 4 keys) against the fp64 oracle at the mixer's bar: every gate strong, a mix with gamma = 0 and
gamma = 1 gates, one and two key halves, ragged and split sequences, every order."""
import numpy as np
import pytest
import torch

import oracle
from gla_testutil import assert_within_bar, inputs_f64, to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, H, grid_h, grid_w, Dk, Dv, dtype, z_mean, share of gamma = 0 gates, share of gamma = 1 gates)
CASES = [
    (1, 3, 16, 20, 64, 64, "f16", -6.0, 0.0, 0.0),      # every chunk exact
    (2, 2, 9, 13, 64, 64, "bf16", -3.0, 0.05, 0.5),     # ragged, mixed channels
    (1, 2, 8, 24, 128, 128, "bf16", -6.0, 0.02, 0.3),   # two key halves and value slices
    (1, 1, 32, 24, 32, 64, "f16", -4.0, 0.0, 0.2),      # split sequence, padded key half
    (1, 1, 40, 24, 128, 64, "f16", -6.0, 0.0, 0.3),     # split, summaries by key half
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-{c[2]}x{c[3]}-d{c[4]}_{c[5]}-{c[6]}-z{c[7]}" for c in CASES])
def test_exact_chunks(case):
    B, H, gh, gw, Dk, Dv, dtype, zm, zero, one = case
    gla.load()
    inp = wl.make_inputs(B, H, gh, gw, Dk, Dv, dtype, seed=9300 + CASES.index(case), tau=1.0, z_mean=zm)
    rng = np.random.Generator(np.random.PCG64(79))
    g = wl.storage_to_f64(inp["g"], dtype)
    u = rng.random(g.shape)
    g[u < zero] = -np.inf
    g[u > 1.0 - one] = 0.0
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
