"""The CUDA-core recurrence in 16 value columns a CTA (narrow values, few key channels, short sequences)
against the fp64 oracle at the mixer's bars: partial blocks of 16 tokens, partial columns, one token,
zero decays, both thread layouts (up to 32 and up to 64 key channels), all types and orders."""
import numpy as np
import pytest
import torch

import oracle
from gla_testutil import assert_within_bar, inputs_f64, to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, H, grid_h, grid_w, Dk, Dv, dtype, tau, z_mean, share of gamma = 0 gates)
CASES = [
    (3, 53, 16, 11, 32, 16, "f32", 16.0, 0.0, 0.0),     # whole blocks and columns
    (2, 80, 7, 19, 20, 24, "f32", 1.0, -1.0, 0.02),     # a last block of five tokens, half a column block
    (5, 33, 9, 15, 7, 7, "f16", 16.0, 0.0, 0.0),
    (1, 157, 12, 12, 31, 61, "bf16", 1.0, -1.0, 0.02),  # four column blocks, the last one ragged
    (1, 311, 11, 13, 61, 14, "f32", 16.0, 0.0, 0.02),
    (2, 3, 4, 4, 64, 64, "f32", 16.0, 0.0, 0.0),        # one block of 16 tokens
    (2, 3, 5, 9, 33, 50, "f16", 1.0, -1.0, 0.0),        # three blocks
    (1, 5, 1, 1, 64, 64, "f32", 16.0, 0.0, 0.0),        # one token
    (2, 2, 1, 17, 8, 1, "f32", 16.0, 0.0, 0.0),         # one column, a block of one token
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-{c[2]}x{c[3]}-d{c[4]}_{c[5]}-{c[6]}" for c in CASES])
def test_narrow_columns(case):
    B, H, gh, gw, Dk, Dv, dtype, tau, zm, zero = case
    gla.load()
    inp = wl.make_inputs(B, H, gh, gw, Dk, Dv, dtype, seed=9400 + CASES.index(case), tau=tau, z_mean=zm)
    if zero > 0:
        rng = np.random.Generator(np.random.PCG64(80))
        g = wl.storage_to_f64(inp["g"], dtype)
        g[rng.random(g.shape) < zero] = -np.inf
        inp["g"] = wl.round_to_storage(g, dtype)
    f = inputs_f64(inp, dtype)
    t = {n: to_torch(inp[n], dtype) for n in ("q", "k", "v", "g")}
    assert gla.simt_plan(B, H, gh, gw, Dk, Dv, t["q"].dtype, 152) == (0, 16)
    for order in wl.ALL_ORDERS:
        ref_o, ref_s = oracle.recurrence(f["q"], f["k"], f["v"], f["g"], gh, gw, order)
        out = torch.full_like(t["v"], float("nan"))
        out, fs = gla.forward(t["q"], t["k"], t["v"], t["g"], gh, gw, order, out=out, schedule="simt")
        torch.cuda.synchronize()
        assert gla.sync_status() == 0
        assert gla.last_schedule()[0] == "simt"
        assert_within_bar(out.float().cpu().numpy().astype(np.float64), ref_o, dtype, f"out order {order}")
        assert_within_bar(fs.cpu().numpy().astype(np.float64), ref_s, dtype, f"state order {order}")
