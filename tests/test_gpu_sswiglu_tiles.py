"""Tiles of the Spatial SwiGLU kernel at their edges against the fp64 oracle: grids cut into several
column tiles (the last one narrower than four columns, or wholly inside its box's padding), rows cut
into strips, launches of one wave and of several, and gates far outside the sigmoid's range.  Bar: the
mixer's, as in test_gpu_sswiglu.py (outputs accumulated in fp32 and rounded once)."""
import numpy as np
import pytest
import torch

import oracle
from gla_testutil import assert_within_bar, to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, grid_h, grid_w, F, dtype, gate scale)
CASES = [
    (1, 9, 41, 72, "f16", 1.0),      # two column tiles of 24: the second ends inside its box
    (2, 5, 121, 136, "bf16", 1.0),   # four column tiles of 32, three slices
    (1, 33, 81, 20, "f32", 1.0),     # three of 28, rows cut
    (1, 11, 3, 16, "bf16", 1.0),     # one column group, several strips
    (1, 7, 5, 8, "f16", 300.0),      # gates to +-1e3: sigmoid 0 and 1
    (1, 6, 9, 12, "f32", 1.0e30),    # e^{-z} overflows
    (7, 37, 39, 520, "bf16", 1.0),   # several waves, a partial slice
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}x{c[2]}-F{c[3]}-{c[4]}" for c in CASES])
def test_tile_edges(case):
    B, gh, gw, F, dtype, scale = case
    gla.load()
    inp = wl.sswiglu_inputs(B, gh, gw, F, dtype, seed=4600 + CASES.index(case))
    h = wl.storage_to_f64(inp["h"], dtype)
    h[..., :F] *= scale
    hs = wl.round_to_storage(h, dtype)
    h = wl.storage_to_f64(hs, dtype)
    t = to_torch(hs, dtype)
    w, b = torch.from_numpy(inp["weight"]).cuda(), torch.from_numpy(inp["bias"]).cuda()
    out = gla.sswiglu_dwconv(t[..., :F], t[..., F:], w, b, gh, gw)
    torch.cuda.synchronize()
    assert gla.sync_status() == 0
    with np.errstate(over="ignore"):
        ref = oracle.sswiglu_dwconv(h[..., :F], h[..., F:], inp["weight"], inp["bias"], gh, gw)
    assert_within_bar(out.float().cpu().numpy().astype(np.float64), ref, dtype, "z")
