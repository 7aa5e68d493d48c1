"""The separate gate kernel where a thread takes four 16-byte vectors (more vectors than the SMs
hold threads), one vector below and above that line and with ragged last blocks, against the fp64
gate of the plain forward's own outputs.  The two calls run the same mixer schedule, so u is one
rounding (2^-9 relative in bf16, 2^-12 in fp16: the half-unit) from the reference plus the gate's
fast exponential and division (a few 2^-22, times |z| <= 8 in the exponent): element bar 2^-8,
2^-11 and 2^-18 of |ref|, with 1e-7 of max|ref| for values that leave the normal range."""
import numpy as np
import pytest
import torch

import oracle
from gla_testutil import to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, H, grid_h, grid_w, Dk, Dv, dtype): vectors = B H T Dv / (8 or 4); 152 SMs hold 311296
CASES = [
    (19, 8, 16, 16, 64, 64, "bf16"),   # 311296: the last launch of one vector a thread
    (19, 8, 1, 257, 64, 64, "bf16"),   # 312512: four a thread, last block 0.19 full
    (40, 8, 13, 11, 128, 128, "f16"),  # 732160: two key halves, 16 lanes a row
    (40, 31, 5, 53, 64, 8, "f16"),     # 328600: one lane a row, ragged
    (41, 8, 7, 9, 64, 64, "f32"),      # 330624: fp32, 16 lanes a row
]
BAR = {"bf16": 2.0 ** -8, "f16": 2.0 ** -11, "f32": 2.0 ** -18}


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-{c[2]}x{c[3]}-d{c[4]}_{c[5]}-{c[6]}" for c in CASES])
def test_vectors_per_thread(case):
    B, H, gh, gw, Dk, Dv, dtype = case
    T = gh * gw
    gla.load()
    seed = 9950 + CASES.index(case)
    inp = wl.make_inputs(B, H, gh, gw, Dk, Dv, dtype, seed=seed)
    rng = np.random.Generator(np.random.PCG64(seed))
    r = wl.round_to_storage(np.clip(rng.standard_normal((B, T, H, Dv)) * 1.5, -8.0, 8.0), dtype)
    w = (1.0 + 0.2 * rng.standard_normal(Dv)).astype(np.float32)
    t = {n: to_torch(inp[n], dtype) for n in ("q", "k", "v", "g")}
    o, _ = gla.forward(t["q"], t["k"], t["v"], t["g"], gh, gw, wl.ROW_FWD)
    u, _ = gla.forward_gated(t["q"], t["k"], t["v"], t["g"], to_torch(r, dtype), torch.from_numpy(w).cuda(),
                             1e-6, gh, gw, wl.ROW_FWD)
    torch.cuda.synchronize()
    assert gla.sync_status() == 0
    ref = oracle.gated_output(o.double().cpu().numpy(), wl.storage_to_f64(r, dtype), w.astype(np.float64), 1e-6)
    err = np.abs(u.double().cpu().numpy() - ref)
    bar = BAR[dtype] * np.abs(ref) + 1e-7 * np.abs(ref).max()
    assert np.all(err <= bar), (err / bar).max()
