"""A split call whose summary pass takes longer than the limit of the bounded waits (1 s): the output pass,
which starts while it runs, must not count that time.  With the test hook GTR_GLA_TEST_DROP_LOAD=2 a grid that
takes 1.5 s stands between the passes, and the output pass starts while it runs; the call reports no timeout
and gives the same bits as without."""
import pytest
import torch

from gla_testutil import to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, H, grid_h, grid_w, Dk, Dv, dtype, gated)
CASES = [
    (1, 6, 40, 40, 64, 64, "f16", False),     # segments of two chunks, outputs stored by the gen warps
    (1, 4, 80, 80, 64, 64, "f16", True),      # of three, with the fused output gate
    (4, 12, 40, 40, 64, 64, "bf16", False),   # of nine, outputs stored by the epi
    (1, 2, 40, 40, 128, 64, "bf16", False),   # two key halves
]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}-d{c[4]}-{c[6]}-{'gated' if c[7] else 'mixer'}" for c in CASES])
def test_summary_pass_longer_than_the_wait_limit(case, monkeypatch):
    B, H, gh, gw, Dk, Dv, dtype, gated = case
    gla.load()
    inp = wl.make_inputs(B, H, gh, gw, Dk, Dv, dtype, seed=8300)
    t = {n: to_torch(inp[n], dtype) for n in ("q", "k", "v", "g")}
    w = torch.ones(Dv, device="cuda")

    def call():
        if gated:
            return gla.forward_gated(t["q"], t["k"], t["v"], t["g"], t["v"], w, 1e-5, gh, gw, wl.ROW_REV)
        return gla.forward(t["q"], t["k"], t["v"], t["g"], gh, gw, wl.ROW_REV)

    out, fs = call()
    assert gla.last_schedule()[0] == "tc_split"
    assert gla.sync_status() == 0
    monkeypatch.setenv("GTR_GLA_TEST_DROP_LOAD", "2")
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record()
    late, fs2 = call()
    end.record()
    assert gla.sync_status() == 0
    assert start.elapsed_time(end) >= 1500.0
    assert torch.equal(out, late) and torch.equal(fs, fs2)
