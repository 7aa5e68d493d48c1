"""A split call whose summary pass takes longer than the limit of the bounded waits (1 s): the output pass,
which starts while it runs, allows for that.  With the test hook GTR_GLA_TEST_DROP_LOAD=2 a grid that takes 1 s
and 0.05 ms per chunk of a segment stands between the passes, and the output pass starts while it runs; the
call reports no timeout and gives the same bits as without."""
import pytest
import torch

from gla_testutil import to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# (B, H, grid_h, grid_w, Dk, Dv, dtype, gated); segments of 6 chunks and more
CASES = [
    (1, 2, 256, 256, 64, 64, "f16", False),    # outputs stored by the gen warps
    (1, 2, 256, 256, 64, 64, "f16", True),     # with the fused output gate
    (4, 13, 120, 34, 40, 64, "bf16", False),   # outputs stored by the epi
    (1, 2, 160, 160, 128, 64, "bf16", False),  # two key halves
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

    assert gla.split_plan(B, H, gh, gw, Dk, Dv, 152)[1] >= 6
    out, fs = call()
    assert gla.last_schedule()[0] == "tc_split"
    assert gla.sync_status() == 0
    monkeypatch.setenv("GTR_GLA_TEST_DROP_LOAD", "2")
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record()
    late, fs2 = call()
    end.record()
    assert gla.sync_status() == 0
    assert start.elapsed_time(end) >= 1000.0
    assert torch.equal(out, late) and torch.equal(fs, fs2)
