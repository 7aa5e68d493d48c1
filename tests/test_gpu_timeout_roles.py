"""The bounded waits' give-up path where a chunk's warps go on to warp-collective work after the wait: the
gate producer (its first wait is for Z, the product of the withheld tile) and launches whose gen warps
store the outputs.  As tests/test_gpu_timeout.py: CTA 0 withholds its first chunk's load, the call reports
GTR_ERR_TIMEOUT without a fault, and the same call without the hook then gives what it gave before."""
import pytest
import torch

from gla_testutil import to_torch
from paper_2609_26590_gb300 import gla
from paper_2609_26590_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

GTR_ERR_TIMEOUT = 5


# 20 x 16: five chunks, whole sequences; f16 at one wave: outputs stored by the gen warps
@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("op", ["mixer", "lowrank"])
def test_roles_give_up_together(op, dtype, monkeypatch):
    gla.load()
    B, H, gh, gw, D, T = 1, 2, 20, 16, 64, 320
    inp = wl.make_inputs(B, H, gh, gw, D, D, dtype, seed=8200)
    t = {n: to_torch(inp[n], dtype) for n in ("q", "k", "v", "g")}
    gp = wl.gate_producer_inputs(B, H, T, D, dtype, seed=8201)
    a, w2, bias = to_torch(gp["a"], dtype), to_torch(gp["w2"], dtype), torch.from_numpy(gp["bias"]).cuda()

    def call():
        if op == "lowrank":
            return gla.forward_lowrank_gate(t["q"], t["k"], t["v"], a, w2, bias, 16.0, gh, gw, wl.COL_FWD)
        return gla.forward(t["q"], t["k"], t["v"], t["g"], gh, gw, wl.COL_FWD, schedule="tc")

    out, fs = call()
    assert gla.last_schedule()[0] == "tc"
    assert gla.sync_status() == 0
    monkeypatch.setenv("GTR_GLA_TEST_DROP_LOAD", "1")
    call()
    assert gla.sync_status() == GTR_ERR_TIMEOUT
    monkeypatch.delenv("GTR_GLA_TEST_DROP_LOAD")
    again, fs2 = call()
    assert gla.sync_status() == 0
    assert torch.equal(out, again) and torch.equal(fs, fs2)
