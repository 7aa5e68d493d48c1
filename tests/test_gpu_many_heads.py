"""A token row of 2^31 output elements (2^24 heads of 128 columns): the stores' token stride does not fit
32 bits.  Two tokens, so the outputs have a closed form: o_1 = (q_1 k_1) v_1 and
o_2 = (q_2 e^{g_2} k_1) v_1 + (q_2 k_2) v_2, compared in slices of heads at the mixer's bar."""
import pytest
import torch

from gla_testutil import REL_L2_16BIT
from paper_2609_26590_gb300 import gla

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
def test_token_rows_past_32_bits(dtype):
    gla.load()
    H, Dk, Dv = 1 << 24, 8, 128
    if torch.cuda.mem_get_info()[0] < 48 << 30:
        pytest.skip("needs 48 GB of device memory")
    gen = torch.Generator(device="cuda").manual_seed(41)
    q, k = (torch.randn(1, 2, H, Dk, generator=gen, device="cuda", dtype=dtype) for _ in range(2))
    g = -0.5 * torch.rand(1, 2, H, Dk, generator=gen, device="cuda", dtype=dtype)
    v = torch.randn(1, 2, H, Dv, generator=gen, device="cuda", dtype=dtype)
    for order in range(4):
        out, _ = gla.forward(q, k, v, g, 1, 2, order, schedule="tc", final_state=False)
        torch.cuda.synchronize()
        assert gla.sync_status() == 0
        a, b = (0, 1) if order % 2 == 0 else (1, 0)  # the first and the second token of the scan
        step = H >> 4
        for h in range(0, H, step):
            qs, ks, gs, vs, o = (x[0, :, h:h + step].float() for x in (q, k, g, v, out))
            s11 = (qs[a] * ks[a]).sum(-1, keepdim=True)
            s21 = (qs[b] * ks[a] * gs[b].exp()).sum(-1, keepdim=True)
            s22 = (qs[b] * ks[b]).sum(-1, keepdim=True)
            for got, ref in ((o[a], s11 * vs[a]), (o[b], s21 * vs[a] + s22 * vs[b])):
                assert torch.isfinite(got).all()
                assert float((got - ref).norm() / ref.norm()) <= REL_L2_16BIT, f"order {order} heads {h}"
        del out
