"""Caches and windows far larger than the prompt in them: the prompt phase clears the free slots and ring rows, in grids that
stay within the device's limits."""
import pytest
import torch

from paper_2503_00979_b200 import binding

pytestmark = pytest.mark.gpu


# 65535 blocks of 256 threads move 16 bytes each: 524 280 rows of 512 bytes.  Nothing is evicted: outputs are those of plain
# attention (f32 sums of 41 terms: 1e-5 is tens of roundings)
@pytest.mark.parametrize("C,R,q_heads", [(524300, 16, 2), (30, 66000, 8)])
def test_short_prompt(C, R, q_heads):
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(5)
    k, v = (torch.randn((1, 1, 1, 40, 128), generator=gen, device="cuda:0") for _ in range(2))
    q = torch.randn((1, 1, q_heads, 40, 128), generator=gen, device="cuda:0")
    q1, k1, v1 = (torch.randn((1, 1, h, 128), generator=gen, device="cuda:0") for h in (q_heads, 1, 1))
    mk = binding.MorphKV(1, 1, q_heads, 1, 128, C, R, "sum", "f32")
    mk.workspace.fill_(0xff)                 # free slots and rows that were not cleared would be NaN
    mk.prefill(k, v, q[:, :, :, 40 - min(R, 40):].contiguous())
    out = mk.decode_step(q1, k1, v1)
    mk.sync()
    kk, vv = (torch.cat([x[0, 0, 0], y[0, 0]]).double() for x, y in ((k, k1), (v, v1)))
    want = torch.softmax(q1[0, 0].double() @ kk.T / 128 ** 0.5, -1) @ vv
    assert (out[0, 0] - want).abs().max() < 1e-5
    vw = mk.view(0)
    assert vw["count"] == 41 and not vw["K"][0, 0, 41:].any() and not vw["ring_q"][0, 0, 41:].any()
    mk.close()
