"""How exact the prompt phase's soft-max normalisers are where the keys that a thread sums first lie far below those that
follow: the sums' reference has to move with the maximum, or the exponents of the weights that count are rounded as numbers
of that distance."""
import numpy as np
import pytest
import torch

from paper_2503_00979_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [1500, 6144])
@pytest.mark.parametrize("below", [0, 10, 30])
def test_keys_that_follow_lower_ones(P, below):
    # the first 32 keys of every tile of 128 lie `below` powers of two under the others
    L, H, G, C, R, dev = 8, 8, 4, 700, 32, torch.device("cuda:0")
    gen = torch.Generator(device=dev)
    gen.manual_seed(6)
    k = torch.randn((L, H, P, 128), generator=gen, device=dev).mul_(0.7)
    q = torch.randn((L, H * G, R, 128), generator=gen, device=dev).mul_(0.7)
    q[..., 0], k[..., 0] = 4.0, 0.0
    k[:, :, torch.arange(P, device=dev) % 128 < 32, 0] = -below * np.sqrt(128) * np.log(2) / 4.0
    k, q = k.bfloat16(), q.bfloat16()
    mk = binding.MorphKV(L, 1, H * G, H, 128, C, R, "sum", "bf16")
    mk.prefill(k[:, None].contiguous(), torch.zeros_like(k)[:, None].contiguous(), q[:, None].contiguous())
    seen = torch.arange(P, device=dev)[None] <= (P - R + torch.arange(R, device=dev))[:, None]
    err = []
    for l in range(L):
        got = mk.view(l)["ring_c"][0][..., :G].double().permute(0, 2, 1).roll(-((P - R) % R), 2)      # [unit][head][window row]
        for u in range(H):
            s = (q[l, u * G:(u + 1) * G].double().reshape(G * R, 128) @ k[l, u].double().T).view(G, R, P) / np.sqrt(128)
            want = torch.logsumexp(s.masked_fill(~seen, -np.inf), -1) / np.log(2)
            err.append((got[u] - want).abs())
    mk.close()
    # The normalisers lie between 8 and 16: rounding them leaves 2^-22 on average, rounding the logarithm that they are added up
    # from at most as much.  (2.5e-7 to 3.4e-7; with a reference that stays behind by 10 and by 30, 5.2e-7 and 9.6e-7.)
    assert torch.stack(err).mean().item() < 2 * 2.0 ** -22
