"""The prompt phase's selection where its radix digits do not separate the keys: prompts whose older tokens share one or two
scores, so that positions decide (the lower one is kept), at lengths on either side of what a warp's registers hold and of
what the list in shared memory holds."""
import pytest
import torch

from paper_2503_00979_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,C", [(1030, 1), (1040, 1003), (3100, 700), (8208, 3000), (8209, 8192), (20011, 3500), (140000, 64)])
@pytest.mark.parametrize("groups", [1, 2])
def test_tied_scores_keep_the_lower_positions(P, C, groups):
    R, dev = 16, torch.device("cuda:0")
    M = P - R
    gen = torch.Generator(device=dev)
    gen.manual_seed(P + groups)
    q = torch.randn((1, 1, 8, R, 128), generator=gen, device=dev)
    k = torch.zeros((1, 1, 2, P, 128), device=dev)
    first = torch.zeros(M, dtype=torch.bool, device=dev)
    if groups == 2:           # some tokens point along the queries' mean and score higher, all of them alike
        first = torch.rand(M, generator=gen, device=dev) < 0.5 * C / M
        k[:, :, :, :M][:, :, :, first] = q.view(1, 1, 2, 4 * R, 128).mean(3, keepdim=True)
    k, q = k.bfloat16(), q.bfloat16()
    mk = binding.MorphKV(1, 1, 8, 2, 128, C, R, "sum", "bf16")
    mk.prefill(k, torch.zeros_like(k), q)
    rank = torch.argsort(torch.where(first, 0, M) + torch.arange(M, device=dev))[:C]
    want = torch.cat([torch.sort(rank).values, torch.arange(M, P, device=dev)])
    got = mk.view(0)["pos"][0, :, :C + R].long()
    assert torch.equal(got, want.expand(2, -1))
    mk.close()
