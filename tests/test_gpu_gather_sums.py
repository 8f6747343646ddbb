"""The prompt phase's gather that takes the window sums along: unit counts at which a CTA's share of the tiles begins and ends
inside a unit and spans several, capacities that end inside a tile (with free slots, which have to come out as zeros), operands
of one, three and eight groups of 32 ring rows, and rows of different lengths.  The sums show in the fused scores of the steps
that follow, which are compared with the oracle's like every other result of the lock-step comparison."""
import pytest
import torch

from paper_2503_00979_b200 import binding, synth
from tests.parity import run_parity, run_parity_ragged

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,q_heads,kv_heads,P,C,R,fusion", [
    (1, 8, 2, 300, 111, 16, "sum"),        # one tile per unit, 64 rows
    (25, 8, 2, 500, 360, 24, "max"),       # 50 units of three tiles: one tile per CTA and two
    (70, 8, 2, 700, 486, 25, "max"),       # 140 units of four tiles, 3.8 per CTA, the last block of the ring a partial one
    (100, 16, 4, 400, 230, 64, "sum"),     # 400 units, 256 rows: two stages
    (3, 2, 2, 600, 400, 200, "max"),       # MHA, 224 rows of seven blocks
    (2, 28, 4, 900, 500, 30, "sum"),       # group padded from 7 to 8
])
def test_sums_of_gathered_rows(layers, q_heads, kv_heads, P, C, R, fusion):
    w = synth.Workload("gather", layers, 1, q_heads, kv_heads, 128, "bf16", P, 12, C, R, fusion, 90 + layers)
    rep = run_parity(w, steps=12, n_units=5, kernel="tc", check_F_every=2)
    assert rep.kernel == "tc" and rep.evictions > 0


def test_rows_of_different_lengths():
    w = synth.Workload("gather_ragged", 20, 3, 8, 2, 128, "bf16", 0, 30, 250, 20, "sum", 6)
    assert run_parity_ragged(w, [700, 262, 9], steps=30).evictions > 0


def test_rows_are_copied_and_free_slots_cleared():
    dev, P, C, R, T = torch.device("cuda:0"), 333, 100, 32, 7
    gen = torch.Generator(device=dev)
    gen.manual_seed(3)
    k, v = (torch.randn((3, 2, 2, P, 128), generator=gen, device=dev).bfloat16() for _ in range(2))
    q = torch.randn((3, 2, 8, R, 128), generator=gen, device=dev).bfloat16()
    mk = binding.MorphKV(3, 2, 8, 2, 128, C, R, "sum", "bf16", evict_interval=T, kernel="tc")
    mk.workspace.fill_(0xff)
    mk.prefill(k, v, q)
    for l in range(3):
        vw = mk.view(l)
        at = vw["pos"][:, :, :C + R].long().unsqueeze(-1).expand(-1, -1, -1, 128)
        for name, src in (("K", k), ("V", v)):
            assert torch.equal(vw[name][:, :, :C + R], torch.gather(src[l], 2, at))
            assert not vw[name][:, :, C + R:].any()
    mk.close()
