"""Prompt-phase scoring at the edges of its forms: a launch for each visit with few and with many runs per unit, runs of two to
fourteen tiles, both visits in one launch with a last cluster of runs that is not full, nothing to select, three blocks of rows."""
import pytest
import torch

from paper_2503_00979_b200 import binding, synth
from tests.parity import run_parity, run_parity_ragged

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,q_heads,kv_heads,P,C,R,fusion", [
    (1, 4, 1, 30000, 900, 20, "sum"),       # 235 tiles, 118 runs of two: every item of the second launch merges them
    (1, 8, 2, 30100, 900, 64, "max"),       # 236 tiles of 256 rows, 59 runs of four
    (3, 8, 2, 5400, 700, 30, "max"),        # 43 tiles, runs of two, the last one shorter
    (1, 32, 8, 12500, 700, 32, "sum"),      # 98 tiles, runs of six
    (2, 8, 2, 60100, 700, 30, "sum"),       # 470 tiles, 34 runs of fourteen
    (96, 32, 8, 500, 300, 32, "max"),       # 3072 tiles of 128 rows: still a launch each; 768 units
    (97, 32, 8, 500, 300, 32, "sum"),       # 3104: one launch, runs shorter than eight tiles by the prompt's end
    (12, 8, 2, 17600, 900, 30, "sum"),      # 3312 tiles: one launch, 18 runs of eight, a last cluster of two
    (9, 28, 4, 8200, 900, 32, "max"),       # 2340 tiles of 256 rows: one launch
    (1, 8, 2, 20000, 20000, 30, "sum"),     # nothing to select: 157 tiles a unit, 53 runs of three in four clusters
    (2, 64, 4, 1500, 500, 100, "sum"),      # 1600 rows in seven pieces, the last of 64
])
def test_forms(layers, q_heads, kv_heads, P, C, R, fusion):
    w = synth.Workload("runs", layers, 1, q_heads, kv_heads, 128, "bf16", P, 2, C, R, fusion, 70 + R)
    rep = run_parity(w, steps=2, n_units=2, kernel="tc", check_F_every=1)
    assert rep.kernel == "tc" and rep.prefill_resyncs <= 1


def test_rows_that_end_in_different_clusters():
    w = synth.Workload("clusters", 4, 3, 8, 2, 128, "bf16", 0, 2, 900, 30, "max", 91)
    rep = run_parity_ragged(w, [40000, 16385, 20000], steps=2, kernel="tc")
    assert rep.units == 4 * 3 * 2


def test_result_does_not_depend_on_the_order_of_items():
    # 3328 tiles: both visits in one launch, items by ticket
    g = torch.Generator(device="cuda:0")
    g.manual_seed(5)
    L, P, C, R = 26, 2000, 700, 32
    k, v = (torch.randn((L, 1, 8, P, 128), generator=g, device="cuda:0").bfloat16() for _ in range(2))
    q = torch.randn((L, 1, 32, R, 128), generator=g, device="cuda:0").bfloat16()
    got = []
    mk = binding.MorphKV(L, 1, 32, 8, 128, C, R, "sum", "bf16")
    for _ in range(6):
        mk.reset()
        mk.prefill(k, v, q)
        got.append([torch.cat([mk.view(l)[name].flatten() for l in range(L)]).clone() for name in ("pos", "ring_c")])
    assert all(torch.equal(a, b) for r in got[1:] for a, b in zip(r, got[0]))
    mk.close()


@pytest.mark.parametrize("P,C", [(1030, 1), (1040, 1003), (4112, 700), (4113, 4000)])
def test_tied_scores_of_many_units(P, C):
    # more units than twice the SMs: the selection in smaller CTAs, up to 4096 candidates; every older token has the same score
    L, R, dev = 38, 16, torch.device("cuda:0")
    gen = torch.Generator(device=dev)
    gen.manual_seed(P)
    q = torch.randn((L, 1, 8, R, 128), generator=gen, device=dev).bfloat16()
    k = torch.zeros((L, 1, 8, P, 128), dtype=torch.bfloat16, device=dev)
    mk = binding.MorphKV(L, 1, 8, 8, 128, C, R, "sum", "bf16")
    mk.prefill(k, k, q)
    want = torch.cat([torch.arange(C, device=dev), torch.arange(P - R, P, device=dev)])
    for l in (0, L // 2, L - 1):
        assert torch.equal(mk.view(l)["pos"][0, :, :C + R].long(), want.expand(8, -1))
    mk.close()
