"""Prompt-phase scoring of some 2300 to 2600 tiles, a launch for each visit of the keys: runs that do not divide the prompt,
one and two operands of window rows, rows of different lengths, the same result again."""
import numpy as np
import pytest
import torch

from paper_2503_00979_b200 import binding, synth
from tests.parity import run_parity, run_parity_ragged

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,q_heads,kv_heads,P,C,R,fusion", [
    (32, 32, 8, 1090, 700, 32, "sum"),      # 2304 tiles, a run for every prompt
    (1, 8, 2, 17500, 1000, 30, "max"),      # 137 tiles, 69 runs of two, the last of one
    (24, 8, 2, 6000, 900, 64, "max"),       # 256 rows: two groups per tile
    (24, 28, 4, 2900, 600, 30, "sum"),      # padded group, 240 rows
    (40, 8, 2, 3500, 800, 100, "sum"),      # two pieces, of 256 and 144 rows
    (72, 4, 4, 1025, 700, 16, "max"),       # 16 rows, a ninth tile of one key
])
def test_selection_of_items_in_one_launch(layers, q_heads, kv_heads, P, C, R, fusion):
    w = synth.Workload("items", layers, 1, q_heads, kv_heads, 128, "bf16", P, 2, C, R, fusion, 40 + layers)
    rep = run_parity(w, steps=2, n_units=4, kernel="tc", check_F_every=1)
    assert rep.kernel == "tc" and rep.evictions == 2 * rep.units and rep.prefill_resyncs <= 1


def test_rows_of_different_lengths_in_one_launch():
    # rows shorter than the window, kept whole, ending inside a run and at its end
    w = synth.Workload("items", 16, 6, 8, 2, 128, "bf16", 0, 3, 900, 32, "sum", 77)
    rep = run_parity_ragged(w, [3000, 7, 500, 1024, 2900, 2048], steps=3, kernel="tc")
    assert rep.units == 16 * 6 * 2


def test_result_does_not_depend_on_the_order_of_items():
    g = torch.Generator(device="cuda:0")
    g.manual_seed(5)
    L, P, C, R = 24, 1500, 700, 32
    k, v = (torch.randn((L, 1, 8, P, 128), generator=g, device="cuda:0").bfloat16() for _ in range(2))
    q = torch.randn((L, 1, 32, R, 128), generator=g, device="cuda:0").bfloat16()
    got = []
    mk = binding.MorphKV(L, 1, 32, 8, 128, C, R, "sum", "bf16")
    for _ in range(4):
        mk.reset()
        mk.prefill(k, v, q)
        got.append([torch.cat([mk.view(l)[name].flatten() for l in range(L)]).clone() for name in ("pos", "ring_c")])
    assert all(torch.equal(a, b) for r in got[1:] for a, b in zip(r, got[0]))
    mk.close()


def test_keys_far_above_those_before_them():
    # the reference of a row's sums is far below the keys that follow: 2^40, and beyond what a float holds
    L, P, C, R = 40, 8200, 300, 8
    k, v = (torch.randn((L, 1, 1, P, 128), device="cuda:0").mul_(0.1).bfloat16() for _ in range(2))
    q = torch.ones((L, 1, 4, R, 128), device="cuda:0").bfloat16()
    for p, x in ((40, 1.0), (200, 3.0), (900, 6.0), (1900, 12.0), (4000, 24.0)):
        k[:, :, :, p] = x
    mk = binding.MorphKV(L, 1, 4, 1, 128, C, R, "sum", "bf16")
    mk.prefill(k, v, q)
    s = torch.einsum("lrd,lkd->lrk", q[:, 0].reshape(L, 4 * R, 128).double(), k[:, 0, 0].double()) / np.sqrt(128)
    mask = torch.arange(P, device="cuda:0")[None] <= (P - R + torch.arange(4 * R, device="cuda:0") % R)[:, None]
    c = torch.logsumexp(s.masked_fill(~mask, -np.inf), -1) / np.log(2)
    for l in (0, L - 1):
        ring = mk.view(l)["ring_c"][0, 0]             # [ring slot][head]; the window starts at slot (P - R) % R
        want = c[l].view(4, R).T.roll((P - R) % R, 0)
        assert torch.allclose(ring[:, :4].double(), want, rtol=1e-6, atol=1e-5)
    mk.close()
