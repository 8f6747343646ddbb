"""Shares of the tensor-core kernel that are cut between units, and units cut into equal parts of their own: unit counts on
either side of a multiple of the grid, one tile and several, and fills that cross from one kind of share to the other while
the cache fills.  Tolerances are those of the lock-step comparison with the oracle."""
import pytest

from paper_2503_00979_b200 import synth
from tests.parity import run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,q_heads,kv_heads,P,C,R,fusion", [
    (74, 8, 2, 250, 240, 16, "sum"),       # 148 units of two tiles: one per CTA
    (149, 4, 1, 110, 100, 16, "max"),      # one more unit than CTAs, one tile each: two units on one CTA
    (75, 8, 2, 620, 610, 16, "sum"),       # 150 units of five tiles: equal shares, cut inside units
    (160, 4, 1, 500, 600, 16, "max"),      # whole units up to 512 slots, shares cut inside units beyond
    (37, 16, 4, 500, 500, 16, "sum"),      # 148 units, from four tiles to five
    (5, 16, 4, 1100, 1000, 16, "max"),     # 20 units in seven parts each
    (2, 4, 1, 1100, 1000, 16, "sum"),      # 2 units in eight parts each
])
def test_shares(layers, q_heads, kv_heads, P, C, R, fusion):
    steps = max(0, C + R - P) + 20
    w = synth.Workload("shares", layers, 1, q_heads, kv_heads, 128, "bf16", P, steps, C, R, fusion, 70 + layers)
    rep = run_parity(w, steps=steps, n_units=5, kernel="tc", check_F_every=7)
    assert rep.kernel == "tc" and rep.evictions > 0


# units shared by more CTAs than the epilogue merges by itself: nine and more segments of one to three tiles, the last with a
# few keys, while the cache fills and when it evicts
@pytest.mark.parametrize("splits", [9, 13, 26])
@pytest.mark.parametrize("q_heads,R,fusion", [(2, 33, "sum"), (8, 16, "max"), (14, 30, "sum"), (32, 9, "max")])
def test_many_segments(splits, q_heads, R, fusion):
    w = synth.Workload("segments", 2, 1, q_heads, 2, 128, "bf16", 3200, 30, 3220 - R, R, fusion, 90 + R)
    rep = run_parity(w, steps=w.steps, n_units=4, kernel="tc", splits=splits, check_F_every=5)
    assert rep.kernel == "tc" and rep.evictions > 0
