"""Launches of a tcgen05 context too small to fill the chip, which the warp-level kernel takes (a cluster per unit): the
cluster sizes, ranges and blocks at which it can go wrong, steps that alternate between layer calls and whole-stack calls,
two layers back to back (a layer's launch starts before the one before it has ended), and the neighbours that stay with
the tcgen05 kernel.  Tolerances are those of the lock-step comparison with the oracle."""
import pytest

from paper_2503_00979_b200 import synth
from tests.parity import run_parity, run_parity_coarse, run_parity_ragged

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,batch,q_heads,kv_heads,C,R,fusion,per_layer", [
    (2, 1, 8, 2, 90, 16, "max", 1),        # one CTA per unit
    (2, 1, 8, 2, 100, 30, "sum", 2),       # 130 slots: two CTAs, the second with a tile of two keys
    (3, 1, 28, 4, 1000, 30, "max", 1),     # nine CTAs, group 7 -> 8
    (2, 1, 16, 2, 2040, 9, "sum", 1),      # seventeen rounds over sixteen CTAs
    (1, 1, 16, 1, 600, 12, "max", 0),      # group of 16, whole stack of one layer
    (2, 2, 4, 4, 500, 64, "sum", 2),       # MHA
    (2, 1, 8, 2, 300, 97, "max", 1),       # blocks of 64 rows
    (2, 1, 64, 4, 200, 20, "sum", 1),      # group of 16: two blocks of 128 rows do not fit, tcgen05 kernel
    (2, 5, 16, 8, 400, 16, "max", 1),      # 40 units of four CTAs: more than the chip's SMs, tcgen05 kernel
])
def test_layer_calls(layers, batch, q_heads, kv_heads, C, R, fusion, per_layer):
    w = synth.Workload("small", layers, batch, q_heads, kv_heads, 128, "bf16", C + R - 3, min(2 * R, 60) + 14, C, R, fusion, 50 + R)
    rep = run_parity(w, steps=w.steps, n_units=4, per_layer=per_layer, check_F_every=5)
    assert rep.kernel == "tc" and rep.evictions > 0


def test_coarse_grained_and_ragged():
    w = synth.Workload("small_T", 1, 1, 8, 2, 128, "bf16", 330, 40, 250, 32, "max", 5)
    assert run_parity_coarse(w, T=5, steps=23, n_units=2).evictions > 0
    w = synth.Workload("small_ragged", 2, 3, 8, 2, 128, "bf16", 0, 40, 250, 20, "sum", 6)
    assert run_parity_ragged(w, [400, 262, 5], steps=40, per_layer=1).evictions > 0
