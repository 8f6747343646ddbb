"""Prompts of different lengths in one batch, scored together on the tensor cores (or the CUDA cores), at the lengths
where a row's range ends: on, before and behind the edge of a 128-key tile, of a CTA's share of the tiles, of the window
and of the capacity; rows that select beside rows that keep everything."""
import pytest

from paper_2503_00979_b200 import synth
from tests.parity import run_parity_ragged

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,C,R,q_heads,fusion,kernel", [
    ([128, 129, 127, 256, 257, 1], 90, 32, 8, "sum", "auto"),
    ([31, 32, 33, 122, 123, 121], 90, 32, 8, "max", "auto"),
    ([3000, 2944, 700, 1025, 5], 500, 30, 8, "max", "auto"),
    ([640, 900, 16], 200, 16, 28, "sum", "auto"),
    ([640, 900, 16], 200, 16, 8, "sum", "simt"),
])
def test_rows_ending_at_edges(lens, C, R, q_heads, fusion, kernel):
    kv = 4 if q_heads == 28 else 2
    w = synth.Workload("ragged_edges", 1, len(lens), q_heads, kv, 128, "bf16", 0, 4, C, R, fusion, 31 + len(lens))
    rep = run_parity_ragged(w, lens, steps=4, kernel=kernel)
    assert rep.evictions > 0 and rep.kernel == ("tc" if kernel == "auto" else "simt")


# the tcgen05 kernel's layer calls and its shares cut between units (more units than SMs), which small launches do not reach
@pytest.mark.parametrize("layers,per_layer", [(2, 1), (20, 0)])
def test_rows_on_the_tensor_core_kernel(layers, per_layer):
    w = synth.Workload("ragged_tc", layers, 4, 8, 2, 128, "bf16", 0, 12, 200, 16, "max", 33)
    rep = run_parity_ragged(w, [300, 40, 210, 129], steps=12, kernel="tc", per_layer=per_layer)
    assert rep.evictions > 0 and rep.step_kernel == "tc"
