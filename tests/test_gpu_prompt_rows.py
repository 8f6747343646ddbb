"""Batches of prompts of different lengths whose units take their items from a table of the rows' lengths: more rows than the table
has entries, rows of one to eight tiles, one long row among short ones."""
import pytest

from paper_2503_00979_b200 import synth
from tests.parity import run_parity_ragged

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,kv_heads,lens,C,R", [
    (1, 1, [128 * (1 + b % 8) - 7 * (b % 5) for b in range(530)], 300, 8),      # two rows to an entry, 2385 tiles
    (3, 2, [6100] + [130, 1, 700, 127, 128, 129, 900] * 2, 400, 16),            # most rows kept whole
    (24, 2, [3000, 2900, 2999, 2945], 500, 32),                                  # nearly equal, 4512 tiles
])
def test_rows_against_the_oracle(layers, kv_heads, lens, C, R):
    w = synth.Workload("rows", layers, len(lens), 4 * kv_heads, kv_heads, 128, "bf16", 0, 1, C, R, "sum", 60 + R)
    rep = run_parity_ragged(w, lens, steps=1, kernel="tc")
    assert rep.units == layers * len(lens) * kv_heads and rep.prefill_resyncs <= 1
