"""The compaction after a policy step of coarse-grained eviction at the sizes where its selection changes: one to sixteen slots
per thread, more evictions than candidates in most groups of lanes, one eviction more than nothing, the whole range of
intervals, and evicted tokens on either side of the kept prefix.  Checked against the oracle in lock step."""
import pytest

from paper_2503_00979_b200 import synth
from tests.parity import run_parity_coarse

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,R,T,fusion", [
    (20, 16, 64, "sum"),       # fewer candidates than lanes of a warp, most of them evicted at once
    (1000, 20, 2, "max"),      # 1022 slots
    (1010, 20, 33, "sum"),     # two slots per thread
    (2100, 16, 64, "max"),     # three
    (4200, 16, 17, "sum"),     # five
    (9000, 16, 64, "max"),     # nine
])
def test_sizes(C, R, T, fusion):
    w = synth.Workload("compact", 1, 1, 4, 2, 128, "bf16", C + R + 5, 40, C, R, fusion, 40 + T)
    assert run_parity_coarse(w, T, steps=2 * T + 3, n_units=2).evictions > 0
