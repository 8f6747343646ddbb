"""A context works in whatever memory it is given: nothing may depend on what the workspace held before the prompt
phase.  The workspace is filled with 0xff bytes (NaN in every float format, -1 in every integer) and the usual lock-step
comparison with the oracle follows."""
import pytest

from paper_2503_00979_b200 import binding, synth
from tests.parity import run_parity

pytestmark = pytest.mark.gpu


# (dtype, d, kv heads, prompt, C, R, fusion): free slots inside the last tile and whole free tiles, empty ring rows, a
# cache that fills up and starts evicting, a padded group, both kernels
@pytest.mark.parametrize("dtype,d,q_heads,P,C,R,fusion,steps", [
    ("bf16", 128, 8, 130, 250, 16, "sum", 170),
    ("bf16", 128, 8, 10, 90, 32, "max", 140),
    ("bf16", 128, 14, 40, 70, 20, "sum", 90),
    ("bf16", 128, 8, 300, 200, 40, "max", 60),
    ("f32", 64, 8, 20, 70, 24, "sum", 110),
    ("bf16", 64, 8, 200, 100, 32, "max", 50),
])
def test_parity_in_a_workspace_full_of_nans(monkeypatch, dtype, d, q_heads, P, C, R, fusion, steps):
    class Poisoned(binding.MorphKV):
        def __init__(self, *a, **k):
            super().__init__(*a, **k)
            self.workspace.fill_(0xFF)

    monkeypatch.setattr(binding, "MorphKV", Poisoned)
    w = synth.Workload("poisoned", 1, 2, q_heads, 2, d, dtype, P, steps, C, R, fusion, 77)
    rep = run_parity(w, steps=steps, n_units=4, chunk=16, check_F_every=7)
    assert rep.evictions > 0
