"""The warp-level decode kernel (f32, head_dim 64, windows beyond the tcgen05 kernel's) at the sizes where it can go wrong:
cache lengths around a 32-key tile and around a CTA's round of eight, blocks of the ring that end within a window, every
padded group, windows whose sums are not kept (they pass through the kernel 64 rows at a time), CURRENT normalisation,
several CTAs per unit.  Tolerances are those of the lock-step comparison with the oracle."""
import pytest

from paper_2503_00979_b200 import synth
from tests.parity import run_parity

pytestmark = pytest.mark.gpu


def _run(dtype, d, q_heads, kv_heads, C, R, P, fusion, **kw):
    steps = max(0, C + R - P) + min(2 * R, 60) + 11
    w = synth.Workload("warp", 1, 1, q_heads, kv_heads, d, dtype, P, steps, C, R, fusion, 70 + R)
    rep = run_parity(w, steps=steps, n_units=2, kernel="simt", check_F_every=5, **kw)
    assert rep.kernel == "simt" and rep.evictions > 0


@pytest.mark.parametrize("dtype,d", [("bf16", 64), ("f32", 64), ("bf16", 128), ("f32", 128)])
@pytest.mark.parametrize("q_heads,C,R,P,fusion", [(2, 22, 9, 33, "max"), (2, 31, 33, 64, "sum"), (4, 230, 26, 260, "max"),
                                                  (6, 256, 5, 270, "sum"), (8, 60, 17, 40, "max"), (14, 250, 10, 300, "max"),
                                                  (32, 70, 7, 90, "max"), (32, 513, 3, 600, "sum")])
def test_tiles_blocks_and_groups(dtype, d, q_heads, C, R, P, fusion):
    _run(dtype, d, q_heads, 2, C, R, P, fusion)


@pytest.mark.parametrize("dtype,d,q_heads,R,norm", [("bf16", 64, 14, 300, "frozen"), ("f32", 64, 8, 700, "frozen"),
                                                    ("bf16", 64, 8, 40, "current"), ("f32", 128, 6, 30, "current")])
def test_windows_that_pass_through_in_pieces(dtype, d, q_heads, R, norm):
    _run(dtype, d, q_heads, 2, 90, R, R + 95, "sum", norm=norm)


@pytest.mark.parametrize("splits", [3, 40])
def test_several_ctas_per_unit(splits):
    _run("bf16", 64, 8, 2, 700, 20, 730, "max", splits=splits)
