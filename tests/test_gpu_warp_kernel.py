"""The warp-level decode kernel (f32, head_dim 64, windows beyond the tcgen05 kernel's) at the sizes where it can go wrong:
cache lengths around a 32-key tile and around a CTA's round of eight, blocks of the ring that end within a window, every
padded group, windows whose sums are not kept (they pass through the kernel 64 rows at a time), CURRENT normalisation,
several CTAs per unit.  Tolerances are those of the lock-step comparison with the oracle."""
import pytest
import torch

from paper_2503_00979_b200 import binding, synth
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


# keys that are not numbers: attention over them is not a number either, wherever they lie among a warp's tiles (one key, a tile
# and more, all of a warp's tiles, all)
@pytest.mark.parametrize("kernel,dtype,d", [("simt", "f32", 64), ("simt", "f32", 128), ("simt", "bf16", 64), ("simt", "bf16", 128),
                                            ("tc", "bf16", 128)])
@pytest.mark.parametrize("C", [300, 1500])
@pytest.mark.parametrize("first,last", [(5, 5), (64, 95), (0, 127), (0, 199)])
def test_keys_that_are_not_numbers(kernel, dtype, d, C, first, last):
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(1)
    k, v, q, q1, k1, v1 = (torch.randn(s, generator=gen, device="cuda:0").to(synth.torch_dtype(dtype))
                           for s in ((1, 1, 1, 200, d), (1, 1, 1, 200, d), (1, 1, 4, 16, d), (1, 1, 4, d), (1, 1, 1, d), (1, 1, 1, d)))
    k[:, :, :, first:last + 1] = float("nan")
    mk = binding.MorphKV(1, 1, 4, 1, d, C, 16, "sum", dtype, kernel=kernel)
    mk.prefill(k, v, q)
    out = mk.decode_step(q1, k1, v1)
    mk.sync()
    assert out.isnan().all()
    mk.close()
