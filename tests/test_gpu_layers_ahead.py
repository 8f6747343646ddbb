"""Layer calls on the tcgen05 kernel that start before the launch ahead of them has ended: the same calls with a synchronisation after
each give the same outputs, positions, scores and normalisers bit for bit, and what is left of another launch does not
count towards the limit of a layer's own waits."""
import pytest
import torch

from paper_2503_00979_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _inputs(layers, batch, q_heads, kv_heads, P, R, n, seed, dtype=torch.bfloat16):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    def rnd(*shape):
        return torch.randn(shape, generator=gen, device=DEV).to(dtype)
    return (rnd(layers, batch, kv_heads, P, 128), rnd(layers, batch, kv_heads, P, 128), rnd(layers, batch, q_heads, min(R, P), 128),
            rnd(n, layers, batch, q_heads, 128), rnd(n, layers, batch, kv_heads, 128), rnd(n, layers, batch, kv_heads, 128))


@pytest.mark.parametrize("layers,batch,q_heads,kv_heads,C,R,kw,lens", [
    (2, 1, 8, 2, 1000, 16, {}, None),                                       # units shared by eight CTAs
    (2, 1, 32, 8, 3000, 32, dict(evict_interval=5), None),                  # a compaction between the layers
    (3, 1, 16, 2, 1100, 64, {}, None),                                      # group of 8: blocks of the window
    (2, 1, 32, 2, 700, 24, {}, None),                                       # group of 16
    (2, 20, 32, 8, 500, 16, {}, None),                                      # more units than CTAs: items of several units
    (2, 2, 16, 2, 600, 40, dict(norm="current"), None),                     # the window in chunks
    (2, 4, 8, 2, 900, 20, {}, [1300, 900, 40, 925]),                        # rows of different lengths
    (4, 1, 8, 2, 600, 16, dict(full_layers=2, max_tokens=1200), None),      # layers that keep every token, then others
    (2, 1, 32, 8, 2000, 200, dict(profile="stored"), None),                 # a window of more than 256 rows
])
def test_back_to_back(layers, batch, q_heads, kv_heads, C, R, kw, lens):
    n, P = 70, max(lens) if lens else C + R - 5
    k, v, qw, q, kn, vn = _inputs(layers, batch, q_heads, kv_heads, P, R, n, 7)
    got = []
    for wait in (True, False):
        mk = binding.MorphKV(layers, batch, q_heads, kv_heads, 128, C, R, "max", "bf16", kernel="tc", **kw)
        assert mk.step_kernel(True) == "tc"
        if lens:
            mk.prefill_ragged(k, v, qw, lens)
        else:
            mk.prefill(k, v, qw)
        out = torch.zeros_like(q)
        for i in range(n):
            for l in range(layers):
                mk.decode_step_layer(l, q[i, l], kn[i, l], vn[i, l], out[i, l])
                if wait:
                    torch.cuda.synchronize()
        mk.sync()
        got.append([out] + [mk.view(l)[name].clone() for l in range(layers) for name in ("pos", "ring_c", "F")])
        mk.close()
    assert all(torch.equal(a, b) for a, b in zip(*got))


def test_limit_of_a_wait_leaves_out_the_launch_ahead():
    # another context's step keeps a few SMs busy for far longer than the limit; the layer behind it is on the others by then
    limit = 100_000                                       # clock ticks: about 50 us
    k, v, qw, q, kn, vn = _inputs(2, 1, 8, 2, 1016, 16, 4, 11)
    slow_in = _inputs(1, 1, 8, 1, 240016, 16, 1, 12, torch.float32)
    slow = binding.MorphKV(1, 1, 8, 1, 128, 240000, 16, "sum", "f32")
    slow.prefill(*slow_in[:3])
    slow_step = [t[0] for t in slow_in[3:]]
    slow_out = slow.decode_step(*slow_step)
    got = []
    for cycles in (0, limit):
        mk = binding.MorphKV(2, 1, 8, 2, 128, 1000, 16, "sum", "bf16", kernel="tc", wait_limit_cycles=cycles)
        mk.prefill(k, v, qw)
        out = torch.zeros_like(q)
        for i in range(4):
            mk.decode_step_layer(0, q[i, 0], kn[i, 0], vn[i, 0], out[i, 0])
            if cycles:
                slow.decode_step(*slow_step, slow_out)
            mk.decode_step_layer(1, q[i, 1], kn[i, 1], vn[i, 1], out[i, 1])
        mk.sync()
        got.append(out)
        mk.close()
    assert torch.equal(*got)
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    a.record()
    slow.decode_step(*slow_step, slow_out)
    b.record()
    slow.sync()
    assert a.elapsed_time(b) * 1e-3 * 2.0e9 > 4 * limit   # a step takes well beyond the limit at any clock
    slow.close()
