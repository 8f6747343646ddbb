"""Launches of a tcgen05 context too small to fill the chip, which the warp-level kernel takes (a cluster per unit): the
cluster sizes, ranges and blocks at which it can go wrong, steps that alternate between layer calls and whole-stack calls,
layers back to back (a layer's launch starts before the one before it has ended), and the neighbours that stay with
the tcgen05 kernel.  Tolerances are those of the lock-step comparison with the oracle."""
import numpy as np
import pytest
import torch

from paper_2503_00979_b200 import binding, synth
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
    (2, 1, 64, 4, 200, 20, "sum", 1),      # group of 16: blocks of four slots
    (2, 1, 32, 2, 300, 100, "max", 1),     # group of 16: two blocks of 128 rows do not fit, tcgen05 kernel
    (3, 1, 48, 4, 1000, 9, "sum", 1),      # group of 12 -> 16, four units of eight CTAs, a last block of one slot
    (2, 5, 16, 8, 400, 16, "max", 1),      # 40 units of four CTAs: more than the chip's SMs, tcgen05 kernel
    (2, 1, 8, 2, 1010, 16, "sum", 0),      # whole stack: 4 units of nine CTAs
    (2, 1, 8, 2, 1000, 16, "max", 0),      # ... of eight rounds: tcgen05 kernel
    (2, 4, 16, 2, 1010, 16, "max", 1),     # group of 8: 8 units of nine CTAs, 72 of 74
    (2, 7, 16, 2, 900, 16, "sum", 1),      # ... 14 units of eight, of 15 that are resident at once
    (2, 8, 16, 2, 900, 16, "sum", 1),      # ... 16 units: tcgen05 kernel
])
def test_layer_calls(layers, batch, q_heads, kv_heads, C, R, fusion, per_layer):
    w = synth.Workload("small", layers, batch, q_heads, kv_heads, 128, "bf16", C + R - 3, min(2 * R, 60) + 14, C, R, fusion, 50 + R)
    rep = run_parity(w, steps=w.steps, n_units=4, per_layer=per_layer, check_F_every=5)
    assert rep.kernel == "tc" and rep.evictions > 0
    units, rounds, wide = (layers if per_layer == 0 else 1) * batch * kv_heads, -(-(C + R) // 128), q_heads // kv_heads > 4
    ctas = min(rounds, 16)
    small = units * ctas <= (74 if wide else 148) and (per_layer != 0 or rounds > 8)
    small |= bool(wide and per_layer and ctas >= 4 and units <= 18 // ctas * 7 + 11 // ctas)
    assert rep.step_kernel == ("simt" if small and (q_heads // kv_heads, R) != (16, 100) else "tc")


def test_coarse_grained_and_ragged():
    w = synth.Workload("small_T", 1, 1, 8, 2, 128, "bf16", 330, 40, 250, 32, "max", 5)
    assert run_parity_coarse(w, T=5, steps=23, n_units=2).evictions > 0
    w = synth.Workload("small_ragged", 2, 3, 8, 2, 128, "bf16", 0, 40, 250, 20, "sum", 6)
    assert run_parity_ragged(w, [400, 262, 5], steps=40, per_layer=1).evictions > 0


# Layer calls with nothing between them, so that a layer's launch does start before the one before it has ended: outputs,
# positions and normalisers bit for bit those of the same calls with a synchronisation after each.  `order`: all layers on one
# stream, a stream for each layer (two launches of a layer are then neighbours in their stream; nothing orders the layers
# against one another), or layer calls alternating with whole-stack steps (a state copy goes ahead of the layer's launch; both
# contexts take the same calls).
@pytest.mark.parametrize("order", ["one stream", "a stream per layer", "alternating"])
@pytest.mark.parametrize("layers,C,kernel,dtype,T", [(2, 90, "auto", "bf16", 1), (3, 500, "auto", "bf16", 1), (2, 90, "auto", "bf16", 5),
                                                     (2, 90, "tc", "bf16", 1), (3, 70, "simt", "f32", 1)])
def test_layer_calls_back_to_back(layers, C, kernel, dtype, T, order):
    w = synth.Workload("back_to_back", layers, 1, 8, 2, 128, dtype, C + 16, 200, C, 16, "max", 8)
    dev, tdt = torch.device("cuda:0"), synth.torch_dtype(dtype)
    st = synth.Stream(w, dev)
    P = w.prompt_len
    k, v = st.kv(np.arange(P))
    qw = st.q(np.arange(P - w.R, P))
    kk, vv = st.kv(np.arange(P, P + w.steps))
    q1, k1, v1 = (x.permute(3, 0, 1, 2, 4).to(tdt).contiguous() for x in (st.q(np.arange(P, P + w.steps)), kk, vv))
    got = []
    for wait in (True, False):
        mk = binding.MorphKV(layers, 1, 8, 2, 128, C, w.R, w.fusion, dtype, kernel=kernel, evict_interval=T)
        mk.prefill(*(x.to(tdt).contiguous() for x in (k, v, qw)))
        streams = [torch.cuda.Stream() for _ in range(layers if order == "a stream per layer" else 1)]
        out = torch.empty_like(q1)
        calls = [(i, l, (q1[i, l], k1[i, l], v1[i, l], out[i, l])) for i in range(w.steps) for l in range(layers)]
        torch.cuda.synchronize()
        for i, l, x in calls:
            s = streams[l % len(streams)]
            if order == "alternating" and i % 3 == 2:
                if l == 0:
                    mk.decode_step(q1[i], k1[i], v1[i], out[i], stream=s)
            else:
                mk.decode_step_layer(l, *x, stream=s)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        mk.sync()
        views = [mk.view(l) for l in range(layers)]
        got.append([out] + [vw[name].clone() for vw in views for name in ("pos", "ring_c", "F")])
        mk.close()
    assert all(torch.equal(a, b) for a, b in zip(*got))
