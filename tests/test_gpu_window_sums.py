"""The fused scores kept across steps (block by block of the recent-query ring) at the sizes where blocks end: windows
that are not a multiple of a block, of one block and two, of many; laps of the ring; prompts that end on either side of
a block's end, shorter than the window, and slots rearranged through a view in mid-sequence."""
import numpy as np
import pytest
import torch

from paper_2503_00979_b200 import binding, synth
from tests.parity import run_parity

pytestmark = pytest.mark.gpu


# a step opens a block of 8 slots at G = 4 (of 32 at G = 1, of 16 beyond 96 slots); two laps and a bit are decoded, F of
# every candidate compared with the oracle's on every third step (rows are f32 sums of at most R*G weights: 1e-3 is
# thousands of roundings away)
@pytest.mark.parametrize("fusion", ["sum", "max"])
@pytest.mark.parametrize("q_heads,R,P", [(8, 8, 151), (8, 9, 152), (8, 16, 160), (8, 23, 161), (8, 17, 7), (2, 33, 150), (2, 64, 159),
                                         (14, 21, 140), (32, 17, 131), (8, 97, 203), (8, 113, 224)])
def test_blocks_and_laps(fusion, q_heads, R, P):
    w = synth.Workload("blocks", 1, 1, q_heads, 2, 128, "bf16", P, max(0, 130 + R - P) + 2 * R + 19, 130, R, fusion, 600 + R)
    rep = run_parity(w, steps=w.steps, n_units=2, kernel="tc", check_F_every=3)
    assert rep.kernel == "tc" and rep.evictions > 0


@pytest.mark.parametrize("per_layer", [False, True])
def test_slots_rearranged_between_steps(per_layer):
    # slot order is free: a holder of a view may move rows (K, V, pos together) before any step that follows the call
    # which handed the view out
    w = synth.Workload("moved", 2, 1, 8, 2, 128, "bf16", 200, 21, 120, 24, "sum", 9)
    dev = torch.device("cuda:0")
    st = synth.Stream(w, dev)
    k, v = st.kv(np.arange(w.prompt_len))
    qw = st.q(np.arange(w.prompt_len - w.R, w.prompt_len))
    got = []
    for swap in (False, True):
        mk = binding.MorphKV(2, 1, 8, 2, 128, w.C, w.R, w.fusion, "bf16")
        mk.prefill(k.bfloat16().contiguous(), v.bfloat16().contiguous(), qw.bfloat16().contiguous())
        outs = []
        for i in range(w.steps):
            if swap and i in (5, 11, 12):
                mk.sync()
                for l in range(w.layers):
                    vw = mk.view(l)
                    perm = torch.randperm(vw["count"], device=dev)
                    for name in ("K", "V", "pos"):
                        vw[name][:, :, :vw["count"]] = vw[name][:, :, :vw["count"]][:, :, perm].clone()
            p = [w.prompt_len + i]
            kk, vv = st.kv(p)
            q1, k1, v1 = (x[:, :, :, 0].bfloat16().contiguous() for x in (st.q(p), kk, vv))
            if per_layer:
                outs.append(torch.stack([mk.decode_step_layer(l, q1[l], k1[l], v1[l]) for l in range(w.layers)]).float())
            else:
                outs.append(mk.decode_step(q1, k1, v1).float())
        mk.sync()
        got.append((torch.stack(outs), [torch.sort(mk.view(l)["pos"][0, :, :w.C + w.R], dim=-1).values.clone() for l in range(w.layers)]))
        mk.close()
    assert all(torch.equal(a, b) for a, b in zip(got[0][1], got[1][1]))
    assert (got[0][0] - got[1][0]).abs().max() < 2e-2


# ---- the same where no call into the library tells of the move: between replays of recorded steps, and before a recording
# that is not replayed before the next direct step; and slots moved to and fro while the cache fills (the steps in between
# score finished blocks and evict nothing)
def _steps(mode, kernel, dtype="bf16", layers=2, batch=1, C=120, P=200, G=4, steps=24, T=1):
    """Outputs and retained positions of `steps` steps; mode None: nothing is moved."""
    w = synth.Workload("moved", layers, batch, 2 * G, 2, 128, dtype, P, steps, C, 24, "sum", 9)
    dev, tdt = torch.device("cuda:0"), synth.torch_dtype(dtype)
    st = synth.Stream(w, dev)
    k, v = st.kv(np.arange(P))
    qw = st.q(np.arange(P - w.R, P))
    kk, vv = st.kv(np.arange(P, P + steps))
    q1, k1, v1 = (x.permute(3, 0, 1, 2, 4).to(tdt).contiguous() for x in (st.q(np.arange(P, P + steps)), kk, vv))
    mk = binding.MorphKV(layers, batch, 2 * G, 2, 128, w.C, w.R, w.fusion, dtype, kernel=kernel, evict_interval=T)
    mk.prefill(*(x.to(tdt).contiguous() for x in (k, v, qw)))
    views = [mk.view(l) for l in range(layers)]
    gen = torch.Generator(device=dev)
    gen.manual_seed(3)

    def move(perm=None):
        torch.cuda.synchronize()
        for l, vw in enumerate(views):
            if mode == "to and fro":
                mk.view(l)
            n = int((vw["pos"][0, 0] >= 0).sum())
            p = torch.randperm(n, device=dev, generator=gen) if perm is None else perm
            for name in ("K", "V", "pos"):
                vw[name][:, :, :n] = vw[name][:, :, :n][:, :, p].clone()
        return p

    out = torch.empty_like(q1)
    mk.decode_step(q1[0], k1[0], v1[0], out[0])          # the views are older than this step
    i = 1
    if mode in ("replays", "recorded after the move"):
        ins = [x[1:3].clone() for x in (q1, k1, v1)]
        o2 = torch.empty_like(out[:2])
        if mode != "replays":
            views = [mk.view(l) for l in range(layers)]
            move()
        g = torch.cuda.CUDAGraph()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(g, stream=side):
            for j in range(2):
                mk.decode_step(ins[0][j], ins[1][j], ins[2][j], o2[j], stream=torch.cuda.current_stream())
        mk.sync()
        if mode != "replays":
            mk.decode_step(q1[1], k1[1], v1[1], out[1])
            i = 2
        while i + 1 < steps:
            if mode == "replays" and i in (5, 9, 15):
                move()
            for dst, src in zip(ins, (q1, k1, v1)):
                dst.copy_(src[i:i + 2])
            g.replay()
            torch.cuda.synchronize()
            out[i:i + 2] = o2
            i += 2
        mk.sync()
        for i in range(i, steps):
            mk.decode_step(q1[i], k1[i], v1[i], out[i])
        del g
    else:
        for i in range(1, steps):
            if mode == "to and fro" and i == 5:
                perm = move()
            if mode == "to and fro" and i == 14:
                n = int((views[0]["pos"][0, 0] >= 0).sum())
                back = torch.cat([torch.argsort(perm), torch.arange(len(perm), n, device=dev)])
                move(back)
            mk.decode_step(q1[i], k1[i], v1[i], out[i])
    mk.sync()
    pos = [torch.sort(mk.view(l)["pos"][:, :, :mk.view(l)["count"]], dim=-1).values.clone() for l in range(layers)]
    mk.close()
    return out.float(), pos


@pytest.mark.parametrize("mode", ["replays", "recorded after the move"])
@pytest.mark.parametrize("kernel,dtype,layers,C", [("tc", "bf16", 2, 120), ("tc", "bf16", 2, 700), ("tc", "bf16", 80, 120),
                                                   ("auto", "bf16", 2, 1200), ("simt", "f32", 2, 120)])
def test_slots_rearranged_without_a_call(mode, kernel, dtype, layers, C):
    # one CTA per unit, units shared by several CTAs, several units per CTA; a cluster per unit; f32
    shape = dict(kernel=kernel, dtype=dtype, layers=layers, C=C, P=C + 80)
    want, got = _steps(None, **shape), _steps(mode, **shape)
    assert all(torch.equal(a, b) for a, b in zip(want[1], got[1]))
    assert (want[0] - got[0]).abs().max() < 2e-2


@pytest.mark.parametrize("kernel,dtype", [("tc", "bf16"), ("simt", "f32")])
def test_slots_rearranged_to_and_fro_while_the_cache_fills(kernel, dtype):
    shape = dict(kernel=kernel, dtype=dtype, C=150, P=150, steps=60)       # evicts from the 25th step on
    want, got = _steps(None, **shape), _steps("to and fro", **shape)
    assert all(torch.equal(a, b) for a, b in zip(want[1], got[1]))
    assert (want[0] - got[0]).abs().max() < 2e-2
