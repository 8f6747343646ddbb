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
