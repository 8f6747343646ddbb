"""Inputs that do not start on the boundary of the widest load: decode tensors at any element, window queries at a multiple of
four, keys and values of a prompt refused.  Results are those of the same values on aligned tensors."""
import numpy as np
import pytest
import torch

from paper_2503_00979_b200 import binding, synth

pytestmark = pytest.mark.gpu


def _at(t, elements):
    """A copy of t that starts `elements` elements behind a 256-byte boundary."""
    buf = torch.empty(t.numel() + 512, dtype=t.dtype, device=t.device)
    first = (-buf.data_ptr() % 256) // t.element_size() + elements
    return buf[first:first + t.numel()].copy_(t.reshape(-1)).view(t.shape)


# outputs of the two scoring paths of the prompt phase (tensor cores; CUDA cores where q_window is not on 16 bytes) differ by
# rounding: at most one step of bf16 in a value, 2^-7 of it, beside 2e-2 for a near tie that falls the other way
@pytest.mark.parametrize("kernel,dtype,d,C,q_at,in_at", [("tc", "bf16", 128, 200, 4, 1), ("tc", "bf16", 128, 1500, 8, 3),
                                                         ("auto", "bf16", 128, 1500, 4, 1), ("simt", "bf16", 64, 200, 4, 5),
                                                         ("simt", "f32", 64, 200, 4, 1)])
@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("per_layer", [False, True])
def test_tensors_that_start_anywhere(kernel, dtype, d, C, q_at, in_at, ragged, per_layer):
    w = synth.Workload("offset", 2, 2, 8, 2, d, dtype, C + 100, 6, C, 16, "sum", 77)
    dev, tdt = torch.device("cuda:0"), synth.torch_dtype(dtype)
    st = synth.Stream(w, dev)
    P = w.prompt_len
    k, v = (x.to(tdt).contiguous() for x in st.kv(np.arange(P)))
    qw = st.q(np.arange(P - w.R, P)).to(tdt).contiguous()
    kk, vv = st.kv(np.arange(P, P + w.steps))
    q1, k1, v1 = (x.permute(3, 0, 1, 2, 4).to(tdt).contiguous() for x in (st.q(np.arange(P, P + w.steps)), kk, vv))
    got = []
    for at_q, at in ((0, 0), (q_at, in_at)):
        mk = binding.MorphKV(2, 2, 8, 2, d, C, w.R, w.fusion, dtype, kernel=kernel)
        if ragged:
            mk.prefill_ragged(k, v, _at(qw, at_q), [P, P - 60])
        else:
            mk.prefill(k, v, _at(qw, at_q))
        outs = []
        for i in range(w.steps):
            if per_layer:
                outs += [mk.decode_step_layer(l, *(_at(x[i, l], at) for x in (q1, k1, v1)), _at(q1[i, l], at)) for l in range(2)]
            else:
                outs.append(mk.decode_step(*(_at(x[i], at) for x in (q1, k1, v1)), _at(q1[i], at)))
        mk.sync()
        got.append(torch.stack(outs).float())
        mk.close()
    assert ((got[0] - got[1]).abs() <= 2e-2 + 2 ** -7 * got[0].abs()).all()


def test_prompt_tensors_that_cannot_be_read_are_refused():
    mk = binding.MorphKV(1, 1, 8, 2, 128, 64, 16, "sum", "bf16")
    k = torch.zeros((1, 1, 2, 50, 128), dtype=torch.bfloat16, device="cuda:0")
    qw = torch.zeros((1, 1, 8, 16, 128), dtype=torch.bfloat16, device="cuda:0")
    for args in ((_at(k, 4), k, qw), (k, _at(k, 1), qw), (k, k, _at(qw, 2))):
        assert binding.mkv_prefill(mk.ctx, *args, 50) == binding.INVALID_ARG
        assert binding.mkv_prefill_ragged(mk.ctx, *args, [50], 50) == binding.INVALID_ARG
    mk.prefill(k, k, qw)
    mk.close()
