"""Tensors that hold less than a call takes are refused on the host, before anything is launched (sizes and dtypes are looked at before
the device of the tensors, so these calls need no GPU)."""
import pytest
import torch

from paper_2605_08587_b200 import binding, kla_bwd, kla_chunk_fwd, kla_decode_step, kla_decode_steps, kla_dg_decode_step

B, T, H, D = 2, 5, 3, 64


def _bwd():
    x = torch.zeros(B, T, H, D, dtype=torch.bfloat16)
    gate, state = torch.zeros(B, T, H), torch.zeros(B, H, D, D)
    return dict(q=x, k=x, v=x, log_alpha=gate, eta=gate, eps=1e-6, d_out=x, init_state=state, d_final_state=state)


def _decode(n=None, diag=False):
    lead = (B, H) if n is None else (n, B, H)
    x = torch.zeros(*lead, D, dtype=torch.bfloat16)
    return dict(q=x, k=x, v=x, log_alpha=torch.zeros(*lead, D) if diag else torch.zeros(lead), eta=torch.zeros(lead), eps=1e-6,
                state_inout=torch.zeros(B, H, D, D), out=torch.zeros_like(x))


def _forward():
    a = _bwd()
    del a["d_out"], a["d_final_state"]
    return dict(a, out=torch.zeros(B, T, H, D), final_state=torch.zeros(B, H, D, D))


def _less(t):
    return t[..., :-1, :] if t.dim() > 3 else t[..., :-1]


CALLS = [(kla_bwd, _bwd, ["k", "log_alpha", "eta", "init_state", "d_final_state"]),
         (kla_decode_step, _decode, ["k", "log_alpha", "eta", "state_inout", "out"]),
         (kla_decode_steps, lambda: _decode(4), ["k", "log_alpha", "eta", "state_inout", "out"]),
         (kla_dg_decode_step, lambda: _decode(diag=True), ["k", "log_alpha", "eta", "state_inout", "out"]),
         (kla_chunk_fwd, _forward, ["out", "final_state"])]


@pytest.mark.parametrize("call, args, name", [(c, a, n) for c, a, names in CALLS for n in names])
def test_a_tensor_that_is_too_small_is_refused(call, args, name):
    binding.load()
    a = args()
    with pytest.raises(ValueError, match="contiguous CUDA tensor"):   # nothing but the device is wrong
        call(**a)
    a[name] = _less(a[name])
    with pytest.raises(ValueError, match="%s holds fewer elements" % name):
        call(**a)


@pytest.mark.parametrize("name", ["k", "v"])
@pytest.mark.parametrize("call, args", [(kla_bwd, _bwd), (kla_decode_step, _decode), (kla_chunk_fwd, _forward)])
def test_tensors_of_another_dtype_are_refused(call, args, name):
    a = args()
    a[name] = a[name].float()
    with pytest.raises(TypeError, match="share one dtype"):
        call(**a)


@pytest.mark.parametrize("call, args", [(kla_bwd, _bwd), (kla_chunk_fwd, _forward)])
def test_offsets_of_packed_input(call, args):
    cu = torch.tensor([0, 2, T], dtype=torch.int32)
    a = {k: v[:1] if k not in ("eps", "init_state", "final_state", "d_final_state") else v for k, v in args().items()}
    with pytest.raises(ValueError, match="contiguous CUDA tensor"):
        call(**a, cu_seqlens=cu, host_seqlens=cu)
    with pytest.raises(ValueError, match="host_seqlens holds fewer elements"):
        call(**a, cu_seqlens=cu, host_seqlens=cu[:2])
    with pytest.raises(TypeError, match="int32"):
        call(**a, cu_seqlens=cu, host_seqlens=cu.long())
    with pytest.raises(TypeError, match="int32"):
        call(**a, cu_seqlens=cu.long(), host_seqlens=cu)
