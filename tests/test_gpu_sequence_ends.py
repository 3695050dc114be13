"""Packed sequences of lengths around the 64-token tiles, beside sequences whose inputs are not finite: TMA fetches whole tiles, so
the last chunk of a sequence arrives with its neighbour's tokens in it, and nothing of them may reach a result."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL_BF16, np64, rel_err
from paper_2605_08587_b200 import kla_bwd, kla_chunk_fwd, workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LENS = [1, 70, 63, 5, 64, 0, 65, 130, 128, 3, 129]
CLEAN = [0, 2, 4, 6, 8, 10]   # the sequences between them hold NaN and infinities
GRADS = ["dq", "dk", "dv", "dlog_alpha", "deta"]


def _packed(d):
    cu = np.concatenate([[0], np.cumsum(LENS)])
    w = W.config2(B=1, H=3, T=int(cu[-1]), d=d, seed=640 + d)
    g = torch.Generator().manual_seed(d)
    d_out = torch.randn(w.v.shape, generator=g).to(w.v.dtype)
    state = 0.02 * torch.randn(len(LENS), 3, d, d, generator=g)
    d_state = torch.randn(len(LENS), 3, d, d, generator=g)
    for n in range(len(LENS)):
        if n not in CLEAN:
            for i, x in enumerate((w.q, w.k, w.v, d_out)):
                x[:, cu[n]:cu[n + 1]] = [float("nan"), float("inf"), float("-inf"), float("nan")][i]
    return w, cu, d_out, state, d_state


def _cu(x):
    t = torch.tensor(x, dtype=torch.int32)
    return t.to(DEV), t


@pytest.mark.parametrize("d", [64, 128])
def test_backward_of_a_sequence_knows_nothing_of_its_neighbours(d):
    w, cu, d_out, state, d_state = _packed(d)

    def call(sl, seqs, bounds):
        dev, host = _cu(bounds)
        return kla_bwd(w.q[:, sl].to(DEV), w.k[:, sl].to(DEV), w.v[:, sl].to(DEV), w.log_alpha[:, sl].to(DEV), w.eta[:, sl].to(DEV), w.eps,
                       d_out[:, sl].to(DEV), init_state=state[seqs].to(DEV), d_final_state=d_state[seqs].to(DEV), cu_seqlens=dev, host_seqlens=host)

    g = call(slice(0, int(cu[-1])), list(range(len(LENS))), cu)
    for n in CLEAN:
        sl = slice(int(cu[n]), int(cu[n + 1]))
        alone = call(sl, [n], [0, LENS[n]])
        ref = oracle.backward(np64(w.q[:, sl]), np64(w.k[:, sl]), np64(w.v[:, sl]), np64(w.log_alpha[:, sl]), np64(w.eta[:, sl]), w.eps,
                              np64(d_out[:, sl]), np64(state[n:n + 1]), np64(d_state[n:n + 1]))
        for name in GRADS:
            assert torch.equal(g[name][:, sl], alone[name]), (n, name)
            assert rel_err(np64(alone[name]), ref[name]) <= TOL_BF16, (n, name)
        assert torch.equal(g["dinit_state"][n], alone["dinit_state"][0]), n
        assert rel_err(np64(alone["dinit_state"]), ref["dinit"]) <= TOL_BF16, n
    assert torch.equal(g["dinit_state"][5].cpu(), d_state[5])   # an empty sequence hands the gradient through


@pytest.mark.parametrize("out_dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("d", [64, 128])
def test_forward_of_a_sequence_knows_nothing_of_its_neighbours(d, out_dtype):
    w, cu, _, state, _ = _packed(d)

    def call(sl, seqs, bounds):
        dev, host = _cu(bounds)
        return kla_chunk_fwd(w.q[:, sl].to(DEV), w.k[:, sl].to(DEV), w.v[:, sl].to(DEV), w.log_alpha[:, sl].to(DEV), w.eta[:, sl].to(DEV), w.eps,
                             init_state=state[seqs].to(DEV), cu_seqlens=dev, host_seqlens=host, out_dtype=out_dtype)

    out, fin = call(slice(0, int(cu[-1])), list(range(len(LENS))), cu)
    for n in CLEAN:
        sl = slice(int(cu[n]), int(cu[n + 1]))
        o, f = call(sl, [n], [0, LENS[n]])
        assert torch.equal(out[:, sl], o) and torch.equal(fin[n], f[0]), n
        ro, rf, _ = oracle.forward(np64(w.q[:, sl]), np64(w.k[:, sl]), np64(w.v[:, sl]), np64(w.log_alpha[:, sl]), np64(w.eta[:, sl]), w.eps, np64(state[n:n + 1]))
        assert rel_err(np64(f), rf) <= TOL_BF16, n
        if out_dtype == torch.float32:
            assert rel_err(np64(o), ro) <= TOL_BF16, n
    assert torch.equal(fin[5].cpu(), state[5])
