"""The four-token scan (fp32 chunk forward, diagonal gates) and several decode steps in one call, at the sizes where their
branches meet: lengths around the 4-token blocks and the 16-token stages, few and many (sequence, head) pairs (8 or 16 state
columns per warp), against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL_F32, np64, rel_err
from paper_2605_08587_b200 import kla_chunk_fwd, kla_decode_step, kla_decode_steps, kla_dg_decode_step, kla_dg_fwd, workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("diag", [False, True])
@pytest.mark.parametrize("B,H,d", [(1, 1, 64), (3, 16, 64), (5, 16, 64), (1, 2, 128), (3, 16, 128)])
@pytest.mark.parametrize("T", [1, 3, 4, 5, 15, 16, 17, 33, 70])
def test_lengths_and_unit_counts(T, B, H, d, diag):
    w = W.config_dg(B=B, H=H, T=T, d=d, seed=1000 + T + H, dtype=torch.float32)
    if not diag:
        w.log_alpha = w.log_alpha[..., 0].contiguous()
    fwd = kla_dg_fwd if diag else kla_chunk_fwd
    out, fin = fwd(w.q.to(DEV), w.k.to(DEV), w.v.to(DEV), w.log_alpha.to(DEV), w.eta.to(DEV), w.eps, init_state=w.init_state.to(DEV))
    ro, rf = oracle.forward(np64(w.q), np64(w.k), np64(w.v), np64(w.log_alpha), np64(w.eta), w.eps, np64(w.init_state), diagonal_gates=diag)[:2]
    assert rel_err(np64(out), ro) <= TOL_F32
    assert rel_err(np64(fin), rf) <= TOL_F32


def test_decay_to_nothing_inside_a_block():
    w = W.config_dg(B=2, H=2, T=40, d=64, seed=1100, dtype=torch.float32)
    w.log_alpha = (w.log_alpha * torch.where(torch.rand(w.log_alpha.shape, generator=torch.Generator().manual_seed(1)) < 0.3, 2000.0, 1.0)).contiguous()
    out, fin = kla_dg_fwd(w.q.to(DEV), w.k.to(DEV), w.v.to(DEV), w.log_alpha.to(DEV), w.eta.to(DEV), w.eps, init_state=w.init_state.to(DEV))
    ro, rf = oracle.forward(np64(w.q), np64(w.k), np64(w.v), np64(w.log_alpha), np64(w.eta), w.eps, np64(w.init_state), diagonal_gates=True)[:2]
    assert rel_err(np64(out), ro) <= TOL_F32
    assert rel_err(np64(fin), rf) <= TOL_F32


@pytest.mark.parametrize("B,H,d,n", [(1, 4, 64, 2), (2, 2, 128, 5), (37, 4, 128, 3)])
def test_steps_in_one_call_equal_single_steps(B, H, d, n):
    w = W.config4(B=B, H=H, d=d, steps=n, seed=1200 + n)
    a, b = w.state.to(DEV).clone(), w.state.to(DEV).clone()
    x = [t.to(DEV) for t in (w.q, w.k, w.v, w.log_alpha, w.eta)]
    o = kla_decode_steps(*x, w.eps, a)
    for s in range(n):
        assert torch.equal(o[s], kla_decode_step(*[t[s].contiguous() for t in x], w.eps, b))
    assert torch.equal(a, b)


@pytest.mark.parametrize("B,H,d", [(1, 1, 64), (5, 3, 128), (64, 8, 128)])
def test_diagonal_decode_step(B, H, d):
    w = W.config_dg(B=B, H=H, T=1, d=d, seed=1300 + B, dtype=torch.float32)
    st = w.init_state.to(DEV).clone()
    o = kla_dg_decode_step(*[t[:, 0].contiguous().to(DEV) for t in (w.q, w.k, w.v, w.log_alpha, w.eta)], w.eps, st)
    ro, rf = oracle.forward(np64(w.q), np64(w.k), np64(w.v), np64(w.log_alpha), np64(w.eta), w.eps, np64(w.init_state), diagonal_gates=True)[:2]
    assert rel_err(np64(o), ro[:, 0]) <= TOL_F32
    assert rel_err(np64(st), rf) <= TOL_F32
