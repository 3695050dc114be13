"""Bounded waits of the backward pass, the span map and the forward on static scratch: a wait made to run out (a copy or a
signal that never comes; nothing faults or hangs) is heard of by a caller who passes a status word and by one who does not, and the context stays usable."""
import numpy as np
import pytest
import torch

import oracle
from helpers import TOL_BF16, np64, rel_err
from paper_2605_08587_b200 import (KLA_FLAG_WY_FORM, KlaError, binding, check, kla_bwd, kla_chunk_fwd, kla_chunk_fwd_static_scratch,
                                   kla_chunk_span_map, workloads as W)

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
RUN_OUT = binding.KLA_INTERNAL_FLAG_TEST_TIMEOUT
TIMEOUT = -10   # KLA_ERR_TIMEOUT


def _args(w):
    return [t.to(DEV) for t in (w.q, w.k, w.v, w.log_alpha, w.eta)]


@pytest.mark.parametrize("packed", [False, True])
@pytest.mark.parametrize("d", [64, 128])
def test_backward_reports_a_wait_that_ran_out(d, packed):
    w = W.config2(B=1, H=2, T=200, d=d, seed=510 + d)
    do, df = W.upstream_grads(w)
    cu = torch.tensor([0, 70, 70, 200], dtype=torch.int32) if packed else None
    kw = dict(cu_seqlens=cu.to(DEV), host_seqlens=cu) if packed else dict(d_final_state=df.to(DEV))
    a = _args(w)

    def call(**more):
        return kla_bwd(*a, w.eps, do.to(DEV), **kw, **more)

    def right(g):
        if packed:
            ref = oracle.backward_packed(*(np64(x)[0] for x in (w.q, w.k, w.v, w.log_alpha, w.eta)), w.eps, cu.numpy(), np64(do)[0])
        else:
            ref = oracle.backward(*(np64(x) for x in (w.q, w.k, w.v, w.log_alpha, w.eta)), w.eps, np64(do), None, np64(df))
        for name in ("dq", "dk", "dv", "dlog_alpha", "deta"):
            assert rel_err(np64(g[name]), np.reshape(ref[name], g[name].shape)) <= TOL_BF16, name

    word = torch.zeros(1, dtype=torch.int32, device=DEV)
    check(DEV)
    call(flags=RUN_OUT, status_word=word)
    assert int(word.item()) == TIMEOUT
    check(DEV)                                  # the caller's own word was given: nothing in the binding's
    word.zero_()
    right(call(status_word=word))               # the same context, the ordinary path
    assert int(word.item()) == 0
    call(flags=RUN_OUT)
    with pytest.raises(KlaError) as e:
        check(DEV)
    assert e.value.code == TIMEOUT
    check(DEV)                                  # cleared
    right(call())
    check(DEV)


@pytest.mark.parametrize("flags", [0, KLA_FLAG_WY_FORM])
def test_span_map_reports_a_wait_that_ran_out(flags):
    w = W.config2(B=1, H=2, T=200, seed=530)
    a = _args(w)[1:]
    word = torch.zeros(1, dtype=torch.int32, device=DEV)
    kla_chunk_span_map(*a, w.eps, flags=flags | RUN_OUT, status_word=word)
    assert int(word.item()) == TIMEOUT
    kla_chunk_span_map(*a, w.eps, flags=flags | RUN_OUT)
    with pytest.raises(KlaError) as e:
        check(DEV)
    assert e.value.code == TIMEOUT
    word.zero_()
    phi, n = kla_chunk_span_map(*a, w.eps, flags=flags, status_word=word)
    assert int(word.item()) == 0
    check(DEV)
    zero = torch.zeros(1, 2, 128, 128, dtype=torch.float64)
    _, fin, _ = oracle.forward(*(np64(x) for x in (w.q, w.k, w.v, w.log_alpha, w.eta)), w.eps, zero.numpy())
    assert rel_err(np64(n), fin) <= TOL_BF16


def test_static_scratch_reports_a_wait_that_ran_out():
    w = W.config2(B=1, H=2, T=130, seed=535)
    a = _args(w)
    want, _ = kla_chunk_fwd(*a, w.eps)
    out = torch.empty_like(want)
    check(DEV)
    kla_chunk_fwd_static_scratch(*a, w.eps, out, flags=RUN_OUT)
    with pytest.raises(KlaError) as e:
        check(DEV)
    assert e.value.code == TIMEOUT
    kla_chunk_fwd_static_scratch(*a, w.eps, out)
    check(DEV)
    assert torch.equal(out, want)


def test_replaying_a_graph_does_not_clear_what_other_calls_reported(monkeypatch):
    """The first call of all may be a captured one: the binding's status word must not become part of that graph."""
    w = W.config2(B=1, H=2, T=130, seed=540)
    do, _ = W.upstream_grads(w)
    a, do = _args(w), do.to(DEV)
    kla_bwd(*a, w.eps, do)                      # (what is loaded on first use is loaded)
    kla_chunk_fwd(*a, w.eps)
    eager = kla_bwd(*a, w.eps, do)
    torch.cuda.synchronize()
    monkeypatch.setattr(binding, "_own_status", {})
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g = kla_bwd(*a, w.eps, do)
        out, fin = kla_chunk_fwd(*a, w.eps)
    check(DEV)                                  # captured, not run: nothing to report
    kla_bwd(*a, w.eps, do, flags=RUN_OUT)
    graph.replay()
    torch.cuda.synchronize()
    with pytest.raises(KlaError) as e:
        check(DEV)
    assert e.value.code == TIMEOUT
    assert all(torch.equal(g[x], eager[x]) for x in g if g[x] is not None)
    graph.replay()
    check(DEV)
