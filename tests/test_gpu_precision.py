"""How exact the tensor-core kernels are: 2-norm errors against the fp64 oracle, held to what their operands' roundings add up to.

PAIR is the rounding of an operand carried as a pair of bf16 values hi + lo, relative to its norm: what the rounding to hi leaves is
uniform within half a unit of hi, so lo, rounded in its turn, is off by 2^-15 / sqrt(84) of the operand's binade in the mean
square, 1 / 1.53 of that relative to values spread over a binade.  The lo lo term that a three-term product drops is as large.
Errors of that kind are independent and add in quadrature."""
import numpy as np
import pytest
import torch

import oracle
from helpers import gpu_chunk, np64, oracle_chunk
from paper_2605_08587_b200 import kla_bwd, kla_chunk_fwd, kla_dg_fwd, workloads as W

pytestmark = pytest.mark.gpu
PAIR = 2.2e-6
SUM = 8 * 0.4 * 0.72 * 2.0 ** -23 / 2


def _norm_err(got, ref):
    return float(np.linalg.norm(np64(got) - ref) / np.linalg.norm(ref))


def _workload(kind):
    if kind == "packed":   # heavy-tailed keys, some of them near zero
        return W.config5(H=4, lengths=[700, 64, 1, 1500, 333], seed=1404)
    B, H, d = dict(d64=(2, 4, 64), d64_two_blocks=(20, 16, 64), d128=(2, 4, 128))[kind]
    return W.config3(B=B, H=H, T=777 if B == 2 else 200, d=d, seed=1400 + d)


@pytest.mark.parametrize("kind", ["d64", "d64_two_blocks", "d128", "packed"])
def test_forward(kind):
    """Output: the pairs of S, P and U and one dropped term, each at most at the output's own size.  Final state: the pair of U, and what
    reaches U from the solve, where only products with off-diagonal blocks are rounded (less than U itself together).  15 % for the
    sample."""
    w = _workload(kind)
    out, fin = gpu_chunk(w, out_dtype=torch.float32)
    ro, rf = oracle_chunk(w)[:2]
    assert _norm_err(out.reshape(ro.shape), ro) <= 1.15 * 4 ** 0.5 * PAIR
    assert _norm_err(fin, rf) <= 1.15 * 1.5 ** 0.5 * PAIR


@pytest.mark.parametrize("d", [64, 128])
def test_forward_that_forgets_little(d):
    """No decay and small steps: what a chunk adds is a small part of the state, so anything lost from the whole state at every chunk
    would add up over the 64 chunks.  Same bounds as above: the pairs are roundings of the parts added, not of the sum."""
    w = W.config3(B=1, H=2, T=4096, d=d, seed=1410 + d)
    w.log_alpha = torch.zeros_like(w.log_alpha)
    w.eta = w.eta * 1e-3
    out, fin = gpu_chunk(w, out_dtype=torch.float32)
    ro, rf = oracle_chunk(w)[:2]
    assert _norm_err(out, ro) <= 1.15 * 4 ** 0.5 * PAIR
    assert _norm_err(fin, rf) <= 1.15 * 1.5 ** 0.5 * PAIR


def _backward_errors(w, seed):
    H, d = w.q.shape[2:]
    w.init_state = (0.02 * torch.randn(w.n_seq, H, d, d, generator=torch.Generator().manual_seed(seed))).float()
    do, df = W.upstream_grads(w)
    dev = "cuda:0"
    cu = w.cu_seqlens
    g = kla_bwd(*[x.to(dev) for x in (w.q, w.k, w.v, w.log_alpha, w.eta)], w.eps, do.to(dev), init_state=w.init_state.to(dev),
                d_final_state=df.to(dev), cu_seqlens=None if cu is None else cu.to(dev), host_seqlens=cu)
    ins = [np64(x) for x in (w.q, w.k, w.v, w.log_alpha, w.eta)]
    if cu is None:
        r = oracle.backward(*ins, w.eps, np64(do), np64(w.init_state), np64(df))
    else:
        r = oracle.backward_packed(*[x[0] for x in ins], w.eps, cu.numpy(), np64(do)[0], np64(w.init_state), np64(df))
    r["dinit_state"] = r["dinit"]
    return {n: _norm_err(g[n].reshape(r[n].shape), r[n]) for n in ("dq", "dk", "dv", "dlog_alpha", "deta", "dinit_state")}


def _check_backward(w, seed, times=1.0):
    for name, err in _backward_errors(w, seed).items():
        # five products in succession (P^T dO or K S_0, U or w, E or F, and two of the gradient) in quadrature; dlog_alpha is a sum of
        # differences of such gradients, twice the size of what is left
        bound = times * 5 ** 0.5 * SUM * (2.0 if name == "dlog_alpha" else 1.0)
        assert err <= bound, "%s: %.2e > %.2e" % (name, err, bound)


@pytest.mark.parametrize("kind", ["d64", "d128", "packed"])
def test_backward(kind):
    _check_backward(_workload(kind), 1420)


@pytest.mark.parametrize("d", [64, 128])
def test_backward_that_forgets_little(d):
    """As for the forward.  What each of 64 chunks adds has such an error of its own; they are of both signs, and a state keeps what
    d / eta tokens, here all of them, have added: twice the bound for the states' part."""
    w = W.config2(B=1, H=2, T=4096, d=d, seed=1430 + d)
    w.log_alpha = torch.zeros_like(w.log_alpha)
    w.eta = w.eta * 1e-3
    _check_backward(w, 1431, times=2.0)


@pytest.mark.parametrize("diag", [False, True])
@pytest.mark.parametrize("d", [64, 128])
def test_recurrence_with_weak_decay(d, diag):
    """fp32 scan, log alpha / 100, eta / 10.  The state is rounded five times in four tokens, each time by a uniform error within half
    a unit in the last place, a unit being 0.72 * 2^-23 of a value in the mean, independently; what it remembers, and the errors with it, decays over
    half of d / eta < 4 000 tokens for errors added in quadrature.  An error in the decay, one for the whole state, would add up."""
    steps = 5 * 4000 / 2 / 4
    bound = steps ** 0.5 * 2.0 ** -24 * 0.72 / 3 ** 0.5
    if diag:
        w = W.config_dg(B=1, H=2, T=4096, d=d, seed=1440 + d, dtype=torch.float32)
    else:
        w = W.config2(B=1, H=2, T=4096, d=d, seed=1440 + d)
        w.q, w.k, w.v = w.q.float(), w.k.float(), w.v.float()
    w.log_alpha, w.eta = w.log_alpha * 1e-2, w.eta * 0.1
    a = [x.to("cuda:0") for x in (w.q, w.k, w.v, w.log_alpha, w.eta)]
    s0 = None if w.init_state is None else w.init_state.to("cuda:0")
    out, fin = (kla_dg_fwd if diag else kla_chunk_fwd)(*a, w.eps, init_state=s0, out_dtype=torch.float32)
    ro, rf, _ = oracle.forward(*[np64(x) for x in (w.q, w.k, w.v, w.log_alpha, w.eta)], w.eps, None if s0 is None else np64(s0), diagonal_gates=diag)
    assert _norm_err(out, ro) <= bound
    assert _norm_err(fin, rf) <= bound


@pytest.mark.parametrize("diag", [False, True])
def test_recurrence_with_decays_on_both_sides_of_one_half(diag):
    """Decays of a block of four tokens from 1 down to 0, no writes: the state keeps the product of them."""
    B, T, H, d = 1, 64, 2, 64
    g = torch.Generator().manual_seed(1450)
    q, k, v = (torch.randn(B, T, H, d, generator=g) for _ in range(3))
    la = -torch.logspace(-6, 0.5, T).reshape(1, T, 1).expand(B, T, H).contiguous() * torch.tensor([1.0, 30.0])   # head 1: down to nothing
    la[:, 0] = 0.0
    s0 = torch.randn(B, H, d, d, generator=g)
    eta = torch.zeros(B, T, H)
    if diag:
        la = (la.unsqueeze(-1) * torch.linspace(0.0, 2.0, d)).contiguous()
    a = [x.to("cuda:0") for x in (q, k, v, la, eta)]
    _, fin = (kla_dg_fwd if diag else kla_chunk_fwd)(*a, 1e-6, init_state=s0.to("cuda:0"), out_dtype=torch.float32)
    ref = s0.double() * torch.exp(la.double().sum(1)).reshape(B, H, d if diag else 1, 1)
    err = ((fin.cpu().double() - ref).abs() / ref.abs().clamp_min(1e-30)).max()
    # 16 blocks: a rounding of the state each, and a decay that is a product of four expf (2 ulp each) where it is below one half
    assert float(err) <= 16 * (1 + 4 * 3) * 2.0 ** -24
