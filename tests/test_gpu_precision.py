"""How exact the tensor-core kernels are: 2-norm errors against the fp64 oracle, held to what their operands' roundings add up to.

PAIR is the rounding of an operand carried as a pair of bf16 values hi + lo, relative to its norm: what the rounding to hi leaves is
uniform within half a unit of hi, so lo, rounded in its turn, is off by 2^-15 / sqrt(84) of the operand's binade in the mean
square, 1 / 1.53 of that relative to values spread over a binade.  The lo lo term that a three-term product drops is as large.
Errors of that kind are independent and add in quadrature."""
import numpy as np
import pytest
import torch

from helpers import gpu_chunk, np64, oracle_chunk
from paper_2605_08587_b200 import workloads as W

pytestmark = pytest.mark.gpu
PAIR = 2.2e-6


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
