"""Many more blocks than SMs, each for a chunk or two: a block gets the tensor memory that the block before it on the SM has only
just given back, so a store of that one still in flight would land in its operands."""
import pytest
import torch

from helpers import TOL_BF16, gpu_chunk, np64, oracle_chunk, rel_err
from paper_2605_08587_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 64, 65])   # one row, a whole chunk, a second chunk of one row
@pytest.mark.parametrize("d", [64, 128])     # two blocks on an SM at a time, one; twelve for each SM in all
def test_blocks_that_follow_each_other_on_an_sm(d, T):
    w = W.config2(B=148 * 6 * 64 // d, H=2, T=T, d=d, seed=820 + T)
    first = gpu_chunk(w)
    again = gpu_chunk(w)
    assert torch.equal(first[0], again[0]) and torch.equal(first[1], again[1])
    seqs = list(range(0, w.q.shape[0], 7))
    ro, rf = oracle_chunk(w, seqs=seqs)
    assert rel_err(np64(first[0])[seqs], ro) <= TOL_BF16
    assert rel_err(np64(first[1])[seqs], rf) <= TOL_BF16
