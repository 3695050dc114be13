"""Head dimension 64 with more blocks than SMs: the chunk kernel's form with two blocks on an SM (two chunk slots)."""
import pytest
import torch

from helpers import TOL_BF16, gpu_chunk, np64, oracle_chunk, rel_err
from paper_2605_08587_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 63, 64, 65, 128, 129, 200, 1000])   # one chunk, both slots, the first reuse of a slot, many
def test_two_blocks_per_sm_match_the_oracle(T):
    w = W.config3(B=20, H=16, T=T, d=64, seed=1200 + T)   # 320 blocks
    out, fin = gpu_chunk(w, out_dtype=torch.float32)
    ro, rf = oracle_chunk(w)[:2]
    assert rel_err(np64(out), ro) <= TOL_BF16
    assert rel_err(np64(fin), rf) <= TOL_BF16


def test_both_forms_agree_bit_for_bit():
    # the same sequences in a launch of 64 blocks (one on an SM) and of 320 (two)
    w = W.config3(B=20, H=16, T=333, d=64, seed=1300)
    out, fin = gpu_chunk(w, out_dtype=torch.float32)
    import copy
    part = copy.copy(w)
    part.B = 4
    for name in ("q", "k", "v", "log_alpha", "eta", "init_state"):
        setattr(part, name, getattr(w, name)[:4].contiguous())
    o, f = gpu_chunk(part, out_dtype=torch.float32)
    assert torch.equal(out[:4], o) and torch.equal(fin[:4], f)
