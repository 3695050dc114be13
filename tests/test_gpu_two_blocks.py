"""Head dimension 64 with more blocks than SMs: the chunk kernel's form with two blocks on an SM (two chunk slots)."""
import pytest
import torch

import oracle
from helpers import TOL_BF16, assert_bf16_out_close, gpu_chunk, np64, oracle_chunk, rel_err
from paper_2605_08587_b200 import KLA_FLAG_COEFF_ETA, KLA_FLAG_QNORM, workloads as W

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


@pytest.mark.parametrize("out_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("variant", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("B", [2, 20])   # 32 blocks: one on an SM; 320: two
def test_layer_edge_variants(B, variant, out_dtype):
    coeff_eta, qnorm = variant
    w = W.config3(B=B, H=16, T=200, d=64, seed=1310 + 2 * coeff_eta + qnorm)   # three chunks and a ragged one: every slot is used again
    if coeff_eta:   # beta = eta is a contraction only on unit keys
        k = w.k.float()
        w.k = (k / k.norm(dim=-1, keepdim=True)).to(w.k.dtype)
    out, fin = gpu_chunk(w, out_dtype=out_dtype, flags=(KLA_FLAG_COEFF_ETA if coeff_eta else 0) | (KLA_FLAG_QNORM if qnorm else 0))
    with oracle.variant(coeff_eta=coeff_eta, qnorm=qnorm):
        ro, rf = oracle_chunk(w)[:2]
    if out_dtype == torch.bfloat16:
        assert_bf16_out_close(out, ro)
    else:
        assert rel_err(np64(out), ro) <= TOL_BF16
    assert rel_err(np64(fin), rf) <= TOL_BF16
