"""Rules of the kernels' source that no run can show: a block that breaks them still gives the right result nearly always."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_08587_b200", "csrc")


def _code(name):
    """Source without comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def _block(text, start):
    """(the text inside the first pair of braces from `start` on, the position after it)."""
    a = text.index("{", start)
    depth = 0
    for i in range(a, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[a + 1:i], i + 1
    raise AssertionError("unbalanced braces")


def test_stores_to_tensor_memory_complete_before_it_is_given_back():
    """Every way out of the chain's loop over chunks (its end, a wait that gave up) passes a wait for the stores."""
    text = _code("chunk_mma.cu")
    at = text.index("__device__ void chain(")
    body, _ = _block(text, at)
    loop = body.index("for (int c = 0; c < nchunks; ++c)")
    inside, after = _block(body, loop)
    assert "return" not in inside                     # it is left by break alone
    rest = body[after:]
    assert "tmem_wait_stores();" in rest
    before_wait = rest[:rest.index("tmem_wait_stores();")]
    assert before_wait.strip() == "", before_wait     # nothing that could skip it
    # and no other kernel stores to tensor memory without this test knowing of it
    others = [f for f in sorted(os.listdir(CSRC)) if f != "chunk_mma.cu" and "tcgen05.st." in _code(f)]
    assert others == []


def test_tiles_that_tma_permutes_start_where_the_permutation_does():
    """TMA's 128-byte swizzle is a function of the shared address, the kernels' sw128() of the place in the tile: every kernel that
    fetches tiles either checks that its shared memory starts on a 1024-byte boundary, and reports it, or rounds up to one."""
    kernels = 0
    for name in sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")):
        text = _code(name)
        # kernels that are given tensor maps (they alone can fetch by them)
        for m in re.finditer(r"__global__[^;{]*?\b(kla_\w+)\(([^{;]*?)\)\s*\{", text, flags=re.S):
            if not re.search(r"CUtensorMap|TileMaps", m.group(2)):
                continue
            kernels += 1
            body, _ = _block(text, m.end() - 1)
            before = re.split(r"tma_load_2d|\bchain<|find_work", body)[0]
            checked = re.search(r"if \(smem_u32\(smem_dyn\) & 1023\) \{[^}]*KLA_ERR_ALIGN[^}]*return;", before, flags=re.S)
            rounded = re.search(r"\(reinterpret_cast<uintptr_t>\(smem_dyn\) \+ 1023\) & ~\(uintptr_t\)1023", before)
            assert checked or rounded, m.group(1)
    assert kernels == 3
