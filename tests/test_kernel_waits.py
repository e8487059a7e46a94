"""Rules that the kernels' waits keep, checked on the sources (a hardware run cannot show that one is broken,
and must not try): by the PTX memory model a tcgen05 operation is ordered after a barrier wait only by
tcgen05.fence::after_thread_sync, so that every access to tensor memory (MMA, load, store) follows the last
barrier wait before it with such a fence in between."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2606_28516_gb300" / "csrc"
FILES = ("route.cu", "tc_gemm.cu", "tc_gemm2.cu")


def _source(name):
    """The file without its comments and macro or wrapper definitions above the first kernel."""
    s = (CSRC / name).read_text()
    s = re.sub(r"//[^\n]*", lambda m: " " * len(m.group()), s)
    return s[s.index("__global__ void"):]


@pytest.mark.parametrize("name", FILES)
def test_tensor_memory_accesses_follow_a_fence(name):
    s = _source(name)
    # fr_bar, kjoin_bar and kdone_bar hand over counts and partial sums in shared or global memory
    waits = [m.start() for m in re.finditer(r"\bmbar_wait(_warp)?\((?!fr_bar|kjoin_bar|kdone_bar)", s)]
    uses = [m for m in re.finditer(r"\b(CM_TMEM_(LD|ST)_X\d+|umma2?_(bf16|tf32_ts|tf32))\(", s)]
    assert uses
    for m in uses:
        last = max((w for w in waits if w < m.start()), default=None)
        assert last is not None, m.group()
        line = s[:m.start()].count("\n")
        assert "tc_fence_after();" in s[last:m.start()], f"{name}, line {line} of the kernels: {m.group()}"
