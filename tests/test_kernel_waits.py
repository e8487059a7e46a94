"""Rules that the kernels' waits keep, checked on the sources (a hardware run cannot show that one is broken,
and must not try): by the PTX memory model a tcgen05 operation is ordered after a barrier wait only by
tcgen05.fence::after_thread_sync, so that every access to tensor memory (MMA, load, store) follows the last
barrier wait before it with such a fence in between; and a bounded wait may run out for single lanes of a
warp, so that a warp takes its outcome together (mbar_wait_warp): what follows is collective over the warp."""
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


@pytest.mark.parametrize("name", FILES)
def test_warps_agree_on_a_wait_that_ran_out(name):
    s = _source(name)
    single = re.findall(r"\bmbar_wait\((\w+)", s)
    # the K split's counter: lane 0 of warp 0 alone
    assert [b for b in single if b != "kjoin_bar"] == []
    for m in re.finditer(r"\bmbar_wait\(kjoin_bar", s):
        assert "if (warp == 0 && lane == 0) {" in s[m.start() - 200:m.start()]


@pytest.mark.parametrize("name", ("route.cu", "tc_gemm.cu"))
def test_producers_wait_for_their_last_copies_whoever_gave_up(name):
    # the issuer can give up on a copy in flight after its producer has issued the last one without a wait that
    # ran out, so that the producer's own outcome does not decide whether copies are in flight
    s = _source(name)
    assert not re.search(r"if \(!ok[^)]*\)\s*\{?\s*for \(", s)
    assert "lim + 10000000ull" in s
