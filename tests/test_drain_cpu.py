"""How a 2-SM GEMM that gave up lets its copies land (csrc/drain.h, compiled here with the host compiler): a
stage's full barrier as the hardware counts it (one arrival that expects both CTAs' bytes, bytes that land
in any order, also before it), producers that stopped after any two stage counts. With what drain_step
supplies every barrier completes, and none before the last byte in flight has landed."""
import ctypes
import itertools
import pathlib
import shutil
import subprocess

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2606_28516_gb300" / "csrc"
SRC = """
#include "drain.h"
extern "C" int step(unsigned k, unsigned n0, unsigned n1) {
    const cm::DrainStep d = cm::drain_step(k, n0, n1);
    return (d.arrive ? 1 : 0) | (d.complete ? 2 : 0);
}
"""


@pytest.fixture(scope="module")
def step(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    t = tmp_path_factory.mktemp("drain")
    (t / "drain.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-I", str(CSRC), "-o", str(t / "drain.so"),
                    str(t / "drain.cpp")], check=True)
    f = ctypes.CDLL(str(t / "drain.so")).step
    f.argtypes = [ctypes.c_uint] * 3
    return f


BYTES = 28672  # one CTA's boxes of a stage


class Barrier:
    """One phase: complete when no arrival is pending and no byte is outstanding."""

    def __init__(self):
        self.pending, self.tx, self.done = 1, 0, False

    def _check(self):
        self.done = self.done or (self.pending == 0 and self.tx == 0)

    def arrive_expect(self, n):
        self.tx += n
        self.pending -= 1
        self._check()

    def land(self, n):
        self.tx -= n
        self._check()


@pytest.mark.parametrize("n0,n1", list(itertools.product(range(4), range(4))))
def test_every_issued_stage_completes_with_its_bytes(step, n0, n1):
    for k in range(max(n0, n1)):
        even, odd = k < n0, k < n1
        bits = step(k, n0, n1)
        events = (["expect"] if even else []) + ["land"] * (even + odd) + ["drain"]
        for order in set(itertools.permutations(events)):
            b, left = Barrier(), even + odd
            for ev in order:
                if ev == "expect":
                    b.arrive_expect(2 * BYTES)
                elif ev == "land":
                    b.land(BYTES)
                    left -= 1
                else:
                    if bits & 1:
                        b.arrive_expect(BYTES)
                    if bits & 2:
                        b.land(BYTES)
                # the producers' and the drain's parts are all in before the drain waits
                if b.done:
                    assert left == 0, (order, k, n0, n1)
            assert b.done, (order, k, n0, n1)


def test_stages_both_or_neither_reached_need_nothing(step):
    assert step(0, 3, 3) == 0 and step(2, 3, 3) == 0 and step(3, 3, 3) == 0
