"""The rule for the expert GEMM's tile width (tc2_grouped_bn, a host function of the library): the narrowest
width while one round of 76 SM pairs holds its tiles and the basis kernel's, counted only where that kernel runs
beside the expert GEMM, which is where the expert GEMM starts early (pdl_wait_role 2)."""
import ctypes
import pathlib
import re

import pytest

from paper_2606_28516_gb300 import clearmoe as cm

API = (pathlib.Path(__file__).resolve().parent.parent / "paper_2606_28516_gb300" / "csrc" / "api.cu").read_text()


@pytest.fixture(scope="module")
def width():
    import __graft_entry__
    __graft_entry__.build()
    f = getattr(cm.lib(), "_ZN2cm14tc2_grouped_bnEliili")
    f.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_int]
    return lambda T, d, G, basis: f(T, d, G, basis, 152)


def test_widths(width):
    # 16 blocks of 256 tokens, d = 768: 96 tiles of 128, 64 of 192, 48 of 256 columns
    assert width(4000, 768, 1, 0) == 192
    assert width(4000, 768, 1, 16) == 256  # 64 + 16 exceed a round
    assert width(788, 768, 1, 0) == 128 and width(788, 768, 1, 4) == 128
    assert width(25216, 768, 1, 0) == 256


def test_basis_pairs_are_counted_only_beside_the_basis():
    bodies = re.split(r"\n(?=\w[^\n]*\([^;]*?\) \{\n)", API)
    seen = 0
    for body in bodies:
        for m in re.finditer(r"tc2_grouped_bn\(([^;]*?), L->num_sms\)", body):
            seen += 1
            depth, parts = 0, [""]
            for ch in m.group(1):
                depth += (ch == "(") - (ch == ")")
                if ch == "," and depth == 0:
                    parts.append("")
                else:
                    parts[-1] += ch
            assert len(parts) == 4
            if parts[3].strip() != "0":
                assert "pdl_wait_role = 2" in body, parts
    assert seen >= 3
