"""The bf16 layer's fc1 evaluates GELU(u) = max(u, 0) - |u| / 2 2^q(|u|), q the degree-6 polynomial of
csrc/common.cuh (GeluE), on v = max(-|u|, -6) with the factor 1/2 in the exponent. On the CPU, in
float32 with the kernel's order (each fma rounded once from a float64 value) and 2^q rounded once, then
off by the exponential instruction's bound (2^-22.5): against the float64 exact-erf GELU the largest
error stays below 3.5e-7 for every u, and over the pre-activations fc1 sees the mean square error is
below that of the Abramowitz & Stegun 7.1.28 form (tests/test_gelu_approx.py has it, and shows that
such errors move a negligible share of the bf16 hidden state's roundings). The coefficients are read
from the source."""
import pathlib
import re

import numpy as np
from scipy.special import ndtr

from test_gelu_approx import gelu_as_f32

SRC = (pathlib.Path(__file__).resolve().parent.parent / "paper_2606_28516_gb300" / "csrc" / "common.cuh").read_text()
BODY = SRC[SRC.index("struct GeluE"):SRC.index("};", SRC.index("struct GeluE"))]
C = [np.float32(re.search(rf"\bC{k} = ([-0-9.e]+)f", BODY).group(1)) for k in range(1, 7)]


def _fma(a, b, c):
    return (a.astype(np.float64) * b.astype(np.float64) + np.asarray(c, np.float64)).astype(np.float32)


def gelu_e(u, off=0.0):
    u = np.asarray(u, np.float32)
    v = np.maximum(-np.abs(u), np.float32(-6))
    q = np.full_like(v, C[5])
    for k in range(4, -1, -1):
        q = _fma(q, v, C[k])
    q = _fma(q, v, np.float32(-1))
    e = (np.exp2(q.astype(np.float64)) * (1 + off)).astype(np.float32)
    return _fma(v, e, np.maximum(u, np.float32(0)))


def exact(u):
    u = np.asarray(u, np.float64)
    return u * ndtr(u)


def test_largest_error():
    u = np.concatenate([np.linspace(-7, 7, 1_000_001), np.linspace(-60, 60, 400_001)]).astype(np.float32)
    for off in (0.0, 2.0 ** -22.5, -(2.0 ** -22.5)):
        err = np.abs(gelu_e(u, off) - exact(u))
        assert (err <= np.maximum(3.5e-7, np.abs(u.astype(np.float64)) * 2.0 ** -24)).all()


def test_mean_square_error_below_the_rational_form():
    rng = np.random.default_rng(0)
    for s in (0.28, 0.39, 0.55, 0.64, 1.0, 2.0):  # 0.02 sqrt(d) for d = 192 .. 1,024, and wider
        u = (s * rng.standard_normal(300_000)).astype(np.float32)
        old = np.mean((gelu_as_f32(u) - exact(u)) ** 2)
        assert np.mean((gelu_e(u) - exact(u)) ** 2) <= old, s


def test_specials():
    r = gelu_e(np.float32([np.nan, 0.0, 1e30, -1e30]))
    assert np.isnan(r[0]) and r[1] == 0 and r[2] == np.float32(1e30) and abs(r[3]) < 1e-8
