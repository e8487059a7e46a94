"""The fp32 layer's tensor-core fc1 evaluates GELU(u) = max(u, 0) - |u| / 2 2^q(|u|), q the degree-10
polynomial of csrc/common.cuh (GeluQ). On the CPU, in float32 with the kernel's order (each fma rounded
once from a float64 value) and 2^q rounded once: against the float64 exact-erf GELU the largest error
stays below 2.5e-7 for every u (half a step of float32 at 4 is 2.4e-7), and over the pre-activations
fc1 sees the mean square error is below that of u (1 + erf(u / sqrt 2)) / 2 in float32 with a correctly
rounded erf, the form it takes the place of. The coefficients are read from the source."""
import pathlib
import re

import numpy as np
from scipy.special import erf, ndtr

SRC = (pathlib.Path(__file__).resolve().parent.parent / "paper_2606_28516_gb300" / "csrc" / "common.cuh").read_text()
BODY = SRC[SRC.index("struct GeluQ"):SRC.index("};", SRC.index("struct GeluQ"))]
C = [np.float32(re.search(rf"\bC{k} = ([-0-9.e]+)f", BODY).group(1)) for k in range(1, 11)]


def _fma(a, b, c):
    return (a.astype(np.float64) * b.astype(np.float64) + np.asarray(c, np.float64)).astype(np.float32)


def gelu_q(u):
    u = np.asarray(u, np.float32)
    t = np.minimum(np.abs(u), np.float32(20))
    q = np.full_like(t, C[9])
    for k in range(8, -1, -1):
        q = _fma(q, t, C[k])
    q = q * t
    e = np.exp2(q.astype(np.float64))
    e = np.where(e < 2.0 ** -126, 0, e).astype(np.float32)
    relu = _fma(np.full_like(u, 0.5), u, np.float32(0.5) * np.abs(u))
    return _fma(np.float32(-0.5) * t, e, relu)


def gelu_erf32(u):
    u = np.asarray(u, np.float32)
    e = erf((u * np.float32(0.70710678118654752440)).astype(np.float64)).astype(np.float32)
    return (np.float32(0.5) * u) * (np.float32(1) + e)


def exact(u):
    u = np.asarray(u, np.float64)
    return u * ndtr(u)


def test_largest_error():
    u = np.concatenate([np.linspace(-6, 6, 1_000_001), np.linspace(-60, 60, 400_001)]).astype(np.float32)
    near = np.abs(u) <= 4
    err = np.abs(gelu_q(u) - exact(u))
    assert err[near].max() <= 2.5e-7
    # past 4 the result is u (or 0) to float32
    assert (err[~near] <= np.maximum(2.5e-7, np.abs(u[~near].astype(np.float64)) * 2.0 ** -24)).all()


def test_mean_square_error_below_the_erf_form():
    rng = np.random.default_rng(0)
    for s in (0.28, 0.39, 0.6, 1.0):  # 0.02 sqrt(d) for d = 192, 384, and wider
        u = (s * rng.standard_normal(400_000)).astype(np.float32)
        new = np.mean((gelu_q(u) - exact(u)) ** 2)
        old = np.mean((gelu_erf32(u) - exact(u)) ** 2)
        assert new <= old, (s, new, old)


def test_specials():
    with np.errstate(invalid="ignore"):
        r = gelu_q(np.float32([np.inf, np.nan, 0.0, 1e30, -1e30]))
    assert r[0] == np.inf and np.isnan(r[1]) and r[2] == 0 and r[3] == np.float32(1e30) and r[4] == 0
