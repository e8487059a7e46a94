"""The bf16 layer's GELU at the values that an approximation treats apart, through the dense FFN: one hidden
unit's bias carries the value, W1 is zero and fc2 passes that unit on. NaN and -inf give NaN and inf gives
inf, as u (1 + erf(u / sqrt 2)) / 2 does; in the negative tail the result follows the float64 GELU (relative
error of the kernel's polynomial there: below 0.05, plus two roundings to bf16) down to -8, and is below 1e-17
from -9 on. Each instantiation of fc1's epilogue: the 1-SM kernel, the 2-SM kernel with eight epilogue warps
and with twelve."""
import math

import pytest
import torch

from paper_2606_28516_gb300 import clearmoe as cm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


@pytest.mark.parametrize("T,d,H", [(5, 64, 64), (300, 128, 256), (20000, 64, 256)])
def test_specials(T, d, H):
    bf = torch.bfloat16
    x = torch.randn(T, d, device="cuda").to(bf)
    W1 = torch.zeros(H, d, dtype=bf, device="cuda")
    W2 = torch.zeros(d, H, dtype=bf, device="cuda")
    W2[:, 3] = 1.0
    out = torch.empty_like(x)
    h = cm.clearmoe_layer_create(T, d, H, 1, 16, cm.BF16)
    try:
        for v in (-math.inf, math.inf, math.nan, -5.5, -6.0, -6.5, -8.0, -9.0, -12.0, -30.0, -1e30, 40.0, 1e30):
            b1 = torch.zeros(H, dtype=bf, device="cuda")
            b1[3] = v
            v = float(b1[3])
            cm.clearmoe_dense_ffn_forward(h, x, W1, b1, W2, out)
            assert cm.clearmoe_layer_status(h) == 0
            got = out.double()
            if math.isnan(v) or v == -math.inf:
                assert bool(torch.isnan(got).all()), v
            elif v > 0:
                assert bool((got == v).all()), v
            else:
                want = v * 0.5 * math.erfc(-v / math.sqrt(2.0)) if v >= -8 else 0.0
                assert bool(((got - want).abs() <= (0.05 + 2.0 ** -7) * abs(want) + (0.0 if want else 1e-17)).all()), v
    finally:
        cm.clearmoe_layer_destroy(h)
