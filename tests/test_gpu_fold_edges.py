"""The fold kernel at the edges of its tiles (32 rows x 128 columns, k chunks of 32): ranks below, at and
past a chunk, widths that end inside a tile, one expert and sixteen, W_shared alone, and matrices that
start off the vector alignment (served element by element). Against the float64 sum; the bound is the
result type's unit roundoff plus the fp32 sums' rounding, r + 2 roundings of 2^-24 on the sum of the
magnitudes of the terms."""
import pytest
import torch

from paper_2606_28516_gb300 import clearmoe as cm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def _rand(g, *shape, dtype, off=0):
    """A contiguous tensor whose first element lies `off` elements past an aligned address."""
    n = 1
    for s in shape:
        n *= s
    return torch.randn(n + off, generator=g, device="cuda").to(dtype)[off:].view(*shape)


@pytest.mark.parametrize("dtype,d,H,E,r,off", [
    ("bf16", 64, 64, 1, 16, 0), ("bf16", 64, 192, 16, 1, 0), ("bf16", 192, 320, 3, 33, 0),
    ("bf16", 128, 256, 2, 64, 0), ("bf16", 64, 128, 4, 40, 1), ("bf16", 64, 128, 4, 40, 2),
    ("f32", 36, 132, 2, 20, 0), ("f32", 4, 4, 1, 4, 0), ("f32", 68, 260, 5, 32, 0), ("f32", 40, 128, 3, 12, 1),
])
def test_fold_and_materialize(dtype, d, H, E, r, off):
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(d * 1000 + H + r)
    U, Vh = _rand(g, d, r, dtype=tdt), _rand(g, r, H, dtype=tdt, off=off)
    S = torch.rand(r, generator=g, device="cuda") + 0.1
    res = [_rand(g, d, H, dtype=tdt, off=off) for _ in range(E)]
    out = [torch.full((d * H + off,), float("nan"), device="cuda").to(tdt)[off:].view(d, H) for _ in range(E + 1)]
    h = cm.clearmoe_layer_create(1, d, H, E, min(max(r, 1), d, H), cm.BF16 if dtype == "bf16" else cm.F32)
    try:
        cm.clearmoe_fold_basis(h, U, S, Vh, res, out[:E])
        cm.clearmoe_materialize_basis(h, U, S, Vh, out[E])
        assert cm.clearmoe_layer_status(h) == 0
    finally:
        cm.clearmoe_layer_destroy(h)
    W = (U.double() * S.double()) @ Vh.double()
    mag = (U.double().abs() * S.double()) @ Vh.double().abs()
    half = 2.0 ** (-8 if dtype == "bf16" else -24)  # unit roundoff: 8 and 24 significant bits
    for e in range(E + 1):
        add = res[e].double() if e < E else torch.zeros_like(W)
        want = W + add
        bound = half * want.abs() * 1.01 + (r + 2) * 2.0 ** -24 * (mag + add.abs()) * (1 + half)
        assert bool(((out[e].double() - want).abs() <= bound).all()), f"matrix {e}"
