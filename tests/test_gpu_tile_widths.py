"""The 2-SM kernels' tile width follows the token count (fc1: 256 or 128 columns by rounds of tiles; experts and
dense fc2: the narrowest tile that runs in one round). Every width sums each output over K in the same
order, so a batch cut into pieces that take other widths gives the same bits: sizes on both sides of
each line, ragged last blocks, one expert and several, both basis forms and the dense FFN."""
import pytest
import torch

import synth
from paper_2606_28516_gb300 import clearmoe as cm

from gpu_util import handle_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


@pytest.mark.parametrize("d,E,r,pieces", [
    (768, 8, 128, (1, 255, 1000, 3000, 9010)), (768, 1, 64, (257, 1800, 6304)), (384, 4, 64, (197, 2000, 5000)),
    (1024, 3, 16, (100, 1400, 4000)),
])
def test_pieces_give_the_same_bits(d, E, r, pieces):
    T = sum(pieces) + 777
    L = synth.make_layer(synth.LayerShape("tiles", T, d, 4 * d, E, r, "bf16", n_cal=2000))
    D = synth.to_torch(L)
    with handle_for(L) as h:
        def forward(x, kind):
            out = torch.full_like(x, float("nan"))
            if kind == "factored":
                cm.clearmoe_ffn_forward(h.h, x, D["W1"], D["b1"], D["U"], D["S"], D["Vh"], D["residuals"], D["Wg"],
                                        D["bg"], out)
            elif kind == "folded":
                cm.clearmoe_ffn_forward_folded(h.h, x, D["W1"], D["b1"], D["residuals"], D["Wg"], D["bg"], out)
            else:
                cm.clearmoe_dense_ffn_forward_ex(h.h, x, D["W1"], D["b1"], D["W2"], D["b2"], out)
            return out

        for kind in ("factored", "folded", "dense"):
            whole = forward(D["x"], kind)
            lo = 0
            for n in (*pieces, 777):
                part = forward(D["x"][lo:lo + n], kind)
                assert torch.equal(part, whole[lo:lo + n]), f"{kind}: rows {lo}..{lo + n}"
                lo += n
        assert cm.clearmoe_layer_status(h.h) == 0
