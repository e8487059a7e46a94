"""fp32 layers whose kernels overlap their predecessors (fc1's products run beside the routing kernel, the
expert GEMM's z segments beside the basis kernel): a chain of layers, each reading the previous one's output
through the same scratch buffers, gives the bits that it gives with a synchronisation after every layer, and
the first layer lies within the fp32 tolerance of the oracle. Few tokens (K split, most SMs idle), ranks that
end inside a K block (r = 16, 48), an expert GEMM of many tiles."""
import numpy as np
import pytest
import torch

import synth
from paper_2606_28516_gb300 import clearmoe as cm

from gpu_util import get_routing, handle_for, oracle_rows, out_error, sample_rows, tol

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


@pytest.mark.parametrize("T,d,E,r,cls", [(49, 192, 4, 16, 0), (788, 192, 4, 48, 197), (1, 64, 1, 16, 1),
                                         (197, 384, 16, 192, 0), (12608, 192, 4, 16, 197)])
def test_chain(T, d, E, r, cls):
    L = synth.make_layer(synth.LayerShape("overlap", T, d, 4 * d, E, r, "f32", n_cal=2000))
    D = synth.to_torch(L)
    W2 = torch.randn(d, 4 * d, device="cuda", generator=torch.Generator("cuda").manual_seed(1)) / (2 * d ** 0.5)

    def layer(h, x):
        y = torch.full_like(x, float("nan"))
        cm.clearmoe_ffn_forward_ex(h.h, x, D["W1"], D["b1"], D["U"], D["S"], D["Vh"], D["residuals"], D["Wg"],
                                   D["bg"], y, W2=W2 if cls else None, cls_stride=cls)
        return y

    with handle_for(L) as h:
        want = [D["x"]]
        for _ in range(8):
            want.append(layer(h, want[-1]))
            torch.cuda.synchronize()
            if not cls and len(want) == 2:
                gr = get_routing(h, T, E)
                rows = sample_rows(gr, T, 512)[:1024]
                y = oracle_rows(L, rows, gr["a"][rows])
                assert out_error(want[1][torch.from_numpy(rows).cuda()], y, "f32") <= tol("f32")
        for _ in range(20):
            got = [D["x"]]
            for _ in range(8):
                got.append(layer(h, got[-1]))
            for a, b in zip(got[1:], want[1:]):
                assert bool(torch.isfinite(a).all()) and torch.equal(a, b)
        assert cm.clearmoe_layer_status(h.h) == 0
