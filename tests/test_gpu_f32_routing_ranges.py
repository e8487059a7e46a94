"""The fp32 routing kernel takes as many ranges of tokens as fc1's prefix table holds (256, or 2,432 / E), so
that fc1's epilogue forms the slots: expert counts on both sides of 2,432 / 256, one range more or less
rows than a multiple. Routing against the
oracle (bit-exact outside near ties; counts, offsets and perm the stable sort), outputs of sampled rows
within the fp32 tolerance."""
import numpy as np
import pytest
import torch

import synth
from paper_2606_28516_gb300 import clearmoe as cm

from gpu_util import check_routing, get_routing, handle_for, oracle_rows, out_error, run_ffn, sample_rows, tol

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


@pytest.mark.parametrize("T,d,E", [(256 * 40, 192, 9), (256 * 40 + 1, 192, 10), (12608, 192, 4), (9001, 384, 16), (4097, 64, 1)])
def test_ranges(T, d, E):
    L = synth.make_layer(synth.LayerShape("ranges", T, d, 4 * d, E, 16, "f32", n_cal=2000))
    D = synth.to_torch(L)
    with handle_for(L) as h:
        out = run_ffn(h, D)
        gr = get_routing(h, T, E)
        assert cm.clearmoe_layer_status(h.h) == 0
    check_routing(gr, L["x"], L["Wg"], L["bg"])
    rows = sample_rows(gr, T, 512)[:2048]
    y = oracle_rows(L, rows, gr["a"][rows])
    assert np.all(np.isfinite(out.float().cpu().numpy()))
    assert out_error(out[torch.from_numpy(rows).cuda()], y, "f32") <= tol("f32")
