"""GEMM kernels whose bounded waits run out: with wait limits of 1 to 200 microseconds
(clearmoe_debug_set_wait) and long K loops the kernels give up between their copies, let what is in flight
land, and return. The call reports CLEARMOE_ETIMEOUT through the status word or completes; afterwards, with
the usual limit, the handle gives the bits that it gave before. The next call's kernels start on the SMs that
the ones that gave up have just left."""
import pytest
import torch

from paper_2606_28516_gb300 import clearmoe as cm

pytestmark = pytest.mark.gpu

LIMITS = (1_000, 4_000, 16_000, 50_000, 200_000)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def _call(kind, T, d, H, E, r, dtype):
    g = torch.Generator(device="cuda").manual_seed(T + d + H)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    w = lambda *s: (0.02 * torch.randn(*s, generator=g, device="cuda")).to(tdt)
    x, out = w(T, d) * 50, torch.empty(T, d, dtype=tdt, device="cuda")
    W1, b1, W2, U, Vh, res, Wg, bg = w(H, d), w(H), w(d, H), w(d, r), w(r, H), w(E, d, H), w(E, d), w(E)
    S = torch.rand(r, generator=g, device="cuda") + 0.5
    h = cm.clearmoe_layer_create(T, d, H, E, r, cm.BF16 if dtype == "bf16" else cm.F32)
    if kind == "dense":
        return h, out, lambda: cm.clearmoe_dense_ffn_forward(h, x, W1, b1, W2, out)
    opts = {"layer": {}, "classes": dict(W2=W2, cls_stride=197), "router_in_fc1": dict(router_in_fc1=True)}[kind]
    return h, out, lambda: cm.clearmoe_ffn_forward_ex(h, x, W1, b1, U, S, Vh, res, Wg, bg, out, **opts)


@pytest.mark.parametrize("kind,T,d,H,E,r,dtype", [
    ("dense", 300, 256, 32768, 1, 64, "bf16"), ("dense", 3000, 768, 16384, 1, 64, "bf16"),
    ("layer", 9973, 768, 4096, 8, 256, "bf16"), ("layer", 300, 768, 4096, 4, 48, "bf16"),
    ("classes", 6304, 768, 4096, 4, 128, "bf16"), ("router_in_fc1", 3000, 768, 4096, 4, 64, "bf16"),
    # fc1 on the 1-SM kernel, its rows gathered by slot; the 1-SM kernel throughout; fp32
    ("layer", 3000, 1024, 8192, 4, 64, "bf16"), ("layer", 1000, 64, 16448, 2, 16, "bf16"),
    ("layer", 3000, 192, 16384, 4, 32, "f32"), ("dense", 300, 512, 8192, 1, 32, "f32"),
])
def test_gives_up_and_recovers(kind, T, d, H, E, r, dtype):
    h, out, call = _call(kind, T, d, H, E, r, dtype)
    try:
        call()
        assert cm.clearmoe_layer_status(h) == 0
        want = out.clone()
        gave_up = []
        for limit in LIMITS:
            for _ in range(4):
                cm.clearmoe_debug_set_wait(h, limit, 0)
                call()
                call()
                st = cm.clearmoe_layer_status(h)
                assert st in (0, cm.ETIMEOUT), (limit, st)
                gave_up.append(st == cm.ETIMEOUT)
                cm.clearmoe_debug_set_wait(h, 1_000_000_000, 0)
                out.fill_(float("nan"))
                call()
                assert cm.clearmoe_layer_status(h) == 0
                assert torch.equal(out, want), limit
        assert gave_up[0]
    finally:
        cm.clearmoe_layer_destroy(h)


@pytest.mark.parametrize("kind", ["layer", "classes", "router_in_fc1"])
def test_first_call_gives_up(kind):
    """A handle whose first calls give up has no routing of an earlier call behind it."""
    args = (kind, 3000, 768, 4096, 4, 64, "bf16")
    h, want, call = _call(*args)
    h2, out, call2 = _call(*args)
    try:
        call()
        assert cm.clearmoe_layer_status(h) == 0
        cm.clearmoe_debug_set_wait(h2, 1_000, 0)
        for _ in range(3):
            call2()
        assert cm.clearmoe_layer_status(h2) == cm.ETIMEOUT
        cm.clearmoe_debug_set_wait(h2, 1_000_000_000, 0)
        call2()
        assert cm.clearmoe_layer_status(h2) == 0 and torch.equal(out, want)
    finally:
        cm.clearmoe_layer_destroy(h)
        cm.clearmoe_layer_destroy(h2)
