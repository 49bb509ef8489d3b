"""The one-launch bf16 scan against the CPU oracle: sequences around the eight steps of a tile and the twelve warps that take tiles in turn
(from about 156 steps on: shorter ones run in one pass), one and two rounds of blocks, every gate / skip / initial state combination; in the layer with one to three Gate rows a token, and with the
checkpoints of the backward pass.  And values that are not finite: what they give step by step."""
import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth
from rom_testlib import TOL, GpuLayer, assert_close, recorded, scan_kernels
from test_gpu_backward import bshape, run_layer_backward
from test_gpu_parity import check_layer, run_scan, small_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disc_mode", [0, 1])
@pytest.mark.parametrize("B,L,De,with_z,with_h0,with_D", [
    (1, 192, 4096, True, True, True),         # twenty-four tiles, two to a warp
    (2, 193, 2048, True, False, True),        # twenty-five, the last of one step
    (1, 287, 4096, False, True, False),       # thirty-six, the last of seven
    (1, 161, 192, True, True, True),          # six blocks: channels that fill no 128
    (2, 289, 320, True, True, False),
    (1, 480, 4096, True, False, False),
    (2, 201, 4096, True, True, False),        # two rounds of blocks, tiles the warps do not share evenly
    (3, 384, 3072, True, False, True),
])
def test_scan_ring(disc_mode, B, L, De, with_z, with_h0, with_D):
    with recorded("rom_scan") as calls:
        y, Y, hl, HL = run_scan(B, L, De, "bf16", disc_mode, with_z, with_h0, with_D, seed=8600 + L, use_ws=True)
    assert scan_kernels(calls[0]) == ["ring"]
    assert_close(y, Y, TOL["bf16"], "y")
    assert_close(hl, HL, 2e-3, "h_last")


@pytest.mark.parametrize("K", [1, 2, 3])
@pytest.mark.parametrize("L,De", [(160, 4096), (199, 192), (201, 256)])
def test_layer_forward_scan_ring(K, L, De):
    with recorded("rom_layer_forward") as calls:
        check_layer(small_shape(B=1, L=L, d_model=64, d_inner=De, E=4, K=K), "unit")
    assert scan_kernels(calls[0]) == ["ring"]


@pytest.mark.parametrize("K", [1, 2])
@pytest.mark.parametrize("L,De", [(161, 2048), (200, 192)])
@pytest.mark.parametrize("disc_mode", [0, 1])
def test_layer_backward_scan_ring(L, De, K, disc_mode):
    with recorded("rom_layer_backward") as calls:
        run_layer_backward(bshape(B=1, L=L, d_model=64, d_inner=De, K=K), disc_mode=disc_mode)
    assert "ring" in scan_kernels(calls[0])


def ring_inputs(B, L, De, delta, A, disc_mode):
    """Inputs of ones, an initial state of ones; the call that scans them, and y and the final state that it writes."""
    one = lambda *shape: torch.ones(*shape, device="cuda")      # noqa: E731
    q = dict(u=one(B, L, De).bfloat16(), delta=one(B, L, De) * delta, A=-one(De, 16) * A, Bm=one(B, L, 16), Cm=one(B, L, 16), D=one(De), h0=one(B, De, 16))
    y, h_last = torch.empty_like(q["u"]), one(B, De, 16)
    cfg = rb.make_config(B, L, 64, De, 16, 4, 16, 1, 1, "bf16", 0, disc_mode)
    ws = torch.empty(rb.scan_workspace_size(cfg), dtype=torch.uint8, device="cuda")

    def call():
        rb.rom_scan(cfg, q["u"], q["delta"], q["A"], q["Bm"], q["Cm"], q["D"], None, q["h0"], y, h_last, ws)
    call()
    assert scan_kernels(call) == ["ring"]
    return q, call, y, h_last


@pytest.mark.parametrize("name", ["u", "z"])
def test_scan_with_its_output_in_the_place_of_an_input(name):
    # the one-launch form, which may go over a sequence twice, does not take it
    B, L, De = 2, 201, 192
    g = torch.Generator(device="cuda").manual_seed(11)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)      # noqa: E731
    q = dict(u=r(B, L, De).bfloat16(), z=r(B, L, De).bfloat16())
    delta, A, Bm, Cm = 0.1 * r(B, L, De).abs(), -(0.5 + 15 * r(De, 16).abs()), r(B, L, 16), r(B, L, 16)
    cfg = rb.make_config(B, L, 64, De, 16, 4, 16, 1, 1, "bf16")
    ws = torch.empty(rb.scan_workspace_size(cfg), dtype=torch.uint8, device="cuda")
    y = torch.empty_like(q["u"])

    def call(t):
        rb.rom_scan(cfg, t["u"], delta, A, Bm, Cm, None, t["z"], None, t.get("y", t[name]), None, ws)
    call(dict(q, y=y))
    again = {k: v.clone() for k, v in q.items()}
    call(again)
    torch.cuda.synchronize()
    got = again[name].float()
    assert (got - y.float()).norm() <= 2e-3 * y.float().norm()      # outputs rounded to bf16 from sums in two orders: an ulp here and there
    assert scan_kernels(lambda: call(dict(q, y=y))) == ["ring"] and scan_kernels(lambda: call(again)) == ["warp", "warp"]


@pytest.mark.parametrize("disc_mode", [0, 1])
@pytest.mark.parametrize("L,De", [(160, 64), (203, 192)])
def test_scan_ring_infinite_state_stays_infinite(L, De, disc_mode):
    # every decay is above zero, their product over a tile (exp(-15)^8) is not: step by step the state is infinite from the first step on
    q, call, y, h_last = ring_inputs(1, L, De, 1.0, 15.0, disc_mode)
    c_bad = 37
    q["h0"][0, c_bad] = float("inf")
    call()
    torch.cuda.synchronize()
    rest = [c for c in range(De) if c != c_bad]
    assert torch.isposinf(y[0, :, c_bad]).all() and torch.isposinf(h_last[0, c_bad]).all()
    assert torch.isfinite(y[:, :, rest]).all() and torch.isfinite(h_last[:, rest]).all()


def test_scan_ring_state_that_becomes_infinite():
    # (with B-bar = Delta B: the zero-order hold takes the input from the state, infinite from infinite)
    L, t_bad, c_bad = 203, 101, 5
    q, call, y, h_last = ring_inputs(1, L, 64, 1.0, 15.0, 1)
    q["u"][0, t_bad, c_bad] = float("inf")
    call()
    torch.cuda.synchronize()
    rest = [c for c in range(64) if c != c_bad]
    assert torch.isposinf(y[0, t_bad:, c_bad]).all() and torch.isposinf(h_last[0, c_bad]).all()
    assert torch.isfinite(y[0, :t_bad]).all() and torch.isfinite(y[:, :, rest]).all()


@pytest.mark.parametrize("disc_mode", [0, 1])
def test_scan_ring_infinite_output_weight(disc_mode):
    # no input in the tile, so that its outputs come from the state before it alone: infinite where C is
    L, t_bad = 203, 101
    q, call, y, h_last = ring_inputs(1, L, 64, 0.1, 0.5, disc_mode)
    q["u"][0, 96:104] = 0
    q["Cm"][0, t_bad, 7] = float("inf")
    call()
    torch.cuda.synchronize()
    assert torch.isposinf(y[0, t_bad]).all()
    assert torch.isfinite(y[0, [t for t in range(L) if t != t_bad]]).all() and torch.isfinite(h_last).all()


@pytest.mark.parametrize("B,L,De,disc_mode,ring", [
    (1, 400, 64, 0, True), (1, 600, 64, 0, False), (1, 800, 512, 1, False), (1, 16000, 2048, 0, False), (1, 2500, 3072, 0, True),
    (1, 1000, 4096, 0, True), (3, 600, 2048, 1, False), (3, 224, 1600, 0, False), (4, 2048, 2048, 0, True), (3, 1371, 2048, 0, False),
    (8, 600, 1024, 1, True), (3, 512, 4096, 0, False),
])
def test_scan_form(B, L, De, disc_mode, ring):
    # the faster of the two forms, as measured
    zeros = lambda *shape: torch.zeros(*shape, device="cuda")      # noqa: E731
    u, y = zeros(B, L, De).bfloat16(), zeros(B, L, De).bfloat16()
    cfg = rb.make_config(B, L, 64, De, 16, 4, 16, 1, 1, "bf16", 0, disc_mode)
    ws = torch.empty(rb.scan_workspace_size(cfg), dtype=torch.uint8, device="cuda")
    delta, A, Bm = zeros(B, L, De), zeros(De, 16) - 1, zeros(B, L, 16)

    def call():
        rb.rom_scan(cfg, u, delta, A, Bm, Bm, None, None, None, y, None, ws)
    call()
    assert scan_kernels(call) == (["ring"] if ring else ["warp", "warp"])


@pytest.mark.parametrize("B,L,De,K,ring", [(3, 300, 2048, 1, True), (3, 300, 2048, 2, True), (3, 600, 2048, 1, False), (2, 600, 192, 1, False),
                                           (2, 500, 192, 1, True), (4, 1476, 1664, 3, False)])
def test_layer_scan_form(B, L, De, K, ring):
    # (in the layer the line lies a little elsewhere)
    s = small_shape(B=B, L=L, d_model=64, d_inner=De, E=4, K=K)
    g = GpuLayer(s, synth.make_inputs(s, recipe="unit"))
    g.forward()
    call = lambda: rb.rom_layer_forward(g.cfg, g.weights, g.dev["x"], g.out, g.idx, g.gates, g.counts, g.ws)      # noqa: E731
    assert scan_kernels(call) == (["ring"] if ring else ["warp", "warp"])
