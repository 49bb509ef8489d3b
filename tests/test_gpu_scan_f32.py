"""The fp32 scan against the fp64 recurrence.  The one-launch form: lengths around the 16 steps of a segment and the 256, 128 and 64 steps
of a round (by the number of blocks), several rounds, without a workspace as well.  The general form in chunks and in one pass with two,
four and eight states to a thread, on the other side of the line between the two.  And values that are not finite."""
import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from test_gpu_parity import run_scan
from rom_testlib import TOL, assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disc_mode", [0, 1])
@pytest.mark.parametrize("B,L,De,use_ws", [
    (1, 2, 64, True), (1, 15, 64, False), (1, 16, 128, True), (2, 17, 64, True), (1, 255, 512, True), (1, 257, 192, False),
    (1, 600, 64, True), (1, 129, 1024, True), (2, 300, 512, False), (3, 65, 1024, True), (5, 130, 1024, True),
    (15, 33, 2176, True), (16, 33, 2048, True),
    (1, 5000, 64, True), (1, 5000, 64, False), (1, 4100, 192, True), (1, 4100, 640, True), (1, 9000, 1024, True), (4, 97, 2048, True),
    (8, 200, 2048, True),
])
def test_scan_f32(disc_mode, B, L, De, use_ws):
    y, Y, hl, HL = run_scan(B, L, De, "f32", disc_mode, True, True, True, seed=7100 + L + De, use_ws=use_ws)
    assert_close(y, Y, TOL["f32"], "y")
    assert_close(hl, HL, TOL["f32"], "h_last")


@pytest.mark.parametrize("what", ["u", "B"])
def test_scan_f32_not_finite_stays_where_it_is(what):
    B, L, De, t_bad, c_bad = 1, 200, 64, 100, 5
    g = torch.Generator(device="cuda").manual_seed(3)
    r = lambda *s: torch.randn(*s, device="cuda", generator=g)      # noqa: E731
    u, d, A = r(B, L, De), torch.rand(B, L, De, device="cuda", generator=g) * 0.1, -torch.rand(De, 16, device="cuda", generator=g) * 15 - 0.5
    Bm, Cm = r(B, L, 16), r(B, L, 16)
    cfg = rb.make_config(B, L, De // 2, De, 16, 4, 16, 1, 1, "f32")
    ref, y = torch.empty_like(u), torch.empty_like(u)
    rb.rom_scan(cfg, u, d, A, Bm, Cm, None, None, None, ref, None)
    if what == "u":
        u[0, t_bad, c_bad] = float("inf")
    else:
        Bm[0, t_bad, 7] = float("nan")
    rb.rom_scan(cfg, u, d, A, Bm, Cm, None, None, None, y, None)
    torch.cuda.synchronize()
    assert torch.equal(y[:, :t_bad], ref[:, :t_bad])
    keep = [c for c in range(De) if c != c_bad] if what == "u" else []
    assert torch.equal(y[:, :, keep], ref[:, :, keep])
    assert not torch.isfinite(y[0, t_bad, c_bad])


@pytest.mark.parametrize("B,L,De", [(1, 1, 64), (1, 200, 64), (1, 3000, 64), (1, 700, 640)])
def test_scan_f32_infinite_state_stays_infinite(B, L, De):
    # every decay is above zero, their product over a segment (0.5 * 15 * 16 steps) is not: step by step the state is infinite from then on
    t_bad, c_bad = L // 3, 5
    u, d = torch.ones(B, L, De, device="cuda"), torch.full((B, L, De), 0.5, device="cuda")
    A, Bm = torch.full((De, 16), -15.0, device="cuda"), torch.ones(B, L, 16, device="cuda")
    cfg = rb.make_config(B, L, De // 2, De, 16, 4, 16, 1, 1, "f32")
    y, h_last = torch.empty_like(u), torch.empty(B, De, 16, device="cuda")
    u[0, t_bad, c_bad] = float("inf")
    rb.rom_scan(cfg, u, d, A, Bm, Bm, torch.ones(De, device="cuda"), None, None, y, h_last)
    torch.cuda.synchronize()
    assert torch.isposinf(y[0, t_bad:, c_bad]).all() and torch.isposinf(h_last[0, c_bad]).all()
    assert torch.isfinite(y[0, :t_bad]).all() and torch.isfinite(y[:, :, [c for c in range(De) if c != c_bad]]).all()


@pytest.mark.parametrize("B,L,De,disc_mode,launches", [
    (1, 256, 512, 0, 1), (1, 4096, 512, 0, 1), (1, 2048, 64, 1, 3), (1, 16384, 64, 0, 3), (1, 4096, 192, 0, 3), (1, 512, 64, 1, 1),
    (24, 1024, 1024, 1, 3), (24, 1024, 1024, 0, 1),
])
def test_scan_f32_form(B, L, De, disc_mode, launches):
    # the faster form, by its launches: one, or (chunks) two and the chain between them
    t = lambda *s: torch.zeros(*s, device="cuda")      # noqa: E731
    cfg = rb.make_config(B, L, De // 2, De, 16, 4, 16, 1, 1, "f32", disc_mode=disc_mode)
    ws = torch.empty(max(rb.scan_workspace_size(cfg), 1), dtype=torch.uint8, device="cuda")
    rb.rom_scan(cfg, t(B, L, De), t(B, L, De), t(De, 16) - 1, t(B, L, 16), t(B, L, 16), None, None, None, t(B, L, De), None, ws)
    assert rb.last_launch_count() == launches
    torch.cuda.synchronize()
