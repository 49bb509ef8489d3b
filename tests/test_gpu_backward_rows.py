"""Row passes of the layer's backward in their bf16 top-1 / top-2 forms (reverse of the combine, dx): token counts off the four tokens
of a block and the eight of a thread, widths off the 128 vectors of a pass, 4, 8 and 16 experts and counts without their own form.
(Sums over too few tokens do not average the bf16 roundings down to the 2e-2 of the comparison: one token leaves 3.8e-2 in dW_x, 70 of
six experts 2.25e-2 in dA, the general forms the same.  Few tokens are therefore compared on the rows themselves: what the reverse of the
combine leaves for dW_out and db_r against the forward's rows in fp64, and dx against the general form.)"""
import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth
from rom_testlib import TOL, GpuLayer, assert_close, np64
from test_gpu_backward import bshape, run_layer_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(B=1, L=131, E=8, K=1, d_model=192, d_inner=320), dict(B=2, L=77, E=8, K=2, d_model=64, d_inner=1088),
    dict(B=1, L=93, E=16, K=1), dict(B=3, L=43, E=16, K=2, d_model=320), dict(B=1, L=70, E=4, K=2), dict(B=1, L=133, E=6, K=2),
    dict(B=1, L=257, E=11, K=1), dict(B=1, L=300, E=18, K=2),
])
def test_backward_row_passes(kw):
    run_layer_backward(bshape(dtype="bf16", **kw))


def few_tokens(T, E, K, d_model=128, d_inner=256):
    s = bshape(B=1, L=T, E=E, K=K, d_model=d_model, d_inner=d_inner)
    p = synth.make_inputs(s, recipe="unit")
    p["b_r"] = torch.zeros(E)
    return s, p, torch.randn(p["x"].shape, generator=torch.Generator().manual_seed(17)).bfloat16()


def backward(s, p, dout):
    cfg = rb.config_from_shape(s)
    dev = {k: (None if v is None else v.cuda().contiguous()) for k, v in p.items()}
    grads = {"d" + n: torch.empty(dev[n].shape, dtype=torch.float32, device="cuda")
             for n in ("W_r", "b_r", "W_inz", "w_conv", "b_conv", "W_x", "W_dt", "b_dt", "A", "D", "W_out") if dev.get(n) is not None}
    dx = torch.empty_like(dev["x"])
    ws = torch.empty(rb.layer_backward_workspace_size(cfg), dtype=torch.uint8, device="cuda")
    rb.rom_layer_backward(cfg, rb.make_weights(dev), dev["x"], dout.cuda(), dx, rb.make_grads(grads), ws)
    torch.cuda.synchronize()
    return dx, grads


@pytest.mark.parametrize("T", [1, 3, 9])
@pytest.mark.parametrize("K,d_inner", [(1, 320), (2, 1088)])
def test_backward_combine_rows_of_few_tokens(T, K, d_inner):
    s, p, dout = few_tokens(T, 5, K, d_inner=d_inner)
    g = GpuLayer(s, p)
    g.forward()
    rows = g.tap("row_of_assign", torch.int32, K).long()
    idx, gate, dO = g.idx.long(), g.gates.double(), dout.cuda().double().view(T, -1)
    Yg, W = g.tap("Ygp", torch.bfloat16, d_inner)[rows[:, 0]].double(), g.dev["W_out"].double()
    P = torch.softmax(g.dev["x"].double().view(T, -1) @ g.dev["W_r"].double().T, dim=1)
    dW, db, db_scale = torch.zeros_like(W), torch.zeros(5, dtype=torch.float64, device="cuda"), 0.0
    for t in range(T):
        for k in range(K):
            e = idx[t, k]
            dW[e] += torch.outer(dO[t], gate[t, k] * Yg[t])
            back = dO[t] @ W[e]
            db += (back @ Yg[t]) * P[t, e] * (torch.nn.functional.one_hot(e, 5) - P[t])
            db_scale += back.norm() * Yg[t].norm() * P[t, e]
    _, got = backward(s, p, dout)
    # The pass recomputes Yg from rows rounded elsewhere (the gate before its SiLU, at top-2 the sums over the slots): bf16 roundings of 2^-8, a
    # few in a row, 2e-2 in 2-norm at most.  A lost 16-byte piece of 1088 channels is 8.6e-2 of a row.
    assert ((got["dW_out"].double() - dW).norm(dim=(1, 2)) <= TOL["bf16"] * dW.norm(dim=(1, 2))).all()
    assert ((got["db_r"].double() - db).abs() <= TOL["bf16"] * db_scale).all()


@pytest.mark.parametrize("T", [1, 3, 9])
@pytest.mark.parametrize("K", [1, 2])
@pytest.mark.parametrize("E", [4, 8, 16])
def test_backward_dx_of_few_tokens(T, K, E):
    """Experts that no token can choose change nothing: with 18 of them the general form writes dx."""
    s, p, dout = few_tokens(T, E, K, d_model=192)
    dx, _ = backward(s, p, dout)
    s2, p2, _ = few_tokens(T, 18, K, d_model=192)
    for n in ("W_r", "W_inz", "W_out"):
        p2[n][:E] = p[n]
    p2["b_r"][E:] = -1e30
    for n in ("x", "w_conv", "b_conv", "W_x", "W_dt", "b_dt", "A", "D"):
        p2[n] = p[n]
    ref, _ = backward(s2, p2, dout)
    # both round the same values at the same points; sums by atomics flip last bits of bf16 (2^-8) in the rows that lead to dx
    assert_close(np64(dx), np64(ref), 2.0 ** -7, "dx")
