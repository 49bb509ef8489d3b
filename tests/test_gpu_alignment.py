"""Pointers that need the alignment of their elements only: biases, skip factors, scan states and routing outputs that start 4, 8 or
12 bytes past a 16-byte boundary give the results of aligned ones, bit for bit, in every kernel that reads them."""
import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth

from rom_testlib import GpuLayer, assert_close, np64
from test_gpu_parity import small_shape

pytestmark = pytest.mark.gpu


def shifted(t, words):
    """A copy of a 4-byte tensor that starts `words` words past a 16-byte boundary."""
    if t is None:
        return None
    buf = torch.empty(t.numel() + 4, dtype=t.dtype, device=t.device)
    v = buf[words:words + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 16 == 4 * words
    return v


@pytest.mark.parametrize("words", [1, 2, 3])
@pytest.mark.parametrize("dtype,B,L,De,use_ws", [
    ("bf16", 2, 385, 64, True),          # chunks, chained states
    ("bf16", 40, 33, 512, False),        # one pass of the warp kernel
    ("bf16", 1, 100, 128, False),        # one pass for few sequences
    ("bf16", 40, 20, 384, False),        # general kernel
    ("bf16", 3, 1, 128, False),
    ("f32", 2, 100, 192, True),
])
def test_scan_unaligned_states_and_skip(dtype, B, L, De, use_ws, words):
    q = {k: v.cuda() for k, v in synth.make_scan_inputs(B, L, De, 16, dtype, 4400, with_z=True, with_h0=True).items()}
    cfg = rb.make_config(B, L, 64, De, 16, 4, 16, 1, 1, dtype)
    ws = torch.empty(max(rb.scan_workspace_size(cfg), 16), dtype=torch.uint8, device="cuda") if use_ws else None
    res = []
    for w in (0, words):
        y, hl = torch.empty_like(q["u"]), shifted(torch.zeros((B, De, 16), device="cuda"), w)
        rb.rom_scan(cfg, q["u"], q["delta"], q["A"], q["Bm"], q["Cm"], shifted(q["D"], w), q["z"], shifted(q["h0"], w), y, hl, ws)
        torch.cuda.synchronize()
        res.append((y, hl.clone()))
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])


def vectors(dev, words):
    return {k: shifted(v, words) if k in ("b_r", "b_conv", "D") else v for k, v in dev.items()}


@pytest.mark.parametrize("kw,flags", [
    (dict(B=40, L=97, K=1), 0),
    (dict(B=40, L=97, K=2), 0),
    (dict(B=2, L=65, K=3), 0),
    (dict(B=3, L=130, K=1), rb.ROM_FLAG_FUSED_SMALL),
    (dict(B=2, L=70, K=2, dtype="f32"), 0),
])
def test_layer_unaligned_vectors(kw, flags):
    s = small_shape(router_bias_scale=0.5, **kw)
    p = synth.make_inputs(s, recipe="unit")
    g = GpuLayer(s, p)      # (a b_conv off the boundary takes the three launches that the fused kernel replaces)
    ref = [g.forward().clone(), g.idx.clone(), g.gates.clone(), g.counts.clone()]
    g = GpuLayer(s, p, flags=flags)
    g.dev = vectors(g.dev, 1)
    g.weights = rb.make_weights(g.dev)
    g.idx, g.gates, g.counts = shifted(g.idx, 1), shifted(g.gates, 2), shifted(g.counts, 3)
    for a, b in zip(ref, [g.forward(), g.idx, g.gates, g.counts]):
        assert torch.equal(a, b)


@pytest.mark.parametrize("B,K", [(1, 1), (2, 2), (9, 1), (1, 3)])
def test_step_unaligned_vectors(B, K):
    s = small_shape(B=B, L=1, K=K, dtype="bf16", router_bias_scale=0.5)
    dev = {k: (None if v is None else v.cuda().contiguous()) for k, v in synth.make_inputs(s, recipe="unit").items()}
    cfg = rb.config_from_shape(s)
    ws = rb.alloc_workspace(cfg, "cuda")
    res = []
    for w in (0, 1):
        conv, ssm = torch.ones((B, s.d_conv - 1, s.d_inner), device="cuda"), torch.ones((B, s.d_inner, 16), device="cuda")
        out = torch.empty((B, s.d_model), dtype=torch.bfloat16, device="cuda")
        d = vectors(dev, w)
        d["b_dt"] = shifted(dev["b_dt"], w)
        rb.rom_layer_step(cfg, rb.make_weights(d), dev["x"][:, 0].contiguous(), conv, ssm, out, None, None, ws)
        torch.cuda.synchronize()
        res.append((out, conv, ssm))
    assert all(torch.equal(a, b) for a, b in zip(*res))


def test_backward_unaligned_vectors():
    s = small_shape(B=2, L=150, K=2, router_bias_scale=0.5)
    dev = {k: (None if v is None else v.cuda().contiguous()) for k, v in synth.make_inputs(s, recipe="unit").items()}
    cfg = rb.config_from_shape(s)
    ws = torch.empty(rb.layer_backward_workspace_size(cfg), dtype=torch.uint8, device="cuda")
    dout = torch.randn(dev["x"].shape, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda").to(torch.bfloat16)
    names = ("W_r", "b_r", "W_inz", "w_conv", "b_conv", "W_x", "W_dt", "b_dt", "A", "D", "W_out")
    res = []
    for w in (0, 1):
        grads = {"d" + n: torch.empty(dev[n].shape, device="cuda") for n in names}
        for n in ("db_r", "dD"):
            grads[n] = shifted(grads[n], w)
        dx = torch.empty_like(dev["x"])
        d = vectors(dev, w)
        rb.rom_layer_backward(cfg, rb.make_weights(d), d["x"], dout, dx, rb.make_grads(grads), ws)
        torch.cuda.synchronize()
        res.append({"dx": dx, **grads})
    for n in res[0]:      # atomic sums: fp32 rounding order (and its bf16 roundings downstream)
        assert_close(np64(res[1][n]), np64(res[0][n]), 1e-2 if n in ("dx", "dW_inz", "dW_r", "dw_conv", "db_conv", "dW_x") else 1e-4, n)
