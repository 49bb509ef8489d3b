"""Edges of the bf16 single-token step's own kernels (few tokens per expert) against the CPU oracle: the register-fed and the
streamed projections on both sides of their dispatch line, one to several passes of 64 token columns, 16 / 32 / 64 columns, a K
range that leaves half a stage, weight tiles cut short, dt ranks off the 32- and 128-wide blocks, every conv width."""
import numpy as np
import pytest
import torch

from oracle import rom_oracle as O
from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth

from rom_testlib import np64
from test_gpu_parity import run_steps, small_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(B=1, E=8, K=1),                                         # one assignment: register-fed projections
    dict(B=3, E=8, K=1, d_model=192, d_inner=320, dt_rank=48),   # the last below the line; partial groups of 8 tokens
    dict(B=2, E=4, K=2, d_model=64, d_inner=64, d_conv=2),       # the first streamed one; half of the only K stage missing
    dict(B=17, E=1, K=1, d_model=192, d_inner=448, dt_rank=144), # 32 columns; rows cut at 448 % 128; more than 128 dt columns
    dict(B=33, E=2, K=2, d_model=128, d_inner=256, d_conv=3),    # 64 columns, slots summed by their own kernels
    dict(B=70, E=1, K=1, d_model=128, d_inner=192),              # two passes of columns
    dict(B=130, E=3, K=3, d_model=64, d_inner=128, router_bias_scale=2.0),
    dict(B=9, E=64, K=8, d_model=128, d_inner=128),              # every expert may be selected, most by one or two tokens
])
def test_step_small_parity(kw):
    run_steps(small_shape(**{**dict(L=4, dtype="bf16"), **kw}), 3)


@pytest.mark.parametrize("kw", [
    dict(B=1, E=64, K=3, d_model=192, d_inner=128),                            # three picks of one token, most expert groups full
    dict(B=1, E=9, K=1, d_model=2112, d_inner=192, router_bias_scale=1.0),     # a second round of the contracted index, a lone ninth expert
    dict(B=2, E=8, K=1, d_model=256, d_inner=2304, d_conv=2),                  # two tokens, two experts: the most blocks that route themselves
    dict(B=2, E=8, K=1, d_model=256, d_inner=2368),                            # more: a launch of its own routes
])
def test_step_route_inside_the_projection(kw):
    run_steps(small_shape(**{**dict(L=4, dtype="bf16"), **kw}), 3)


@pytest.mark.parametrize("B,E,K,d_model,launches", [
    (1, 8, 1, 2048, 4), (1, 64, 1, 1280, 4), (1, 64, 1, 1344, 5), (1, 24, 1, 1600, 5), (2, 8, 1, 512, 4), (2, 8, 1, 576, 5), (2, 64, 1, 128, 5),
])
def test_step_routes_inside_only_few_logits(B, E, K, d_model, launches):
    s = small_shape(B=B, L=1, E=E, K=K, d_model=d_model, d_inner=128, dtype="bf16")
    p = synth.make_inputs(s, recipe="unit")
    idx, gates = one_step(s, p, B)[3:5]
    assert rb.last_launch_count() == launches
    ref_idx, ref_gate, _, _ = O.route(np64(p["x"]).reshape(B, d_model), np64(p["W_r"]), np64(p["b_r"]), K, 0)
    np.testing.assert_array_equal(idx.cpu().numpy(), ref_idx)
    np.testing.assert_allclose(gates.cpu().numpy(), ref_gate, rtol=2e-6, atol=1e-30)


def one_step(s, p, B, flags=0):
    """One token for the first B sequences of p from seeded states; (out, conv_state, ssm_state, idx, gates, workspace)."""
    cfg = rb.config_from_shape(s.replace(B=B, L=1), flags=flags)
    dev = {k: (None if v is None else v.cuda().contiguous()) for k, v in p.items()}
    conv = synth._randn(771, (s.B, s.d_conv - 1, s.d_inner))[:B].cuda()
    ssm = synth._randn(772, (s.B, s.d_inner, s.d_state), 0.3)[:B].cuda()
    out = torch.empty((B, s.d_model), dtype=synth.torch_dtype(s), device="cuda")
    idx = torch.empty((B, s.K), dtype=torch.int32, device="cuda")
    gates = torch.empty((B, s.K), dtype=torch.float32, device="cuda")
    ws = rb.alloc_workspace(cfg, "cuda")
    rb.rom_layer_step(cfg, rb.make_weights(dev), dev["x"][:B, 0].contiguous(), conv, ssm, out, idx, gates, ws)
    torch.cuda.synchronize()
    return out, conv, ssm, idx, gates, ws


@pytest.mark.parametrize("scale", [2.0 ** -80, 2.0 ** -68, 2.0 ** 70])
@pytest.mark.parametrize("B", [1, 2, 9])
def test_step_route_products_outside_fp32(B, scale):
    """Router products below and above the range of fp32: logits are fp64 sums of exact products, so the routing is the oracle's."""
    s = small_shape(B=B, L=1, E=8, K=2, d_model=320, dtype="bf16")
    p = synth.make_inputs(s, recipe="unit")
    p["x"], p["W_r"], p["W_inz"] = p["x"] * scale, p["W_r"] * scale, torch.zeros_like(p["W_inz"])
    _, _, _, idx, gates, _ = one_step(s, p, B)
    ref_idx, ref_gate, _, _ = O.route(np64(p["x"]).reshape(B, s.d_model), np64(p["W_r"]), None, s.K, 0)
    np.testing.assert_array_equal(idx.cpu().numpy(), ref_idx)
    np.testing.assert_allclose(gates.cpu().numpy(), ref_gate, rtol=2e-6, atol=1e-30)


@pytest.mark.parametrize("K,sizes", [(1, (4, 9, 70)), (2, (2, 7, 64))])
def test_step_result_does_not_depend_on_the_batch(K, sizes):
    """From four assignments on, a sequence's output and states are the same to the last bit whatever the batch around it."""
    s = small_shape(B=sizes[-1], L=1, E=8, K=K, d_model=1024, d_inner=2048, dtype="bf16")
    p = synth.make_inputs(s, recipe="unit")
    ref = one_step(s, p, sizes[-1])
    for B in sizes[:-1]:
        got = one_step(s, p, B)
        for name, a, b in zip(("out", "conv state", "ssm state", "idx", "gates"), got, ref):
            assert torch.equal(a, b[:B]), f"{name}: {B} against {sizes[-1]} sequences"
