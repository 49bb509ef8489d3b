"""The walking form of the Mamba2-style block's conv (enough tokens that its threads fill the GPU), through the layer against the
oracle: lengths that four, 16 and 32 steps do not divide, many sequences, every conv width, too few blocks for it; and its note of values that are not finite."""
import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth
from rom_testlib import assert_close, np64
from test_gpu_mamba2 import m2shape, run_mamba2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw,headdim", [
    (dict(B=1, L=9005, d_conv=3, K=1), 64), (dict(B=75, L=70, d_conv=2, K=2), 64), (dict(B=150, L=33, K=1), 32),
    (dict(B=150, L=70, d_conv=2, K=2), 64), (dict(B=222, L=70, d_conv=3, K=1), 64),      # 450 blocks of 16 steps, 444 of 32
])
def test_m2_conv_walk(kw, headdim):
    run_mamba2(m2shape(**{**dict(d_model=64, d_inner=512, E=2), **kw}), headdim)


@pytest.mark.parametrize("B", [75, 150])
def test_m2_conv_walk_not_finite(B):
    s = m2shape(B=B, L=70, d_model=64, d_inner=512, E=2, K=1)
    b, at = 40, 38
    p = synth.make_mamba2_inputs(s, 64)
    p["W_in"][:, s.d_inner + 3:2 * s.d_inner:64, 0] = 4      # one channel of every head follows x[t, 0]
    p["W_r"][:, 0] = 0
    p["x"][:, :, 0] = 0
    cfg = rb.config_from_shape(s)
    outs = []
    for v in (0.0, 3e38):
        p["x"][b, at, 0] = v
        dev = {k: (None if t is None else t.cuda().contiguous()) for k, t in p.items()}
        ws = torch.empty(rb.mamba2_workspace_size(cfg, 64), dtype=torch.uint8, device="cuda")
        out = torch.empty_like(dev["x"])
        rb.rom_mamba2_layer_forward(cfg, 64, rb.make_mamba2_weights(dev), dev["x"], out, None, None, None, ws)
        torch.cuda.synchronize()
        outs.append(out)
    assert not torch.isfinite(outs[1][b, at]).all() and torch.isfinite(outs[1][b, :at]).all()
    # the launch that follows a value that is not finite sums the steps of each block of 16 in another order: one unit of bf16
    rest = [i for i in range(s.B) if i != b]
    assert_close(np64(outs[1][rest]), np64(outs[0][rest]), 2.0 ** -7, "other sequences")
    assert_close(np64(outs[1][b, :at]), np64(outs[0][b, :at]), 2.0 ** -7, "the steps before")
