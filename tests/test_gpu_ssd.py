"""Edges of the chunked matrix form of the Mamba2-style recurrence (64 channels per head, bf16) against the CPU oracle: chunks of
64 steps cut short, one and several segments, decays that underflow inside a chunk, no D / dt bias, top-2."""
import math

import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth

from rom_testlib import assert_close, np64
from test_gpu_mamba2 import m2shape, run_mamba2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(B=1, L=1, E=4, K=1),
    dict(B=3, L=63, E=4, K=1),
    dict(B=2, L=64, E=4, K=2),
    dict(B=1, L=65, E=2, K=1, d_conv=2),
    dict(B=2, L=257, E=4, K=2, d_conv=3),            # segments of two and three chunks
    dict(B=1, L=2050, E=4, K=1),                     # many segments, the last a few steps long
    dict(B=1, L=300, E=2, K=1, d_inner=1024),        # two groups of eight heads
])
def test_ssd_parity(kw):
    run_mamba2(m2shape(**{**dict(d_inner=512), **kw}), 64)


@pytest.mark.parametrize("big", [(2,), (0, 1, 2, 3, 5, 8, 64, 65, 66, 67), (1, 60, 70, 128)])
def test_ssd_decay_between_late_steps_after_large_ones(monkeypatch, big):
    """Steps whose dt A runs into the hundred thousands (decay 0) before ordinary ones in the same chunk: the decay between two later
    steps is a difference of running sums and must keep the precision of a single step's product."""
    s = m2shape(B=1, L=140, E=4, K=1, d_inner=512)
    p = synth.make_mamba2_inputs(s, 64)
    H = s.d_inner // 64
    p["W_in"][:, -H:] = 0
    p["W_in"][:, -H:, 0] = 64                        # dt pre-activation: 64 x[t, 0], i.e. 0 or 64
    p["x"][:, :, 0] = 0
    p["x"][:, list(big), 0] = 1
    p["dt_bias"] = torch.full((H,), math.log(math.expm1(1e-4)))
    p["A"] = -8000.0 * (1.0 + 0.1 * torch.arange(H, dtype=torch.float32))
    p["D"] = None
    monkeypatch.setattr(synth, "make_mamba2_inputs", lambda shape, headdim: p)
    run_mamba2(s, 64)


@pytest.mark.parametrize("at", [5, 31, 38, 100])
def test_ssd_steps_before_one_that_is_not_finite(at):
    """A token whose channels overflow leaves every earlier token's output as it is: the recurrence is causal.  The steps of its own
    block of 16 are summed in another order, which may move the roundings to bf16 behind it by one unit (2^-8 of a value)."""
    s = m2shape(B=1, L=140, E=4, K=1, d_inner=512)
    p = synth.make_mamba2_inputs(s, 64)
    p["W_in"][:, s.d_inner + 3:2 * s.d_inner:64, 0] = 4      # one channel of every head follows x[t, 0]
    p["W_r"][:, 0] = 0
    p["x"][:, :, 0] = 0
    cfg = rb.config_from_shape(s)
    outs = []
    for v in (0.0, 3e38):
        p["x"][0, at, 0] = v
        dev = {k: (None if t is None else t.cuda().contiguous()) for k, t in p.items()}
        ws = torch.empty(rb.mamba2_workspace_size(cfg, 64), dtype=torch.uint8, device="cuda")
        out = torch.empty_like(dev["x"])
        rb.rom_mamba2_layer_forward(cfg, 64, rb.make_mamba2_weights(dev), dev["x"], out, None, None, None, ws)
        torch.cuda.synchronize()
        outs.append(out[0])
    assert torch.isfinite(outs[0]).all() and not torch.isfinite(outs[1][at]).all()
    block = at // 16 * 16
    assert torch.equal(outs[0][:block], outs[1][:block])
    assert torch.isfinite(outs[1][:at]).all()
    assert_close(np64(outs[1][block:at]), np64(outs[0][block:at]), 2.0 ** -7, "the steps before")
