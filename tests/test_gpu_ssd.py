"""Edges of the chunked matrix form of the Mamba2-style recurrence (64 channels per head, bf16) against the CPU oracle: chunks of
64 steps cut short, one and several segments, decays that underflow inside a chunk, no D / dt bias, top-2."""
import math

import pytest
import torch

from paper_2506_18145_b200 import synth

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
