"""Edges of the chunked matrix form of the Mamba2-style recurrence (64 channels per head, bf16) against the CPU oracle: chunks of
64 steps cut short, one and several segments, decays that underflow inside a chunk, no D / dt bias, top-2."""
import pytest

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
