"""Edges of the bf16 single-token step's own kernels (few tokens per expert) against the CPU oracle: the register-fed and the
streamed projections on both sides of their dispatch line, one to several passes of 64 token columns, 16 / 32 / 64 columns, a K
range that leaves half a stage, weight tiles cut short, dt ranks off the 32- and 128-wide blocks, every conv width."""
import pytest

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
