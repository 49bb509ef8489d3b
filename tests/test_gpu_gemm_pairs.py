"""Edges of the grouped GEMM on CTA pairs, through the layer, its backward and the FFN-MoE: odd and even row-tile counts per expert
(half-empty pairs), experts without a row, column counts that are no multiple of 256, a K range of one block."""
import pytest

from test_gpu_backward import bshape, run_layer_backward
from test_gpu_parity import check_layer, run_ffn, small_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(B=1, L=256, E=1, K=1),                                            # one pair
    dict(B=1, L=300, E=2, K=1, d_model=64, d_inner=320),                   # one K block; 640 columns
    dict(B=3, L=353, E=4, K=2, d_model=320, d_inner=192, router_bias_scale=3.0),      # most experts nearly empty, one with many tiles
    dict(B=2, L=512, E=8, K=8, d_model=256, d_inner=128),                  # every expert: exactly eight tiles
])
def test_pairs_layer_and_backward(kw):
    check_layer(small_shape(dtype="bf16", **kw), "unit")
    run_layer_backward(bshape(dtype="bf16", **kw))


@pytest.mark.parametrize("kw,d_ff", [(dict(B=1, L=700, E=4, K=1), 384), (dict(B=2, L=333, E=3, K=2, d_model=192), 128)])
def test_pairs_ffn(kw, d_ff):
    run_ffn(small_shape(dtype="bf16", **kw), d_ff)
