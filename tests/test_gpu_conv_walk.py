"""Edges of the short convolution that walks 32 or 64 steps per thread, through the layer: walks cut short after one to four steps,
lengths below one group of four rows past a walk's start, fewer taps, channel counts that leave a block part empty."""
import pytest

from test_gpu_parity import check_layer, small_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(B=40, L=97, K=1),                                         # four walks, the last of one step
    dict(B=40, L=98, K=2),
    dict(B=160, L=3, K=2, d_inner=64),                             # shorter than the taps
    dict(B=50, L=67, K=1, d_conv=3, d_inner=192),
    dict(B=50, L=92, K=2, d_conv=2, d_inner=1088),                 # two column blocks, the second nearly empty
    dict(B=600, L=130, K=2, d_model=64, d_inner=64),               # walks of 64
    dict(B=1200, L=65, K=1, d_model=64, d_inner=64),
])
def test_conv_walk(kw):
    check_layer(small_shape(dtype="bf16", **kw), "unit")
