"""The small fp32 products of the layer in all their tilings against the oracle: contractions of up to 256, beyond, and off the stages of
64 and 128; x Proj with few blocks, with many and in between; rows and columns that no tile divides."""
import pytest

from test_gpu_parity import check_layer, small_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(B=1, L=37, d_model=320, d_inner=448, E=4, K=1, dt_rank=20),      # 320 and 448: stages of 64 (x Proj of 448: 128, cut short)
    dict(B=1, L=37, d_model=384, d_inner=576, E=4, K=1, dt_rank=20),      # 384 and 576: three and five stages of 128, whole and cut short
    dict(B=1, L=800, d_model=64, d_inner=576, E=2, K=1, dt_rank=260),     # x Proj of 250 blocks (292 columns) in stages of 128
    dict(B=1, L=200, d_model=64, d_inner=256, E=3, K=2),                  # 256: the last x Proj in 16 x 16 tiles, the last in stages of 64
    dict(B=2, L=700, d_model=192, d_inner=320, E=4, K=1, dt_rank=260),    # x Proj of many blocks (292 columns), a dt Proj beyond 256
])
def test_layer_fp32_tilings(kw):
    check_layer(small_shape(dtype="f32", **kw), "unit")
