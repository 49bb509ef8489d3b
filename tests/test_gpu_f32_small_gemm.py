"""The small fp32 products of the layer in all their tilings against the oracle: contractions of up to 256, beyond, and off the stages of
64 and 128; x Proj with few blocks, with many and in between; rows and columns that no tile divides."""
import pytest
import torch

from paper_2506_18145_b200 import binding as rb
from paper_2506_18145_b200 import synth
from rom_testlib import GpuLayer, launched_kernels
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


@pytest.mark.parametrize("kw,tile", [
    (dict(B=1, L=70, E=4, d_model=64, d_inner=128), "Li32ELi32ELi4ELi4ELi4ELi64E"),
    (dict(B=1, L=300, E=4, d_model=128, d_inner=512), "Li32ELi32ELi4ELi4ELi8ELi128E"),
    (dict(B=1, L=4700, E=4, d_model=512, d_inner=64), "Li128ELi128ELi8ELi8ELi1ELi16E"),
])
def test_layer_fp32_top1_rows_leave_at_their_tokens(kw, tile):
    """The Out Proj in each of its tilings writes the tokens' rows itself, in an instance of its own."""
    s = small_shape(K=1, dtype="f32", **kw)
    check_layer(s, "unit")
    g = GpuLayer(s, synth.make_inputs(s, recipe="unit"))
    names = [n for n, _ in launched_kernels(lambda: rb.rom_layer_forward(g.cfg, g.weights, g.dev["x"], g.out, g.idx, g.gates, g.counts, g.ws))]
    torch.cuda.synchronize()
    gemms = [n for n in names if "gemm_f32" in n]
    assert [n for n in gemms if "Lb1E" in n] == [n for n in gemms if tile + "Lb1E" in n] and sum("Lb1E" in n for n in gemms) == 1
    assert not any("combine" in n for n in names)
