"""Edges of the bf16 warp scan against the CPU oracle: one pass over short sequences, tiles of eight steps cut short, chunk counts from four to
many with the last chunk short or empty, channel counts that leave a block part empty, every gate / skip / initial state combination; in
the layer with one to three Gate rows a token, and with the checkpoints of the backward pass."""
import pytest

from rom_testlib import TOL, assert_close, recorded, scan_kernels
from test_gpu_backward import bshape, run_layer_backward
from test_gpu_parity import check_layer, run_scan, small_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disc_mode", [0, 1])
@pytest.mark.parametrize("B,L,De,with_z,with_h0,with_D,kernels", [
    (1, 2, 64, True, True, True, ["warp"]),
    (2, 95, 192, True, False, True, ["warp"]),                # half a block of channels missing
    (1, 97, 64, False, True, False, ["warp"]),
    (40, 33, 448, True, True, True, ["warp"]),
    (3, 385, 320, True, True, False, ["ring"]),               # (few chunks: one launch)
    (3, 224, 1600, True, True, True, ["warp", "warp"]),       # four chunks, half a block of channels missing
    (1, 1500, 64, False, True, False, ["warp", "warp"]),
    (2, 1003, 320, True, True, False, ["warp", "warp"]),
    (1, 3001, 128, True, False, True, ["warp", "warp"]),      # as many chunks as the rule allows
])
def test_scan_warp_chunked(disc_mode, B, L, De, with_z, with_h0, with_D, kernels):
    with recorded("rom_scan") as calls:
        y, Y, hl, HL = run_scan(B, L, De, "bf16", disc_mode, with_z, with_h0, with_D, seed=8800 + L, use_ws=True)
    assert scan_kernels(calls[0]) == kernels
    assert_close(y, Y, TOL["bf16"], "y")
    assert_close(hl, HL, 2e-3, "h_last")


@pytest.mark.parametrize("B,L,De", [(2, 200, 64), (2, 250, 64), (2, 300, 64), (2, 340, 64), (2, 390, 64),
                                    (3, 224, 1600), (3, 300, 1600), (3, 350, 1600), (3, 400, 1600), (2, 700, 64), (3, 777, 320)])
def test_scan_warp_chained_states(B, L, De):
    """Chunked (from 1600 channels or 700 steps on): three to fifteen chunks after the first: every block chains the states before it, four at a
    time; h_last leaves with the last."""
    with recorded("rom_scan") as calls:
        y, Y, hl, HL = run_scan(B, L, De, "bf16", 0, True, True, True, seed=8900 + L, use_ws=True)
    assert scan_kernels(calls[0]) == (["warp", "warp"] if De == 1600 or L >= 700 else ["ring"])
    assert_close(y, Y, TOL["bf16"], "y")
    assert_close(hl, HL, 2e-3, "h_last")


@pytest.mark.parametrize("K", [1, 2, 3])
def test_layer_forward_chunked(K):
    with recorded("rom_layer_forward") as calls:
        check_layer(small_shape(B=1, L=1003, d_model=64, d_inner=192, E=4, K=K), "unit")
    assert scan_kernels(calls[0]) == ["warp", "warp"]


@pytest.mark.parametrize("K", [1, 2])
@pytest.mark.parametrize("disc_mode", [0, 1])
def test_layer_backward_chunked(K, disc_mode):
    with recorded("rom_layer_backward") as calls:
        run_layer_backward(bshape(B=2, L=903, d_model=64, d_inner=192, K=K), disc_mode=disc_mode)
    assert scan_kernels(calls[0])[:2] == ["warp", "warp"]
