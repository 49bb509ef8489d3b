"""The one-launch bf16 scan against the CPU oracle: sequences around the eight steps of a tile and the twelve warps that take tiles in turn,
one and two rounds of blocks, every gate / skip / initial state combination; in the layer with one to three Gate rows a token, and with the
checkpoints of the backward pass."""
import pytest

from paper_2506_18145_b200 import binding as rb
from rom_testlib import TOL, assert_close
from test_gpu_backward import bshape, run_layer_backward
from test_gpu_parity import check_layer, run_scan, small_shape

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disc_mode", [0, 1])
@pytest.mark.parametrize("B,L,De,with_z,with_h0,with_D", [
    (1, 96, 4096, True, True, True),          # twelve tiles
    (2, 97, 2048, True, False, True),         # thirteen, the last of one step
    (1, 103, 4096, False, True, False),
    (2, 201, 4096, True, True, False),        # two rounds of blocks, tiles the warps do not share evenly
    (3, 384, 3072, True, False, True),
])
def test_scan_ring(disc_mode, B, L, De, with_z, with_h0, with_D):
    y, Y, hl, HL = run_scan(B, L, De, "bf16", disc_mode, with_z, with_h0, with_D, seed=8600 + L, use_ws=True)
    assert rb.last_launch_count() == 1
    assert_close(y, Y, TOL["bf16"], "y")
    assert_close(hl, HL, 2e-3, "h_last")


@pytest.mark.parametrize("K", [1, 2, 3])
def test_layer_forward_scan_ring(K):
    check_layer(small_shape(B=1, L=150, d_model=64, d_inner=4096, E=4, K=K), "unit")


@pytest.mark.parametrize("L", [100, 145])
@pytest.mark.parametrize("disc_mode", [0, 1])
def test_layer_backward_scan_ring(L, disc_mode):
    run_layer_backward(bshape(B=1, L=L, d_model=64, d_inner=4096, K=1), disc_mode=disc_mode)
