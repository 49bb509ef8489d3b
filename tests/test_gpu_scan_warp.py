"""Edges of the bf16 warp scan against the CPU oracle: tiles of eight steps cut short, chunk counts from one to many with the last
chunk short or empty, channel counts that leave a block part empty, every gate / skip / initial state combination."""
import pytest

from test_gpu_parity import run_scan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("disc_mode", [0, 1])
@pytest.mark.parametrize("B,L,De,with_z,with_h0,with_D", [
    (1, 2, 64, True, True, True),
    (2, 95, 192, True, False, True),         # one chunk, half a block of channels missing
    (1, 97, 64, False, True, False),         # two chunks of about 48
    (3, 385, 320, True, True, False),
    (1, 3001, 128, True, False, True),       # as many chunks as the rule allows
    (40, 33, 448, True, True, True),
])
def test_scan_warp_chunked(disc_mode, B, L, De, with_z, with_h0, with_D):
    run_scan(B, L, De, "bf16", disc_mode, with_z, with_h0, with_D, seed=8800 + L, use_ws=True)


@pytest.mark.parametrize("L", [200, 250, 300, 340, 390])
def test_scan_warp_chained_states(L):
    """Three to seven chunks after the first: every block chains the states before it, four at a time; h_last leaves with the last."""
    run_scan(2, L, 64, "bf16", 0, True, True, True, seed=8900 + L, use_ws=True)
