"""Backward of the selective scan over chunks whose gradient pre-pass is cut into pieces: one to eight pieces, the last of a chunk or of
the sequence shorter or empty, several groups of eight in the chain, both discretisations and storage types, against the CPU oracle."""
import pytest

from test_gpu_backward import run_scan_backward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("disc_mode", [0, 1])
@pytest.mark.parametrize("B,L,De,with_dh", [(1, 200, 64, True), (1, 700, 64, False), (2, 333, 192, True), (3, 1025, 64, True)])
def test_scan_backward_pieces(dtype, disc_mode, B, L, De, with_dh):
    run_scan_backward(B, L, De, dtype, disc_mode, True, True, True, with_dh, seed=9700 + L)
