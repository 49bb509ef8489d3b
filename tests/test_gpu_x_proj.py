"""x Proj of the tensor path against fp64 on the rows it was given: clusters of two, four and eight CTAs on both sides of their lines
(8, 33 and 66 row tiles; 8, 16 and 32 K blocks), uneven shares of the contracted index, row and column counts that no tile divides, and
sizes that stay with the general GEMM."""
import pytest
import torch

from paper_2506_18145_b200 import synth
from rom_testlib import GpuLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,De,R", [
    (1, 2048, 16), (127, 2112, 128), (2048, 2048, 64), (2049, 1088, 48), (4200, 1024, 80), (4300, 512, 16), (8448, 576, 128), (8449, 576, 32),
    (300, 448, 16), (130, 64, 16), (200, 1024, 144), (1024, 2112, 48), (1025, 2048, 16),
])
def test_x_proj(T, De, R):
    s = synth.RomShape("xp", 1, T, 64, De, 16, 4, R, 2, 1, "bf16", 8100 + De + R)
    g = GpuLayer(s, synth.make_inputs(s, recipe="unit"))
    delta_r, Bm, Cm = g.tap("delta_r", torch.bfloat16, R), g.tap("Bm", torch.float32, 16), g.tap("Cm", torch.float32, 16)
    delta_r.fill_(float("nan")); Bm.fill_(float("nan")); Cm.fill_(float("nan"))
    g.forward()
    U, W = g.tap("U", torch.bfloat16, De).double(), g.dev["W_x"].double()
    ref, mag = U @ W.T, U.abs() @ W.abs().T
    got = torch.cat([delta_r.double(), Bm.double(), Cm.double()], dim=1)
    # fp32 sums of De products (2^-24 of their magnitudes each); delta leaves in bf16 (8 significant bits)
    bound = mag * De * 2.0 ** -24 + 1e-30
    bound[:, :R] += ref[:, :R].abs() * 2.0 ** -8
    assert ((got - ref).abs() <= bound).all(), float(((got - ref).abs() / bound).max())
