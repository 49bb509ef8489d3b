"""Gate-weighted sum of two experts' rows (and the Out Proj before it) against fp64 on the rows it was given: widths below, at and beyond
the 1024 elements that a warp takes at once, token counts that leave part of a block without work."""
import pytest
import torch

from paper_2506_18145_b200 import synth
from rom_testlib import GpuLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,Dm", [(1, 64), (5, 320), (131, 1024), (258, 1088), (67, 2112)])
def test_combine_two(T, Dm):
    s = synth.RomShape("cb", 1, T, Dm, 128, 16, 4, 16, 4, 2, "bf16", 6600 + Dm)
    g = GpuLayer(s, synth.make_inputs(s, recipe="unit"))
    g.out.fill_(float("nan"))
    g.forward()
    rows = g.tap("row_of_assign", torch.int32, 2).long()
    Yg, W = g.tap("Ygp", torch.bfloat16, 128).double(), g.dev["W_out"].double()
    ref, bound = torch.zeros((T, Dm), dtype=torch.float64, device="cuda"), torch.zeros((T, Dm), dtype=torch.float64, device="cuda")
    for k in range(2):
        y, w = Yg[rows[:, k]], W[g.idx[:, k].long()]
        o = torch.einsum("tc,tdc->td", y, w) * g.gates[:, k:k + 1].double()
        mag = torch.einsum("tc,tdc->td", y.abs(), w.abs()) * g.gates[:, k:k + 1].double()
        ref += o
        bound += o.abs() * 2.0 ** -8 + mag * 130 * 2.0 ** -24      # an expert's row in bf16, fp32 sums of 128 products
    bound += ref.abs() * 2.0 ** -8 + 1e-30                          # the result in bf16
    got = g.out.view(T, Dm).double()
    assert ((got - ref).abs() <= bound * 1.01).all(), float(((got - ref).abs() / bound).max())
